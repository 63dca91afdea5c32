"""The work that a user of the NormPre step has it do, as measurable cases.

A user's training loop calls the optimizer once per step on all hidden weight
matrices of a model.  Steps alternate the active axis (rows on even steps,
columns on odd ones), so one pass of a step case is two consecutive steps,
one of each orientation, on the same weights, gradients and momenta; the
step counter goes on from pass to pass as in training.  Plans (workspaces,
launch descriptors) are made once and kept, as a training loop keeps them.
The stand-alone Newton-Schulz call takes a batch of matrices and is one call.

Values follow the synthetic sets of the repository's benchmark: gradients
N(0, 1) or Student-t (3 degrees of freedom) times log-normal row and column
scales, a prior momentum drawn like a gradient (or zero), weights
N(0, 0.02^2).  Matrices of one shape lie one after the other in one flat
buffer, each at a 16-byte boundary; the flat buffers of W and M are the
outputs, whole.
"""
import math

import torch

LR = 0.02
MU = 0.95
DECAY = 0.1
TARGET_RMS = 0.2
NS_STEPS = 5
NS_COEF = (3.4445, -4.7750, 2.0315)
NS_EPS = 1e-7
SKETCH_SEED = 20260929
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
# a 64-bit pass over more Newton-Schulz operations than this takes too long
EXACT_FLOPS = 1.3e13


def _step(name, shapes, layers, variant, **kw):
    case = dict(name=name, kind="step", shapes=shapes, layers=layers, variant=variant, entry="plan", w="f32", g="bf16",
                precision="f32" if variant == "L" else "bf16", rank=32, oversample=8, dist="normal", row_sigma=1.0,
                col_sigma=1.0, momentum=True)
    case.update(kw)
    return case


def listed():
    gpt2 = "768x2304,768x768,768x3072,3072x768"
    llama = "2048x2048,2048x2048,2048x2048,2048x2048,2048x5504,2048x5504,5504x2048"
    odd_llama = "2048x2048,2048x2048,2048x2048,2048x2048,2048x5461,2048x5461,5461x2048"
    qwen3 = "2048x2048,2048x1024,2048x1024,2048x2048,2048x6144,2048x6144,6144x2048"
    return [
        # one small matrix: launches and dependent latency are all there is
        _step("single_256x1024_G", "256x1024", 1, "G", g="f32", col_sigma=0.0, momentum=False),
        _step("single_256x1024_L", "256x1024", 1, "L", g="f32", col_sigma=0.0, momentum=False, rank=16),
        # GPT-2 Small, the ordinary size: through the torch optimizer (where gradients
        # have their parameters' type), and from a plan with BF16 gradients
        _step("gpt2_small_G", gpt2, 12, "G", entry="optimizer", g="f32"),
        _step("gpt2_small_L", gpt2, 12, "L"),
        # LLaMA ~1B, FP32 parameters, heavy-tailed gradients
        _step("llama_1b_L", llama, 16, "L", dist="student_t3", col_sigma=0.0),
        # two layers with the paper's odd FFN width 5461: unaligned rows
        _step("ffn_5461_G", odd_llama, 2, "G", dist="student_t3", col_sigma=0.0),
        _step("ffn_5461_L", odd_llama, 4, "L", dist="student_t3", col_sigma=0.0),
        # Qwen3 ~1.7B in pure BF16: the largest set; G is bound by the matrix units, L by memory
        _step("qwen3_1p7b_G", qwen3, 28, "G", w="bf16", row_sigma=1.5, col_sigma=1.5),
        _step("qwen3_1p7b_L", qwen3, 28, "L", w="bf16", precision="bf16", row_sigma=1.5, col_sigma=1.5),
        # small matrices of odd and ragged sizes, tall and wide, in one plan
        _step("ragged_G", "50x203,300x256,131x130,1000x40,333x777", 2, "G", entry="optimizer", g="f32"),
        _step("ragged_L", "50x203,300x256,131x130,1000x40,333x777", 2, "L", w="bf16", precision="bf16"),
        # the stand-alone orthogonalization of one layer's momenta
        dict(name="newton_schulz_4x1024x4096", kind="ns", batch=4, rows=1024, cols=4096, row_sigma=1.0, col_sigma=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A transformer's matrix set (or a stand-alone batch) of another size: the
    hidden width over its logarithm from 64 to 2048, widths multiples of 64 or
    as they fall, the weight, gradient and sketch options of the listed cases."""
    if rng.random() < 0.15:
        rows, cols = _log_int(rng, 64, 4096), _log_int(rng, 64, 4096)
        if rng.random() < 0.5:
            rows, cols = -(-rows // 64) * 64, -(-cols // 64) * 64
        return dict(kind="ns", batch=rng.randint(1, 8), rows=rows, cols=cols, row_sigma=1.0,
                    col_sigma=rng.choice([0.0, 1.0]))
    hidden = _log_int(rng, 64, 2048)
    even = rng.random() < 0.5
    if even:
        hidden = -(-hidden // 64) * 64
    ffn = int(hidden * rng.uniform(2.0, 4.0))
    if even:
        ffn = -(-ffn // 64) * 64
    if rng.random() < 0.5:      # fused query-key-value, two MLP matrices
        shapes = [(hidden, 3 * hidden), (hidden, hidden), (hidden, ffn), (ffn, hidden)]
    else:                       # grouped queries, gated MLP
        kv = max(1, hidden // rng.choice([1, 2, 4]))
        shapes = [(hidden, hidden), (hidden, kv), (hidden, kv), (hidden, hidden), (hidden, ffn), (hidden, ffn),
                  (ffn, hidden)]
    variant = rng.choice(["G", "G", "L", "L", "L", "muon"])
    per_layer = sum(r * c for r, c in shapes)
    most = 24 if variant == "L" else 12
    layers = max(1, min(_log_int(rng, 1, most), int(2.5e8 / per_layer)))
    w = rng.choice(["f32", "f32", "bf16"])
    entry = rng.choice(["plan", "optimizer"])
    g = w if entry == "optimizer" else rng.choice(["bf16", "bf16", "f32"])
    precision = "bf16"
    if variant == "L" and w == "f32" and rng.random() < 0.75:
        precision = "f32"
    return dict(kind="step", shapes=",".join("%dx%d" % s for s in shapes), layers=layers, variant=variant,
                entry=entry, w=w, g=g, precision=precision, rank=rng.choice([32, 32, 32, 16, 8, 64]), oversample=8,
                dist=rng.choice(["normal", "student_t3"]), row_sigma=rng.choice([1.0, 1.5]),
                col_sigma=rng.choice([0.0, 1.0, 1.5]), momentum=rng.random() < 0.8)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _shapes(case):
    """Every matrix (rows, cols), in the order of the parameter list."""
    per_layer = [tuple(int(x) for x in s.split("x")) for s in case["shapes"].split(",")]
    return per_layer * case["layers"]


def _gradient(gen, case, shape):
    z = torch.randn(shape, device="cuda", generator=gen)
    if case.get("dist") == "student_t3":
        chi2 = torch.zeros(shape, device="cuda")
        for _ in range(3):
            chi2 += torch.randn(shape, device="cuda", generator=gen).square_()
        z /= (chi2 / 3.0).sqrt_()
    z *= torch.exp(case["row_sigma"] * torch.randn(shape[:-1] + (1,), device="cuda", generator=gen))
    if case["col_sigma"] > 0:
        z *= torch.exp(case["col_sigma"] * torch.randn(shape[:-2] + (1, shape[-1]), device="cuda", generator=gen))
    return z


class _Set:
    """W, G and M of every matrix: views into one flat buffer per shape."""

    def __init__(self, case, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        shapes = _shapes(case)
        groups = sorted(set(shapes), key=shapes.index)
        self.shapes = shapes
        self.stride = {s: -(-(s[0] * s[1]) // 8) * 8 for s in groups}
        self.groups = groups

        def flat(dtype):
            return {s: torch.zeros(shapes.count(s) * self.stride[s], dtype=dtype, device="cuda") for s in groups}

        self.flat_w, self.flat_g, self.flat_m = flat(DTYPES[case["w"]]), flat(DTYPES[case["g"]]), flat(torch.float32)
        self.W, self.G, self.M = (self.views(f) for f in (self.flat_w, self.flat_g, self.flat_m))
        for w, g, m in zip(self.W, self.G, self.M):
            g.copy_(_gradient(gen, case, tuple(g.shape)))
            if case["momentum"]:
                m.copy_(_gradient(gen, case, tuple(m.shape)).to(g.dtype))
            w.copy_(torch.randn(w.shape, device="cuda", generator=gen) * 0.02)

    def views(self, flats):
        """The matrices of the per-shape flat buffers, in the order of the list."""
        seen, out = {s: 0 for s in self.groups}, []
        for s in self.shapes:
            o = seen[s] * self.stride[s]
            seen[s] += 1
            out.append(flats[s][o:o + s[0] * s[1]].view(s))
        return out

    def outputs(self, w, m):
        return {"W": [w[s] for s in self.groups], "M": [m[s] for s in self.groups]}


def _ns_input(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["batch"], case["rows"], case["cols"])
    return _gradient(gen, case, shape).to(torch.bfloat16)


def prepare(case, seed):
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre, NormPreOptimizer
    if case["kind"] == "ns":
        return {"kind": "ns", "X": _ns_input(case, seed)}
    s = _Set(case, seed)
    config = dict(precision=C.NORMPRE_PREC_F32 if case["precision"] == "f32" else C.NORMPRE_PREC_BF16,
                  rank=case["rank"], oversample=case["oversample"], seed=SKETCH_SEED)
    state = {"kind": case["entry"], "set": s, "t": 0}
    if case["entry"] == "optimizer":
        params = [torch.nn.Parameter(w) for w in s.W]
        opt = NormPreOptimizer(params, lr=LR, momentum=MU, weight_decay=DECAY, target_rms=TARGET_RMS,
                               variant=case["variant"], **config)
        for p, g, m in zip(params, s.G, s.M):
            p.grad = g
            opt.state[p]["momentum_buffer"] = m
        state["opt"] = opt
    else:
        variant = {"G": C.NORMPRE_G, "L": C.NORMPRE_L, "muon": C.NORMPRE_MUON}[case["variant"]]
        state["plan"] = NormPre.for_tensors(s.W, s.G, variant=variant, momentum=MU, weight_decay=DECAY,
                                            target_rms=TARGET_RMS, **config)
    return state


def run(state):
    if state["kind"] == "ns":
        from paper_2609_36692_gb300.optim import newton_schulz
        return newton_schulz(state["X"])
    s = state["set"]
    for _ in range(2):
        if state["kind"] == "optimizer":
            state["opt"].step()
        else:
            state["plan"].step(state["t"], LR, s.W, s.G, s.M)
        state["t"] += 1
    return s.outputs(s.flat_w, s.flat_m)


# --------------------------------------------------------------------------
# work and tolerances
# --------------------------------------------------------------------------
def _ns_flops(rows, cols):
    """Five iterations, the two symmetric products at half of their square."""
    s, big = min(rows, cols), max(rows, cols)
    return NS_STEPS * (s * s * big + s ** 3 + 2 * s * s * big)


def work(case):
    if case["kind"] == "ns":
        n = case["batch"] * case["rows"] * case["cols"]
        return {"bytes": 4 * n, "flops": case["batch"] * _ns_flops(case["rows"], case["cols"])}
    size = {"f32": 4, "bf16": 2}
    nbytes = flops = 0
    for r, c in _shapes(case):
        # one step: G, M and W read, M and W written
        nbytes += r * c * (size[case["g"]] + 8 + 2 * size[case["w"]])
        # the sketch, one power iteration, the projection and its application
        flops += _ns_flops(r, c) if case["variant"] != "L" else 10 * r * c * min(r, c, case["rank"] + case["oversample"])
    return {"bytes": 2 * nbytes, "flops": 2 * flops}


def tolerance(case):
    """Of the updated weights, which two steps change by a fifth of their size;
    about four times the error measured against 64 bits."""
    if case["kind"] == "ns":
        return {"rel": 0.03}          # bf16 operands through 15 products: 7e-3 to 1e-2
    if case["w"] == "bf16":
        return {"rel": 0.012}         # one rounding of W per step: 2.4e-3 (with Newton-Schulz up to 4.4e-3)
    if case["variant"] != "L":
        return {"rel": 0.012}         # bf16 Newton-Schulz: 2e-3 to 4e-3 (smallest matrices)
    if case["precision"] == "bf16":
        return {"rel": 0.002}         # one rounding of Psi: 5e-4
    return {"rel": 1.6e-5}            # 32-bit sums: 1e-6 to 4e-6


# --------------------------------------------------------------------------
# the same in 64 bits, plain torch
# --------------------------------------------------------------------------
def _newton_schulz64(x):
    a, b, c = NS_COEF
    tall = x.shape[0] > x.shape[1]
    x = x.mT if tall else x
    x = x / (x.norm() + NS_EPS)
    for _ in range(NS_STEPS):
        gram = x @ x.mT
        x = a * x + (b * gram + c * (gram @ gram)) @ x
    return x.mT if tall else x


def _omega64(matrix, t, n, l):
    """The sketch matrix: Philox4x32-10 words in pairs through Box-Muller."""
    mask = 0xFFFFFFFF
    blocks = -(-(n * l) // 4)
    zero = torch.zeros(blocks, dtype=torch.int64, device="cuda")
    c = [torch.arange(blocks, device="cuda"), zero + matrix, zero + (t & mask), zero + (t >> 32)]
    k0, k1 = SKETCH_SEED & mask, SKETCH_SEED >> 32

    def mul(m, x):
        low, high = m * (x & 0xFFFF), m * (x >> 16)
        return (high + (low >> 16)) >> 16, (((high & 0xFFFF) << 16) + low) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u = [((x >> 9).double() + 0.5) * 2.0 ** -23 for x in c]
    z = []
    for p in (0, 2):
        radius = (-2.0 * u[p].log()).sqrt()
        z += [radius * (2.0 * math.pi * u[p + 1]).cos(), radius * (2.0 * math.pi * u[p + 1]).sin()]
    return torch.stack(z, 1).reshape(-1)[:n * l].view(n, l)


def _localized64(psi, case, matrix, t):
    """Psi (active axis first) with its leading modes above one brought to one."""
    l = min(psi.shape[0], case["rank"] + case["oversample"])
    y = psi @ _omega64(matrix, t, psi.shape[1], l)
    y = psi @ (psi.mT @ y)
    q, _ = torch.linalg.qr(y)
    b = q.mT @ psi
    lam, z = torch.linalg.eigh(b @ b.mT)
    lam, z = lam.flip(0)[:case["rank"]], z.flip(1)[:, :case["rank"]]
    gain = torch.where(lam > 1.0, lam.clamp_min(1e-300).rsqrt() - 1.0, torch.zeros_like(lam))
    return psi + (q @ z) @ (gain[:, None] * (z.mT @ b))


def _step64(case, matrix, t, w, g, m):
    m = MU * m + g
    if case["variant"] == "muon":
        update = _newton_schulz64(m)
    else:
        x, wa = (m, w) if t % 2 == 0 else (m.mT, w.mT)
        x = x - (x * wa).sum(1, keepdim=True) * wa
        norm = x.norm(dim=1, keepdim=True)
        psi = torch.where(norm > 0, x / norm.clamp_min(1e-300), torch.zeros_like(x))
        update = _newton_schulz64(psi) if case["variant"] == "G" else _localized64(psi, case, matrix, t)
        update = update if t % 2 == 0 else update.mT
    rms = update.square().mean().sqrt()
    scale = torch.where(rms > 0, TARGET_RMS / rms.clamp_min(1e-300), torch.zeros_like(rms))
    return w - LR * (scale * update + DECAY * w), m


def exact(case, seed):
    if case["kind"] == "ns":
        x = _ns_input(case, seed)
        if case["batch"] * _ns_flops(case["rows"], case["cols"]) > EXACT_FLOPS:
            return None
        return torch.stack([_newton_schulz64(x[i].double()) for i in range(case["batch"])])
    if case["variant"] != "L" and work(case)["flops"] > EXACT_FLOPS:
        return None
    s = _Set(case, seed)
    flat_w = {k: torch.zeros(v.numel(), dtype=torch.float64, device="cuda") for k, v in s.flat_w.items()}
    flat_m = {k: torch.zeros(v.numel(), dtype=torch.float64, device="cuda") for k, v in s.flat_m.items()}
    for i, (w64, m64) in enumerate(zip(s.views(flat_w), s.views(flat_m))):
        w, g, m = s.W[i].double(), s.G[i].double(), s.M[i].double()
        for t in range(2):
            w, m = _step64(case, i, t, w, g, m)
        w64.copy_(w)
        m64.copy_(m)
    return s.outputs(flat_w, flat_m)
