"""The kernels' dispatch at the sizes where it can go wrong: tile edges,
remainders, unaligned rows, the smallest and largest of each range, against
the fp64 oracle."""
import numpy as np
import pytest

from synth import inputs as S

from helpers import f32, max_row_rel, to_device, to_host

pytestmark = pytest.mark.gpu


# ---------------------------------------------------------------------------
# stand-alone Newton-Schulz: buffers read and written in place or copied,
# large and small inputs, the caller's workspace
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", [(2, 256, 512), (1, 255, 513), (3, 40, 1000), (1, 512, 256), (2, 128, 131),
                                   (2, 3, 5)])
def test_newton_schulz_input_scale(shape, precision):
    """The prescale through the copying and the direct path, below 1e-15 (where
    the norm is summed in fp64) and far above one (3 x 5: past 1e18, in fp64 too;
    the Gram matrix of larger ones would leave the range of fp32 there), and with
    the result over the input: with eps = 0 the iteration only sees X / ||X||, and a power of two
    changes no rounding, so the results are equal bit for bit; and the norm
    itself through one step of X <- 1 X (T = X / ||X|| to one rounding)."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import newton_schulz
    rng = np.random.default_rng(shape[1])
    x = torch.from_numpy(rng.standard_normal(shape).astype(np.float32)).cuda()
    x = x.to(torch.bfloat16) if precision == 0 else x
    T = newton_schulz(x, precision=precision, ns_eps=0.0)
    for scale in (2.0 ** -53, 2.0 ** 53 if shape[2] > 5 else 2.0 ** 60):
        assert torch.equal(newton_schulz(x * scale, precision=precision, ns_eps=0.0), T)
    # T over X
    y = x.clone()
    cfg = C.normpre_default_config(precision=precision, ns_eps=0.0)
    C.normpre_newton_schulz(cfg, *shape, y.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert torch.equal(y, T)
    # C = 1 I: exact products, X / ||X|| rounded once (fp32 scale and product: 2^-23)
    u = to_host(newton_schulz(x, precision=precision, ns_eps=0.0, ns_steps=1, ns_coef=(1.0, 0.0, 0.0)))
    X = to_host(x).astype(np.float64)
    ref = X / np.sqrt((X * X).sum(axis=(1, 2), keepdims=True))
    assert np.all(np.abs(u - ref) <= (2.0 ** -8 if precision == 0 else 2.0 ** -22) * np.abs(ref))


# Widths of the tiles of the Gram product and of the update at 152 SMs: 128 and 256;
# 64 and 128 (the update on two-CTA clusters); 64 and 256 (80 tiles, which narrower
# ones would bring to two waves); 128 and 256, the tall ones 128 and 128; 64 and 64
@pytest.mark.parametrize("shape", [(4, 1024, 4096), (4, 4096, 1024), (1, 1024, 2048), (1, 2048, 1024), (1, 1280, 2048),
                                   (1, 2048, 1280), (90, 128, 256), (90, 256, 128), (1, 384, 640)])
@pytest.mark.parametrize("coef,steps", [((0.0, 1.0, 0.0), 1), ((0.0, 0.0, 1.0), 1), ((3.4445, -4.7750, 2.0315), 5)])
def test_newton_schulz_tile_widths(shape, coef, steps):
    """Every product against fp64 at the tile widths that the small shapes and
    the model sets do not take.  One step rounds to bf16 at most three times, at
    2^-9 each in the norm; a lost or misplaced tile is some hundredths of the whole."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(sum(shape))
    x = torch.randn(shape, device="cuda", generator=gen).bfloat16()
    _check_newton_schulz(x, coef, steps, 3 * 2.0 ** -9 if steps == 1 else 2e-2)


# at 152 SMs: the Gram product plain behind a larger update, the others too, and
# every launch dependent, with the trigger at its head
@pytest.mark.parametrize("shape", [(3, 300, 700), (6, 700, 300), (20, 500, 512), (40, 128, 100)])
def test_newton_schulz_fp32_launches(shape):
    """Five fp32 steps: the iteration's gain of at most 3.4445 a step (the largest
    slope of its polynomial) on some 1e-6 a step."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(sum(shape))
    _check_newton_schulz(torch.randn(shape, device="cuda", generator=gen), (3.4445, -4.7750, 2.0315), 5, 5e-4)


def _check_newton_schulz(x, coef, steps, tol):
    import torch
    from paper_2609_36692_gb300.optim import newton_schulz
    shape = x.shape
    precision = 0 if x.dtype == torch.bfloat16 else 1
    T = newton_schulz(x, ns_steps=steps, ns_coef=coef, precision=precision).double()
    ref = x.double()
    ref = ref.mT if shape[1] > shape[2] else ref
    ref = ref / (ref.flatten(1).norm(dim=1)[:, None, None] + f32(1e-7))
    a, b, c = (f32(v) for v in coef)
    for _ in range(steps):
        gram = ref @ ref.mT
        ref = a * ref + (b * gram + c * (gram @ gram)) @ ref
    ref = ref.mT if shape[1] > shape[2] else ref
    err = (T - ref).flatten(1).norm(dim=1) / ref.flatten(1).norm(dim=1)
    assert err.max() <= tol, err


def test_newton_schulz_workspace():
    import torch
    from paper_2609_36692_gb300 import normpre as C
    cfg = C.normpre_default_config()
    x = torch.randn(2, 100, 300, device="cuda").to(torch.bfloat16)
    t0, t1 = torch.empty_like(x), torch.empty_like(x)
    n = C.normpre_newton_schulz_workspace(cfg, *x.shape)
    ws = torch.full((n,), 255, dtype=torch.uint8, device="cuda")   # its contents do not matter
    s = torch.cuda.current_stream().cuda_stream
    C.normpre_newton_schulz_ws(cfg, *x.shape, x.data_ptr(), t0.data_ptr(), ws.data_ptr(), n, s)
    C.normpre_newton_schulz(cfg, *x.shape, x.data_ptr(), t1.data_ptr(), s)
    assert torch.equal(t0, t1)
    with pytest.raises(C.NormPreError) as e:
        C.normpre_newton_schulz_ws(cfg, *x.shape, x.data_ptr(), t0.data_ptr(), ws.data_ptr(), n - 1, s)
    assert e.value.status == C.NORMPRE_ERR_ARG


# ---------------------------------------------------------------------------
# momentum + tangent + normalization: rows that are not whole 16-byte pieces,
# rows past the register form, blocks of 32 to 256 rows in the column sums
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("w_dtype", ["f32", "bf16"])
@pytest.mark.parametrize("t", [0, 1])
@pytest.mark.parametrize("rows,cols,n", [(33, 1, 1), (1, 33, 2), (257, 1029, 2), (520, 2047, 1), (3, 16391, 1),
                                         (70, 16384, 1), (4097, 264, 3), (2000, 3001, 2)])
def test_normalize_any_width(rows, cols, n, t, w_dtype):
    """Psi per active row against the oracle at 1e-5 (fp32 sums), M_t to its
    rounding, and the G update of odd widths."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    cs = S.custom_config("width_%dx%d" % (rows, cols), [(rows, cols)] * n, g_dtype="bf16", w_dtype=w_dtype,
                         row_sigma=1.0, col_sigma=1.0)
    mats = [S.make_matrix(cs, i) for i in range(n)]
    W, G, M = to_device(mats, "bf16", w_dtype)
    opt = NormPre([(rows, cols)] * n, [w_dtype] * n, ["bf16"] * n, variant=C.NORMPRE_L, precision=1, rank=4,
                  oversample=4)
    opt.step(t, 0.02, W, G, M)
    torch.cuda.synchronize()
    opt.status()
    for i in range(n):
        m = mats[i]["M"].astype(np.float64) * f32(0.95) + mats[i]["G"]
        assert np.all(np.abs(to_host(M[i]) - m) <= 2.5e-7 * np.abs(m) + 1e-30)
        x, w = (m, mats[i]["W"].astype(np.float64)) if t == 0 else (m.T, mats[i]["W"].astype(np.float64).T)
        x = x - (x * w).sum(1, keepdims=True) * w
        nrm = np.linalg.norm(x, axis=1, keepdims=True)
        psi = opt.read(i, C.NORMPRE_BUF_PSI).astype(np.float64)
        assert max_row_rel(psi if t == 0 else psi.T, x / nrm) <= 1e-5
        assert int(opt.read(i, C.NORMPRE_BUF_STATS)[0][1]) == x.shape[0]
    opt.close()


@pytest.mark.parametrize("tangent", [0, 1, 2])
@pytest.mark.parametrize("rows,cols,n", [(4096, 264, 1), (1000, 777, 2), (600, 256, 12),
                                         (512, 20000, 4)])
def test_normalize_columns_large_momentum(rows, cols, n, tangent):
    """Entries of 1.5e18: the sum of a row lane stays in the range of fp32 (at most
    32 rows), that of a column does not.  Psi per column against fp64 at 1e-5 (fp32
    sums), through a step and through the allocation-free entry point."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    gen = torch.Generator(device="cuda").manual_seed(rows + n)
    draw = lambda f: [torch.randn(rows, cols, device="cuda", generator=gen) * f for _ in range(n)]  # noqa: E731
    W, G, M0 = draw(0.02), [g.bfloat16() for g in draw(1.5e18)], draw(1e17)
    M = [x.clone() for x in M0]
    opt = NormPre([(rows, cols)] * n, ["f32"] * n, ["bf16"] * n, variant=C.NORMPRE_L, precision=1, rank=4,
                  oversample=4, tangent=tangent)
    x64 = []
    for i in range(n):
        m, w = M0[i].double() * f32(0.95) + G[i].double(), W[i].double()
        assert m.square().sum(0).min() > torch.finfo(torch.float32).max
        a = (m * w).sum(0)
        a = a if tangent == 0 else a / w.square().sum(0) if tangent == 2 else 0 * a
        x64.append(m - a * w)
    if tangent == 0:      # the entry point without a handle; its W is not updated
        m, psi = M0[0].clone(), torch.empty_like(M0[0])
        C.normpre_normalize_cols_noalloc(rows, cols, 0.95, G[0].data_ptr(), C.NORMPRE_BF16, m.data_ptr(),
                                         W[0].data_ptr(), C.NORMPRE_F32, psi.data_ptr(),
                                         torch.cuda.current_stream().cuda_stream)
        assert max_row_rel(to_host(psi).T, (x64[0] / x64[0].norm(dim=0)).T.cpu().numpy()) <= 1e-5
    opt.step(1, 0.02, W, G, M)
    assert opt.status() == C.NORMPRE_OK
    for i in range(n):
        psi = opt.read(i, C.NORMPRE_BUF_PSI).astype(np.float64)
        assert max_row_rel(psi.T, (x64[i] / x64[i].norm(dim=0)).T.cpu().numpy()) <= 1e-5
        assert int(opt.read(i, C.NORMPRE_BUF_STATS)[0][1]) == cols
    opt.close()


@pytest.mark.parametrize("w_dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols", [(1, 5), (37, 1), (9, 255), (50, 2049), (300, 257)])
def test_update_g_any_width(rows, cols, w_dtype):
    """The RMS-matched update from the library's own T: one fp32 rounding."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    cs = S.custom_config("upd_%dx%d" % (rows, cols), [(rows, cols)], g_dtype="bf16", w_dtype=w_dtype)
    mats = [S.make_matrix(cs, 0)]
    W, G, M = to_device(mats, "bf16", w_dtype)
    opt = NormPre([(rows, cols)], [w_dtype], ["bf16"])
    opt.step(0, 0.02, W, G, M)
    torch.cuda.synchronize()
    opt.status()
    T = opt.read(0, C.NORMPRE_BUF_T).astype(np.float64)
    w0 = mats[0]["W"].astype(np.float64)
    ref = w0 - f32(0.02) * (f32(0.2) * T / np.sqrt((T * T).mean()) + f32(0.1) * w0)
    tol = 1e-6 if w_dtype == "f32" else 2.0 ** -8   # fp32 fma and scale; half a bf16 spacing, doubled for ties
    assert np.all(np.abs(to_host(W[0]) - ref) <= tol * (np.abs(ref) + 0.004))
    opt.close()


# ---------------------------------------------------------------------------
# CholeskyQR in one cluster launch and the Jacobi eigensolver: sketch widths
# at the edges of the register and pair layouts, panels of 1 to 8 CTAs, a rank
# below the sketch width, and panels that only the launch chain takes
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("t", [0, 1])
@pytest.mark.parametrize("rows,cols,rank,oversample", [(300, 200, 1, 0), (64, 700, 2, 1), (513, 90, 7, 0),
                                                       (1025, 130, 9, 4), (2049, 70, 16, 0), (4097, 96, 24, 8),
                                                       (130, 600, 33, 0), (520, 1030, 39, 8), (700, 600, 40, 8),
                                                       (260, 700, 49, 0), (300, 400, 64, 1), (300, 310, 64, 8),
                                                       (9000, 72, 8, 8), (400, 9, 16, 8),
                                                       # l % 4 == 0 with panels whose matrix stride is odd
                                                       (4, 5, 8, 8), (12, 39, 32, 8), (67, 16, 64, 8)])
def test_sketch_basis_and_ritz_pairs(rows, cols, rank, oversample, t):
    """Q orthonormal on its kept columns, the Ritz pairs those of (Psi_a^T Q)'s
    Gram matrix in fp64: residuals and orthonormality at 2e-5 of the largest
    value (l eps with l <= 72 and the sums' own rounding), values descending."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    n = 3
    cs = S.custom_config("ritz_%dx%d_%d" % (rows, cols, rank), [(rows, cols)] * n, row_sigma=1.0, col_sigma=1.0)
    mats = [S.make_matrix(cs, i) for i in range(n)]
    W, G, M = to_device(mats, "f32", "f32")
    opt = NormPre([(rows, cols)] * n, ["f32"] * n, ["f32"] * n, variant=C.NORMPRE_L, precision=1, rank=rank,
                  oversample=oversample)
    opt.step(t, 0.02, W, G, M)
    torch.cuda.synchronize()
    opt.status()
    for i in range(n):
        psi = opt.read(i, C.NORMPRE_BUF_PSI).astype(np.float64)
        psi = psi if t == 0 else psi.T
        Q = opt.read(i, C.NORMPRE_BUF_Q).astype(np.float64)
        Z = opt.read(i, C.NORMPRE_BUF_Z).astype(np.float64)
        lam = opt.read(i, C.NORMPRE_BUF_RITZ)[0].astype(np.float64)
        l = min(psi.shape[0], rank + oversample)
        assert Q.shape == (psi.shape[0], l) and Z.shape == (l, l) and lam.shape == (l,)
        kept = np.linalg.norm(Q, axis=0) > 0.5
        assert np.count_nonzero(kept) >= min(l, psi.shape[1])
        assert np.abs(Q.T @ Q - np.diag(kept.astype(np.float64))).max() <= 2e-5
        gamma = (Q.T @ psi) @ (Q.T @ psi).T
        assert np.abs(Z.T @ Z - np.eye(l)).max() <= 2e-5
        assert np.abs(gamma @ Z - Z * lam).max() <= 2e-5 * lam[0]
        assert np.all(np.diff(lam) <= 0)
    opt.close()


# ---------------------------------------------------------------------------
# NormPre-L apply, bf16 W or Psi: two W columns a lane where the launch has
# enough units and its rows have an even width, one column a lane elsewhere
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("w_dtype,precision", [("bf16", 0), ("f32", 0), ("bf16", 1)])
@pytest.mark.parametrize("t", [0, 1])
@pytest.mark.parametrize("rows,cols,n,rank", [(130, 520, 30, 40), (1000, 510, 12, 16), (513, 1030, 8, 36),
                                              (37, 1300, 30, 32), (641, 2, 31, 16), (256, 770, 33, 64),
                                              (1, 1290, 30, 4)])
def test_apply_two_columns_a_lane(rows, cols, n, rank, t, w_dtype, precision):
    """W_new against cw W + ct (Psi + D), D = Q K Q^T Psi, formed in fp64 from the
    step's own Psi, Q, Ritz pairs and ||T||^2.  D within 2^-14 of its largest entry:
    the panels are fp32 (a bf16 Psi is contracted with a two-term split, 2^-16), the
    product a three-product split, 2^-20; a split without one of its lo terms, cut
    off at 2^-10, is out by 2^-11.  W_new is rounded to bf16, half a spacing (2^-8 of
    it at most), or to fp32."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    gen = torch.Generator(device="cuda").manual_seed(rows + cols)
    td = torch.bfloat16 if w_dtype == "bf16" else torch.float32
    G = [torch.randn(rows, cols, device="cuda", generator=gen).bfloat16() for _ in range(n)]
    M = [torch.randn(rows, cols, device="cuda", generator=gen) for _ in range(n)]
    W0 = [(torch.randn(rows, cols, device="cuda", generator=gen) * 0.02).to(td) for _ in range(n)]
    W = [x.clone() for x in W0]
    opt = NormPre([(rows, cols)] * n, [w_dtype] * n, ["bf16"] * n, variant=C.NORMPRE_L, precision=precision, rank=rank,
                  oversample=0)
    opt.step(t, 0.5, W, G, M)
    assert opt.status() == C.NORMPRE_OK
    for i in range(n):
        psi = opt.read(i, C.NORMPRE_BUF_PSI).astype(np.float64)
        pa = psi if t == 0 else psi.T
        Q = opt.read(i, C.NORMPRE_BUF_Q).astype(np.float64)
        Z = opt.read(i, C.NORMPRE_BUF_Z).astype(np.float64)
        lam = opt.read(i, C.NORMPRE_BUF_RITZ)[0].astype(np.float64)
        nrm2 = float(opt.read(i, C.NORMPRE_BUF_STATS)[0][2])
        gain = 1.0 / np.sqrt(np.maximum(lam, 1.0)) - 1.0     # of the values above one
        D = Q @ ((Z * gain) @ (Z.T @ (Q.T @ pa)))
        D = D if t == 0 else D.T
        w0, w1 = (x[i].double().cpu().numpy() for x in (W0, W))
        ct = 0.5 * f32(0.2) * np.sqrt(rows * cols / nrm2)
        ref = (1.0 - 0.5 * f32(0.1)) * w0 - ct * (psi + D)
        size = np.abs(w0) + ct * (np.abs(psi) + np.abs(D))
        tol = 2.0 ** -14 * ct * np.abs(D).max() + 2.0 ** -21 * size
        if w_dtype == "bf16":
            tol = tol + 2.0 ** -8 * (np.abs(ref) + tol)
        assert np.all(np.abs(w1 - ref) <= tol), (i, (np.abs(w1 - ref) / tol).max())
    opt.close()


# ---------------------------------------------------------------------------
# non-finite gradients: the step is reported, nothing faults, and the handle's
# next step on finite inputs is that of a fresh one
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("variant,precision,rank", [(1, 1, 32), (1, 0, 32), (1, 1, 64), (0, 0, 32), (2, 0, 32)])
def test_nonfinite_gradient_is_reported(variant, precision, rank, value):
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import NormPre
    gen = torch.Generator(device="cuda").manual_seed(3)
    shapes = [(256, 320), (90, 200)]
    draw = lambda f: [torch.randn(s, device="cuda", generator=gen) * f for s in shapes]  # noqa: E731
    W0, G0, M0 = draw(0.02), draw(1.0), draw(1.0)
    out = []
    for poison in (True, False):
        opt = NormPre(shapes, ["f32"] * 2, ["f32"] * 2, variant=variant, precision=precision, rank=rank)
        for t in (0, 1):
            if poison:
                W, G, M = ([x.clone() for x in v] for v in (W0, G0, M0))
                G[0][7, 11] = value
                opt.step(t, 0.02, W, G, M)
                assert opt.status(raise_on_error=False) != C.NORMPRE_OK
            W, M = [x.clone() for x in W0], [x.clone() for x in M0]
            opt.step(t, 0.02, W, G0, M)
            assert opt.status() == C.NORMPRE_OK
            out.append(W)
        opt.close()
    for a, b in zip(out[:2], out[2:]):
        assert all(torch.equal(x, y) for x, y in zip(a, b))


# ---------------------------------------------------------------------------
# stream capture: the dependent launches of a step as edges of a graph
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("variant,precision", [(0, 0), (0, 1), (1, 1), (1, 0), (2, 0)])
@pytest.mark.parametrize("shapes", [[(256, 512)], [(256, 512), (300, 77), (512, 256), (256, 512), (40, 1100)]])
def test_captured_step_equals_eager(shapes, variant, precision):
    """A captured pair of steps, replayed twice, updates W and M as the same four
    steps launched one by one, bit for bit."""
    import torch
    from paper_2609_36692_gb300.optim import NormPre
    gen = torch.Generator(device="cuda").manual_seed(9)
    draw = lambda f: [torch.randn(s, device="cuda", generator=gen) * f for s in shapes]  # noqa: E731
    W, G, M = draw(0.02), [g.bfloat16() for g in draw(1.0)], draw(1.0)
    W2, M2 = [w.clone() for w in W], [m.clone() for m in M]
    eager, captured = (NormPre.for_tensors(W, G, variant=variant, precision=precision, rank=16) for _ in range(2))
    for t in (0, 1, 0, 1):
        eager.step(t, 0.02, W, G, M)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        for t in (0, 1):
            captured.step(t, 0.02, W2, G, M2)
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert eager.status() == 0 and captured.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(W + M, W2 + M2))
    eager.close()
    captured.close()
