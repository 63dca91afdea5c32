"""The kernels' dispatch at the sizes where it can go wrong: tile edges,
remainders, unaligned rows, the smallest and largest of each range, against
the fp64 oracle."""
import numpy as np
import pytest

import oracle as O
from synth import inputs as S

from helpers import f32, max_row_rel, oracle_config, rel_fro, to_device, to_host

pytestmark = pytest.mark.gpu


# ---------------------------------------------------------------------------
# stand-alone Newton-Schulz: buffers read and written in place or copied,
# inputs whose squares leave the fp32 range, the caller's workspace
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,scale", [((2, 256, 512), 1.0), ((1, 255, 513), 1.0), ((3, 40, 1000), 1e-25),
                                         ((1, 512, 256), 1e25), ((2, 128, 131), 3e-20)])
def test_newton_schulz_input_scale(shape, scale, precision):
    """The prescale of inputs whose squares overflow or vanish in fp32, through
    the copying and the direct path, and with the result over the input: the
    iteration only sees X / ||X||, so the result is that of the unscaled X
    (eps = 0) within the mode's tolerance."""
    import torch
    from paper_2609_36692_gb300 import normpre as C
    from paper_2609_36692_gb300.optim import newton_schulz
    rng = np.random.default_rng(shape[1])
    X = rng.standard_normal(shape).astype(np.float32)
    x = torch.from_numpy(X).cuda().to(torch.bfloat16 if precision == 0 else torch.float32) * scale
    X = to_host(x).astype(np.float64) / scale
    T = to_host(newton_schulz(x, precision=precision, ns_eps=0.0))
    tol = 2e-2 if precision == 0 else 1e-4
    for b in range(shape[0]):
        ref = O.newton_schulz(X[b], 5, tuple(f32(c) for c in (3.4445, -4.7750, 2.0315)), 0.0)
        assert rel_fro(T[b], ref) <= tol
    # T over X
    cfg = C.normpre_default_config(precision=precision, ns_eps=0.0)
    C.normpre_newton_schulz(cfg, *shape, x.data_ptr(), x.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(to_host(x), T)


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


