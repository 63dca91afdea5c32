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


