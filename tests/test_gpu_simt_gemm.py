"""The float32 GEMM's tiles, K splits and ragged edges, through float32 Hessian-vector
products against the float64 oracle.

Each case's layers put a product (forward and data products at B rows, weight products with
K = B) on the edges of the 32-, 64- and 128-wide tiles, of the K blocks (8, 16, 32) and of
the cluster's K shares, in every operand layout and, over both sweeps, every product mask the
executors issue.

Tolerance: a float32 sum of K products errs by at most K eps relative to the sum of their
magnitudes and by about sqrt(K) eps = 2.3e-6 for K = 1500 on random signs; three layers and
their tangents add a few of those.  2e-5 holds that with room, and is 5 times below the bar
of the float32 paths.
"""
import numpy as np
import pytest

from paper_2505_00793_gb300 import synth
from tests.gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu

CASES = {
    "one_element": ([1, 1], 1, True),
    "edge32": ([33, 65, 31], 32, True),
    "edge64": ([64, 129, 63, 7], 65, False),
    "narrow_out": ([500, 333, 10], 257, True),      # 32-wide tiles, K split over a cluster
    "mid": ([130, 1023, 257, 3], 300, True),        # 64-wide tiles and splits
    "wide": ([300, 1500, 1400], 700, True),         # 128-wide tiles
    "long_k": ([40, 72, 40], 1500, False),          # weight products with a long K
}


@pytest.mark.parametrize("rr", [False, True])
@pytest.mark.parametrize("name", list(CASES))
def test_hvp_fp32_tiles(name, rr):
    torch, native = need_gpu()
    from oracle import metagrad as om
    dims, B, bias = CASES[name]
    w = synth.Workload(name, dims, "tanh", "squared", "fp32", B=B, T=1, B_outer=1, alpha=0.1,
                       has_bias=bias)
    inp = synth.make_inputs(w)
    v = synth.random_direction(w.n_params)
    x, y = inp.inner_x[0], inp.inner_y[0]
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    Hv, g = (torch.full((w.n_params,), float("nan"), device="cuda") for _ in range(2))
    tl = torch.empty(B, device="cuda")
    mf = native.MixFlow.for_workload(w)
    mf.hvp(B, d(inp.theta0), d(x), d(y), d(v), Hv, tangent_losses=tl, grad=g,
           hvp_mode=native.MF_HVP_REV_REV if rr else native.MF_HVP_MIXED_FOR)
    mf.sync()
    mf.close()
    assert rel_l2(Hv.cpu(), om.hvp(w, inp.theta0, x, y, v)) < 2e-5
    assert rel_l2(g.cpu(), om.grad(w, inp.theta0, x, y)) < 2e-5
    assert rel_l2(tl.cpu(), om.tangent_losses(w, inp.theta0, x, y, v)) < 2e-5
