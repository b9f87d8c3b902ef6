"""The decoder backward's small passes against the float64 oracle: the scan of the token counts
over one pass and several (4096 counts each) with ragged ends, the token lists and gain sums on
the side stream and on the working stream, and parameters that are not 16-byte aligned (the
block-per-row norm).

Tolerance: the float32 decoders' bar, 1e-4.
"""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2
from paper_2505_00793_gb300 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("side", [True, False])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("V", [8, 4088, 4096, 4104, 8200])
def test_decoder_backward_passes(V, shift, side):
    torch, native = need_gpu()
    from oracle import metagrad as om
    w = synth.decoder("dec_passes", 16, 2, 24, 2, V, 16, B=3, T=1, B_outer=1,
                      alpha=0.1).with_(precision="fp32")
    inp = synth.make_inputs(w)
    ids = inp.inner_x[0]
    ids[0, 0] = V - 1   # the last id's segment
    v = synth.random_direction(w.n_params, 2, 3)
    wt = np.linspace(0.3, 1.0, w.B).astype(np.float32)

    def dev(a):
        t = torch.empty(a.size + shift, device="cuda")[shift:]
        return t.copy_(torch.from_numpy(a))

    d = native.to_device_inputs(w, inp)
    Hv, g = (dev(np.full(w.n_params, np.nan, np.float32)) for _ in range(2))
    mf = native.MixFlow.for_workload(w)
    mf.set_option(native.MF_OPT_CONCURRENT, int(side))
    for mode in (native.MF_HVP_MIXED_FOR, native.MF_HVP_REV_REV):
        for _ in range(3):   # eager, captured, replayed
            mf.hvp(w.B, dev(inp.theta0), d["inner_x"][0], d["inner_y"][0], dev(v), Hv,
                   ex_w=torch.from_numpy(wt).cuda(), grad=g, hvp_mode=mode)
        mf.sync()
        assert rel_l2(g.cpu().numpy(), om.grad(w, inp.theta0, ids, ids, wt)) < 1e-4
        assert rel_l2(Hv.cpu().numpy(), om.hvp(w, inp.theta0, ids, ids, v, wt)) < 1e-4
    mf.close()


@pytest.mark.gpu
@pytest.mark.parametrize("d,H,rows,S", [(264, 33, 1, 16), (520, 65, 5, 24), (776, 97, 3, 200),
                                        (1024, 16, 2, 616), (1032, 129, 2, 16),
                                        (1024, 16, 8, 520), (2056, 257, 1, 8)])
def test_norm_widths(d, H, rows, S):
    """RMSNorm kernels by row width and batch: rows kept by a warp, by a block (one and two
    column groups a thread, ragged ends, fewer than eight rows in the last block), and walked;
    primal and dual (both schedules), on either side of the rules that choose."""
    torch, native = need_gpu()
    from oracle import metagrad as om
    w = synth.decoder("norms", d, H, 8, 1, 16, S, B=rows, T=1, B_outer=1,
                      alpha=0.1).with_(precision="fp32")
    inp = synth.make_inputs(w)
    ids = inp.inner_x[0]
    v = synth.random_direction(w.n_params, 2, 3)
    one = np.ones(w.B, np.float32)
    d_in = native.to_device_inputs(w, inp)
    mf = native.MixFlow.for_workload(w)
    ref = om.grad(w, inp.theta0, ids, ids, one), om.hvp(w, inp.theta0, ids, ids, v, one)
    for mode in (native.MF_HVP_MIXED_FOR, native.MF_HVP_REV_REV):
        Hv, g = (torch.full((w.n_params,), float("nan"), device="cuda") for _ in range(2))
        mf.hvp(w.B, d_in["theta0"], d_in["inner_x"][0], d_in["inner_y"][0],
               torch.from_numpy(v).cuda(), Hv, grad=g, hvp_mode=mode)
        mf.sync()
        assert rel_l2(g.cpu().numpy(), ref[0]) < 1e-4
        assert rel_l2(Hv.cpu().numpy(), ref[1]) < 1e-4
    mf.close()
