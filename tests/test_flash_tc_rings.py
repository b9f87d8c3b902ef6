"""The rings of the tcgen05 attention (csrc/flash_tc.cu) on the GPU; their barrier protocols are
model-checked in test_flash_tc_protocol.

Sequences whose tiles go round every ring at least once, and the smallest, through
Hessian-vector products against the float64 oracle (2e-2, the bar of bf16 decoders) and against
the warp-level kernels (1e-2: bf16 rounding points of P and dS differ).
"""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2
from paper_2505_00793_gb300 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("S", [128, 256, 384, 640, 1024])
def test_ring_lengths(S):
    torch, native = need_gpu()
    from oracle import metagrad as om
    w = synth.decoder("rings", 128, 2, 128, 1, 64, S, B=2, T=1, B_outer=1, alpha=1e-2)
    inp = synth.make_inputs(w)
    ids = inp.inner_x[0]
    v = synth.random_direction(w.n_params, 2, 3)
    d = native.to_device_inputs(w, inp)
    tv = torch.from_numpy(v).cuda()
    out = {}
    for flash in (1, 2, 3):
        mf = native.MixFlow.for_workload(w)
        mf.set_option(native.MF_OPT_FLASH_ATTN, flash)
        for mode in (native.MF_HVP_MIXED_FOR, native.MF_HVP_REV_REV):   # dual, and primal too
            Hv, g = (torch.full((w.n_params,), float("nan"), device="cuda") for _ in range(2))
            mf.hvp(w.B, d["theta0"], d["inner_x"][0], d["inner_y"][0], tv, Hv, grad=g,
                   hvp_mode=mode)
            mf.sync()
            out[flash, mode] = g.cpu().numpy(), Hv.cpu().numpy()
        mf.close()
    one = np.ones(w.B, np.float32)
    ref = om.grad(w, inp.theta0, ids, ids, one), om.hvp(w, inp.theta0, ids, ids, v, one)
    for (flash, mode), got in out.items():
        for x, r, y in zip(got, ref, out[2, mode]):
            assert rel_l2(x, r) < 2e-2, (flash, mode, rel_l2(x, r))
            assert rel_l2(x, y) < 1e-2, (flash, mode, rel_l2(x, y))
