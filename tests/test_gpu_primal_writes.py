"""What a primal decoder pass leaves alone: a training step has no tangent, so the tangent
buffers of the MLP branch (as wide as the hidden layer, the largest of the workspace here) keep
what the allocator left in them.
"""
import ctypes as C

import pytest

from gpu_util import need_gpu
from paper_2505_00793_gb300 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_rollout_leaves_tangents_untouched(prec):
    torch, native = need_gpu()
    d, F, L, B, S = 16, 2048, 2, 32, 32
    w = synth.decoder("primal", d, 2, F, L, 16, S, B=B, T=2, B_outer=1, alpha=1e-2)
    w = w.with_(precision=prec)
    inp = native.to_device_inputs(w, synth.make_inputs(w))
    held = []

    @C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
    def alloc(nbytes, stream, ctx):
        held.append(torch.full(((nbytes + 3) // 4,), -1, dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        return held[-1].data_ptr()

    @C.CFUNCTYPE(None, C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
    def free(ptr, nbytes, stream, ctx):
        pass

    mf = native.MixFlow.for_workload(w)
    mf._check(mf._lib.mf_set_allocator(mf.h, C.cast(alloc, C.c_void_p), C.cast(free, C.c_void_p),
                                       None), "mf_set_allocator")
    out = torch.empty(w.n_params, device="cuda")
    mf.inner_rollout(native.loop_desc_for(w), inp["theta0"], inp["eta"], inp["inner_x"],
                     inp["inner_y"], out)
    mf.sync()
    assert len(held) == 1 and torch.isfinite(out).all()
    es = 2 if prec == "bf16" else 4
    untouched = int((held[0] == -1).sum()) * 4
    mf.close()
    # per block phi''(z) z' (float32) and a', and one dz': each N x F
    assert untouched >= B * S * F * (L * (4 + es) + es)
