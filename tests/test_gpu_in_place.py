"""Caller parameter vectors used in place of workspace slots: a call gives the same bits whether
theta_0 and the result vectors are separate and aligned (used in place), offset by one float
(copied), or overlap one another (copied), with and without segmented checkpoints, a fused
per-layer update and Adam, and leaves theta_0 as it was.
"""
import math

import numpy as np
import pytest

from gpu_util import need_gpu
from paper_2505_00793_gb300 import synth

EX, PLR = synth.EXAMPLE_WEIGHTS, synth.PARAM_LOGLR
CASES = {
    # name: (workload, loop fields, options)
    "mlp_bf16": (synth.Workload("ip1", [64, 136, 24], "silu", "squared", "bf16", B=20, T=5,
                                B_outer=9, momentum=0.9, meta_kind=EX | PLR,
                                loglr_mean=math.log(0.05), loglr_std=0.1), {}, {}),
    "mlp_segments": (synth.Workload("ip2", [64, 136, 24], "tanh", "ce", "fp32", B=20, T=7,
                                    B_outer=9, alpha=0.1), dict(ckpt_every=3), {}),
    "mlp_per_layer": (synth.Workload("ip3", [64, 136, 24], "gelu", "ce", "bf16", B=20, T=3,
                                     B_outer=9, alpha=0.1), {}, {"MF_OPT_LAYER_UPDATES": 1}),
    "mlp_adam": (synth.Workload("ip4", [64, 136, 24], "tanh", "squared", "fp32", B=20, T=4,
                                B_outer=9, optimizer="adam", adam_eps=1e-3, alpha=1e-2), {}, {}),
    "mlp_one_step": (synth.Workload("ip5", [64, 136, 24], "tanh", "ce", "fp32", B=20, T=1,
                                    B_outer=9, alpha=0.1), {}, {}),
    "decoder": (synth.decoder("ip6", 64, 1, 72, 1, 40, 64, B=2, T=3, B_outer=2, alpha=1e-2),
                {}, {}),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(CASES))
def test_vectors_in_place(name):
    torch, native = need_gpu()
    w, kw, opts = CASES[name]
    d = native.to_device_inputs(w, synth.make_inputs(w))
    P = w.n_params
    loop = native.loop_desc_for(w, native.MF_HVP_MIXED_FOR, **kw)
    th = d["theta0"].clone()

    def vec(shift):
        return torch.full((P + shift,), float("nan"), device="cuda")[shift:]

    def run(theta, dth, thT):
        mf = native.MixFlow.for_workload(w)
        for k, v in opts.items():
            mf.set_option(getattr(native, k), v)
        V, de = torch.full((1,), float("nan"), device="cuda"), vec(0)[:0].new_empty(w.n_eta)
        out = []
        for call in range(3):   # eager, captured, replayed
            theta.copy_(th)
            mf.meta_grad(loop, theta, d["eta"], d["inner_x"], d["inner_y"], d["outer_x"],
                         d["outer_y"], de, dth, V)
            mf.sync()
            if dth.data_ptr() != theta.data_ptr():
                assert torch.equal(theta, th)
            out.append([x.cpu().numpy().copy() for x in (de, dth, V)])
            theta.copy_(th)
            mf.inner_rollout(loop, theta, d["eta"], d["inner_x"], d["inner_y"], thT)
            mf.sync()
            out[-1].append(thT.cpu().numpy().copy())
        mf.close()
        for o in out[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(o, out[0]))
        return out[0]

    ref = run(vec(1), vec(1), vec(1))
    assert all(np.isfinite(x).all() for x in ref)
    same, a, b = vec(0), vec(0), vec(4)
    for got in (run(vec(0), a, b), run(vec(0), vec(1), vec(3)), run(same, same, same)):
        for x, y in zip(got, ref):
            np.testing.assert_array_equal(x, y)
