"""Small float32 MLPs, whose calls run as one block's program: sizes at the program's limits,
calls of more operations than one program holds, every optimiser and store, and caller tensors
that are not 16-byte aligned, against the float64 oracle.

Tolerance: sums of at most 41 products and T <= 24 steps in float32 leave about 1e-6; 2e-5
allows for Adam's division by small second moments (eps = 1e-3).
"""
import math

import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2
from paper_2505_00793_gb300 import synth

EX, PLR, SLR = synth.EXAMPLE_WEIGHTS, synth.PARAM_LOGLR, synth.SCALAR_LOGLR
CASES = {
    # name: (workload, loop fields)
    "one_weight": (synth.Workload("p1", [1, 1], "ident", "squared", "fp32", B=1, T=1, B_outer=1,
                                  alpha=0.1), {}),
    "at_limit": (synth.Workload("p2", [40, 40, 8], "silu", "ce", "fp32", B=12, T=2, B_outer=12,
                                alpha=0.1), {}),
    "past_limit": (synth.Workload("p3", [40, 40, 8], "silu", "ce", "fp32", B=13, T=2, B_outer=12,
                                  alpha=0.1), {}),
    "many_operations": (synth.Workload("p4", [6, 9, 9, 3], "tanh", "squared", "fp32", B=5, T=24,
                                       B_outer=7, momentum=0.5, meta_kind=EX | PLR,
                                       loglr_mean=math.log(0.05), loglr_std=0.1), {}),
    "scalar_lr": (synth.Workload("p5", [7, 31, 33, 2], "gelu", "ce", "fp32", B=9, T=6, B_outer=4,
                                 momentum=0.9, meta_kind=EX | SLR,
                                 extra={"scalar_loglr": math.log(0.05)}), dict(ckpt_every=4)),
    "adam": (synth.Workload("p6", [5, 8, 3], "tanh", "squared", "fp32", B=6, T=9, B_outer=5,
                            optimizer="adam", adam_eps=1e-3, alpha=1e-2), dict(ckpt_slots=2)),
    "no_bias": (synth.Workload("p7", [12, 30, 5], "silu", "squared", "fp32", B=16, T=3,
                               B_outer=20, alpha=0.1, has_bias=False), {}),
}


def _unaligned(t):
    """The same float values 4 bytes past a 16-byte boundary."""
    import torch
    if t.dtype != torch.float32 or t.numel() == 0:
        return t
    u = torch.empty(t.numel() + 1, device=t.device)[1:]
    u.copy_(t.flatten())
    return u.view(t.shape)


@pytest.mark.gpu
@pytest.mark.parametrize("rr", [False, True])
@pytest.mark.parametrize("name", list(CASES))
def test_small_program(name, rr):
    torch, native = need_gpu()
    from oracle import metagrad as om
    w, kw = CASES[name]
    inp = synth.make_inputs(w)
    ref = om.meta_grad(w, inp)
    mode = native.MF_HVP_REV_REV if rr else native.MF_HVP_MIXED_FOR
    loop = native.loop_desc_for(w, mode, **kw)
    for move in (lambda t: t, _unaligned):
        d = {k: move(v) for k, v in native.to_device_inputs(w, inp).items()}
        nan = lambda n: move(torch.full((n,), float("nan"), device="cuda"))
        d_eta, d_th, V = nan(w.n_eta), nan(w.n_params), nan(1)
        mf = native.MixFlow.for_workload(w)
        for _ in range(3):   # eager, captured, replayed
            mf.meta_grad(loop, d["theta0"], d["eta"], d["inner_x"], d["inner_y"], d["outer_x"],
                         d["outer_y"], d_eta, d_th, V)
        mf.sync()
        mf.close()
        assert rel_l2(d_eta.cpu(), ref["d_eta"]) < 2e-5
        assert rel_l2(d_th.cpu(), ref["d_theta0"]) < 2e-5
        assert abs(float(V) - ref["V"]) < 2e-5 * abs(ref["V"])


@pytest.mark.gpu
def test_rollout_and_label_check():
    """The rollout entry point, and a label out of range found inside a program."""
    torch, native = need_gpu()
    from oracle import metagrad as om
    w = CASES["scalar_lr"][0]
    inp = synth.make_inputs(w)
    d = native.to_device_inputs(w, inp)
    out = torch.empty(w.n_params, device="cuda")
    mf = native.MixFlow.for_workload(w)
    loop = native.loop_desc_for(w)
    mf.inner_rollout(loop, d["theta0"], d["eta"], d["inner_x"], d["inner_y"], out)
    mf.sync()
    assert rel_l2(out.cpu(), om.rollout(w, inp)[0][-1].numpy()) < 2e-5
    bad = d["inner_y"].clone()
    bad.view(-1)[3] = w.dims[-1]
    mf.inner_rollout(loop, d["theta0"], d["eta"], d["inner_x"], bad, out)
    with pytest.raises(native.MixflowError) as e:
        mf.sync()
    assert e.value.status == 1
    mf.inner_rollout(loop, d["theta0"], d["eta"], d["inner_x"], d["inner_y"], out)
    mf.sync()
    assert rel_l2(out.cpu(), om.rollout(w, inp)[0][-1].numpy()) < 2e-5
    mf.close()
