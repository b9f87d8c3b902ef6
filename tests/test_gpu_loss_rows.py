"""The MLP loss at the widths where its kernels change (a warp per row up to 128 columns, a
block per row above), through Hessian-vector products against the float64 oracle: rows of
ragged width, one and many rows, with labels and with float targets.

Tolerance: a row's float32 sums over C columns err by about sqrt(C) eps = 6e-6 at C = 3000;
2e-5 leaves room for the two layers' products, and bf16 operands take 2e-2.
"""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2
from paper_2505_00793_gb300 import synth


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("loss", ["ce", "squared"])
@pytest.mark.parametrize("rows,cols", [(1, 128), (70, 129), (3, 131), (33, 260), (5, 1001), (2, 3000)])
def test_loss_rows(rows, cols, loss, prec):
    torch, native = need_gpu()
    from oracle import metagrad as om
    w = synth.Workload("loss_rows", [24, 40, cols], "tanh", loss, prec, B=rows, T=1, B_outer=1,
                       alpha=0.1)
    inp = synth.make_inputs(w)
    x, y = inp.inner_x[0], inp.inner_y[0]
    v = synth.random_direction(w.n_params)
    wt = np.linspace(0.3, 1.0, rows).astype(np.float32)
    d = native.to_device_inputs(w, inp)
    Hv, g = (torch.full((w.n_params,), float("nan"), device="cuda") for _ in range(2))
    tl = torch.full((rows,), float("nan"), device="cuda")
    mf = native.MixFlow.for_workload(w)
    mf.hvp(rows, d["theta0"], d["inner_x"][0], d["inner_y"][0], torch.from_numpy(v).cuda(), Hv,
           ex_w=torch.from_numpy(wt).cuda(), tangent_losses=tl, grad=g)
    mf.sync()
    mf.close()
    tol = 2e-5 if prec == "fp32" else 2e-2
    assert rel_l2(g.cpu().numpy(), om.grad(w, inp.theta0, x, y, wt)) < tol
    assert rel_l2(Hv.cpu().numpy(), om.hvp(w, inp.theta0, x, y, v, wt)) < tol
    assert rel_l2(tl.cpu().numpy(), om.tangent_losses(w, inp.theta0, x, y, v)) < tol
