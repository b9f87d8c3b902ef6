"""The rings of the tcgen05 attention (csrc/flash_tc.cu): its barrier protocol on the CPU and
its numbers on the GPU.

Forward: K and V tiles travel in rings of their own (one or two stages).
  producer   per key tile j: k_empty[s] parity ((j / n) & 1) ^ 1, K; then v_empty[s], V
  MMA        q_full; scores(0); per tile: s_free parity j & 1, scores(j + 1) (k_full; commit
             s_full, k_empty), p_full parity j & 1, v_full, P V (commit v_empty, o_done)
  4 warps    s_full parity j & 1; read S; arrive s_free; for j > 0 o_done parity (j - 1) & 1;
             write P; arrive p_full
Backward: rings of two to four stages (the model of test_flash_tc_protocol), and in the key-tile
kernel two slots of row statistics: a warp that has passed p_full of tile i - 1 reads slot i & 1
and, with its share of tile i's operands, writes slot (i + 1) & 1.

Numbers: sequences whose tiles go round every ring at least once, and the smallest, through
Hessian-vector products against the float64 oracle (2e-2, the bar of bf16 decoders) and against
the warp-level kernels (1e-2: bf16 rounding points of P and dS differ).
"""
import random

import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2
from paper_2505_00793_gb300 import synth
from test_flash_tc_protocol import _schedule, run_backward
from test_gemm_persist_protocol import Bar, Deadlock


def run_forward(n, seed, stages, early_release=False, warps=4):
    """One CTA's forward; early_release plants a mistake: K's stage freed before its commit."""
    rnd = random.Random(seed)
    q_full, s_full, o_done = Bar(1), Bar(1), Bar(1)
    full = {r: [Bar(1) for _ in range(stages)] for r in "kv"}
    empty = {r: [Bar(1) for _ in range(stages)] for r in "kv"}
    s_free, p_full = Bar(warps), Bar(warps)
    tile = {r: [None] * stages for r in "kv"}
    busy = {r: [False] * stages for r in "kv"}
    st = {"S": None, "S_issued": None, "P": [None] * warps, "P_read": False, "O": -1, "out": 0}
    events = []

    def wait(bar, parity):
        while not bar.try_wait(parity):
            yield

    def producer():
        q_full.arrive_expect_tx(1)
        events.append(("tx", q_full))
        for j in range(n):
            s = j % stages
            for r in "kv":
                yield from wait(empty[r][s], ((j // stages) & 1) ^ 1)
                assert not busy[r][s], "stage refilled while an MMA may read it"
                full[r][s].arrive_expect_tx(1)
                tile[r][s] = j
                events.append(("tx", full[r][s]))
                yield

    def scores(j):
        s = j % stages
        yield from wait(full["k"][s], (j // stages) & 1)
        assert tile["k"][s] == j
        busy["k"][s] = True
        st["S_issued"] = j
        events.append(("commit", "s", j))
        if early_release:
            empty["k"][s].arrive()
        else:
            events.append(("commit", "k", j))
        yield

    def mma():
        yield from wait(q_full, 0)
        yield from scores(0)
        for j in range(n):
            yield from wait(s_free, j & 1)
            if j + 1 < n:
                yield from scores(j + 1)
            yield from wait(p_full, j & 1)
            yield from wait(full["v"][j % stages], (j // stages) & 1)
            assert tile["v"][j % stages] == j and all(p == j for p in st["P"])
            busy["v"][j % stages] = True
            st["P_read"] = True
            events.append(("commit", "v", j))
            events.append(("commit", "o", j))
            yield

    def softmax(w):
        for j in range(n):
            yield from wait(s_full, j & 1)
            assert st["S"] == j and st["S_issued"] == j, "scores read before written or after"
            yield
            s_free.arrive()
            yield
            if j > 0:
                yield from wait(o_done, (j - 1) & 1)
            assert not st["P_read"], "P rewritten, or O rescaled, under the products"
            st["P"][w] = j
            p_full.arrive()
            yield
        yield from wait(o_done, (n - 1) & 1)
        assert st["O"] == n - 1
        st["out"] += 1

    def on_event(ev):
        if ev[0] == "tx":
            ev[1].complete_tx(1)
            return
        what, j = ev[1:]
        if what == "s":
            st["S"] = j
            if early_release:
                busy["k"][j % stages] = False
            s_full.arrive()
        elif what in "kv":
            busy[what][j % stages] = False
            empty[what][j % stages].arrive()
        else:
            st["P_read"], st["O"] = False, j
            o_done.arrive()

    _schedule([producer(), mma()] + [softmax(w) for w in range(warps)], events, on_event, rnd)
    return st["out"]


def run_statistics(n, seed, warps=8, slots=2):
    """The key-tile kernel's statistics slots."""
    rnd = random.Random(seed)
    s_full, o_done, s_free, p_full = Bar(1), Bar(1), Bar(warps), Bar(warps)
    slot = [[0] * warps] + [[None] * warps for _ in range(slots - 1)]   # slot 0 before the loop

    def mma():
        s_full.arrive()
        yield
        for i in range(n):
            while not s_free.try_wait(i & 1):
                yield
            if i + 1 < n:
                s_full.arrive()
            while not p_full.try_wait(i & 1):
                yield
            o_done.arrive()
            yield

    def warp(w):
        for i in range(n):
            while i > 0 and not p_full.try_wait((i - 1) & 1):
                yield
            while not s_full.try_wait(i & 1):
                yield
            s_free.arrive()
            yield
            assert slot[i % slots] == [i] * warps, "statistics of another tile"
            yield
            while i > 0 and not o_done.try_wait((i - 1) & 1):
                yield
            slot[(i + 1) % slots][w] = i + 1
            p_full.arrive()
            yield

    _schedule([mma()] + [warp(w) for w in range(warps)], [], None, rnd)


@pytest.mark.parametrize("stages", [1, 2])
def test_forward_rings(stages):
    for seed in range(200):
        assert run_forward(1 + seed % 9, seed, stages) == 4
    caught = 0
    for seed in range(60):
        try:
            run_forward(9, seed, stages, early_release=True)
        except (AssertionError, Deadlock):
            caught += 1
    assert caught > 15   # the orders in which the refill beats the product


@pytest.mark.parametrize("stages", [3, 4])
def test_backward_rings(stages):
    for seed in range(150):
        assert run_backward(1 + seed % 11, seed, stages=stages) == 8


def test_statistics_slots():
    for seed in range(100):
        run_statistics(1 + seed % 7, seed)
    with pytest.raises(AssertionError):
        for seed in range(20):
            run_statistics(6, seed, slots=1)


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
