"""How the tcgen05 GEMMs' epilogue warps leave a wait whose limit expires
(csrc/tc_gemm_impl.cuh, csrc/tc_gemm_persist.cu).

On the CPU: the one-SM epilogue's waits and barriers as coroutines, a lane each, in which any set
of lanes may see the limit expire while the accumulator arrives for the others.  Every schedule
must reach the CTA's last barrier, and the tile is stored by all warps or by none.  The two rules
that fail are planted: a lane's own result in front of the barriers, and a warp's.  The sources are
checked to take no lane's own result from a limited wait of the epilogue warps.

On the GPU: limits on both sides of a product's duration.  A call either reports the timeout or
gives the bits of a call under the default limit, and the handle stays usable.
"""
import os
import random
import re

import numpy as np
import pytest

from gpu_util import need_gpu
from paper_2505_00793_gb300 import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_00793_gb300", "csrc")


class Meet:
    """A barrier of n lanes: a generation ends when all of them have arrived."""

    def __init__(self, n):
        self.n, self.in_, self.gen, self.votes, self.result = n, 0, 0, True, True

    def arrive(self, vote=True):
        self.in_ += 1
        self.votes = self.votes and vote
        if self.in_ == self.n:
            self.result, self.votes, self.in_, self.gen = self.votes, True, 0, self.gen + 1


def run_epilogue(rule, seed, warps=4, lanes=2, columns=2, p_expire=0.5, drained=True):
    """One CTA's epilogue warps.  Returns the set of (warp, lane, columns) stored, or None when
    some lane never reaches the last barrier."""
    rnd = random.Random(seed)
    syncwarp = [Meet(lanes) for _ in range(warps)]
    epi, last = Meet(warps * lanes), Meet(warps * lanes)
    acc = [False]          # the accumulator's barrier
    stored = set()

    def meet(m, vote=True):
        g = m.gen
        m.arrive(vote)
        while m.gen == g:
            yield
        return m.result

    def lane(w, i):
        def wait(limited):
            while not acc[0]:
                if limited and rnd.random() < p_expire:
                    return False
                if not limited and not drained and rnd.random() < 0.05:
                    return False   # even the drain gave up
                yield
            return True

        ok = yield from wait(True)
        if rule != "lane":
            ok = yield from meet(syncwarp[w], ok)
        if rule == "cta" and not ok:
            yield from meet(syncwarp[w], (yield from wait(False)))
        if rule == "cta" or ok:
            for c in range(columns):
                if c > 0:
                    yield from meet(epi)
                yield from meet(syncwarp[w])      # the TMEM loads are warp-collective
                done = yield from meet(epi, ok)
                if rule == "cta" and not done:
                    break
                stored.add((w, i, c))
        yield from meet(last)

    actors = [lane(w, i) for w in range(warps) for i in range(lanes)]
    for step in range(20000):
        if not actors:
            return stored
        if step == 40:
            acc[0] = True      # the products complete while some limits have expired
        k = rnd.randrange(len(actors))
        try:
            next(actors[k])
        except StopIteration:
            actors.pop(k)
    return None


@pytest.mark.parametrize("drained", [True, False])
def test_every_schedule_ends(drained):
    none = whole = 0
    for seed in range(400):
        p = (0.0, 0.005, 0.02, 0.5)[seed % 4]
        columns = 1 + seed % 2
        stored = run_epilogue("cta", seed, columns=columns, p_expire=p, drained=drained)
        assert stored is not None, seed
        assert len(stored) in (0, 8 * columns)
        none += not stored
        whole += bool(stored)
    assert none > 50 and whole > 50


@pytest.mark.parametrize("rule", ["lane", "warp"])
def test_model_catches_planted_mistakes(rule):
    stuck = sum(run_epilogue(rule, seed, p_expire=0.02) is None for seed in range(60))
    assert stuck > 20


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_limited_waits_are_voted():
    """A wait of the epilogue warps on the accumulator returns one answer a warp; the one-SM
    kernel's barriers of all epilogue warps stand under no condition on it."""
    src = _source("tc_gemm_impl.cuh")
    one = src[src.index("tc_dual_gemm_kernel("):src.index("typedef CUresult")]
    pair = src[src.index("tc2_dual_gemm_kernel("):src.index("launch_cfg2(")]
    for body, n in ((one, 3), (pair, 1)):
        waits = re.findall(r"(\w+)\(&(acc_bar|recv_bar), 0, p\.status, (p\.wait_ns|DRAIN_NS)\)", body)
        epilogue = waits[1:]   # the first one is the MMA issuer's, a single thread
        assert len(epilogue) == n and {w for w, _, _ in epilogue} == {"mbar_wait_warp"}
    assert not re.search(r"if \(ok\b", one)
    src = _source("tc_gemm_persist.cu")
    waits = re.findall(r"(\S+)\s*pwait<false>\(&acc_full", src)
    assert waits == ["(!__all_sync(0xffffffffu,"]


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", ["one_sm", "pair", "persistent"])
@pytest.mark.parametrize("limit_us", [0, 1, 3, 6, 12, 40])
def test_limits_around_a_product(kernel, limit_us):
    torch, native = need_gpu()
    # unsplit and split products of one-SM tiles; more than 128 rows for the pair tiles
    w = synth.Workload("limit", [128, 256, 512, 136, 10], "gelu", "ce", "bf16", B=160, T=2,
                       B_outer=96, alpha=0.05)
    d = native.to_device_inputs(w, synth.make_inputs(w))
    mf = native.MixFlow.for_workload(w)
    bufs = [torch.empty(n, device="cuda") for n in (w.n_eta, w.n_params, 1)]

    def call():
        mf.meta_grad(native.loop_desc_for(w), d["theta0"], d["eta"], d["inner_x"], d["inner_y"],
                     d["outer_x"], d["outer_y"], *bufs)
        mf.sync()
        return [b.cpu().numpy().copy() for b in bufs]

    try:
        mf.set_option(native.MF_OPT_CUDA_GRAPHS, 0)
        mf.set_option(native.MF_OPT_GEMM_2SM, 0 if kernel == "one_sm" else 2)
        mf.set_option(native.MF_OPT_GEMM_PERSISTENT, int(kernel == "persistent"))
        ref = call()
        mf.set_option(native.MF_OPT_WAIT_LIMIT_US, limit_us)
        for _ in range(4):
            try:
                got = call()
            except native.MixflowError as e:
                assert e.status == 6   # MF_ERR_TIMEOUT
            else:
                assert limit_us > 0
                assert all(np.array_equal(a, b) for a, b in zip(got, ref))
        mf.set_option(native.MF_OPT_WAIT_LIMIT_US, 2000000)
        assert all(np.array_equal(a, b) for a, b in zip(call(), ref))
    finally:
        mf.set_option(native.MF_OPT_WAIT_LIMIT_US, 2000000)
        mf.set_option(native.MF_OPT_GEMM_PERSISTENT, 2)
        mf.set_option(native.MF_OPT_GEMM_2SM, 1)
        mf.close()
