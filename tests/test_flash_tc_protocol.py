"""Barrier protocols of the tcgen05 fused attention (csrc/flash_tc.cu), model-checked on the CPU.

Each role of a CTA is a coroutine over mbarriers with PTX phase semantics (the `Bar` model of
tests/test_gemm_persist_protocol.py: a phase completes when its pending arrivals and
transaction bytes reach zero; `try_wait.parity P` succeeds once the phase of parity P has
completed).  TMA bytes land in any order; tcgen05.commit arrivals keep their issue order.  An
MMA is taken to write its TMEM accumulator or read its shared-memory operands at any time
between its issue and its commit, so the checks are:
- nobody reads a TMEM score tile, a stage or an A-operand tile that a later write has been
  issued over, or before the write it needs has committed;
- no stage is refilled, and no A-operand tile rewritten, while an issued MMA may still read it;
- random interleavings end without deadlock, and the outputs are read after the last
  accumulating product committed.

Backward (key-tile and query-tile kernels; rings of n = 2 to 4 stages):
  producer   resident tiles once (res_full); tile i into stage i % n: waits st_empty[s] parity
             ((i / n) & 1) ^ 1
  MMA        res_full parity 0; scores(0); per tile i: s_free parity i & 1, then scores(i + 1)
             (st_full parity ((i + 1) / n) & 1, commit s_full), p_full parity i & 1, the
             accumulating products (commit st_empty[i % n], then o_done)
  8 warps    s_full parity i & 1; read the scores; arrive s_free; for i > 0 o_done parity
             (i - 1) & 1; write the A operands; arrive p_full; at the end o_done parity
             (n - 1) & 1, then the outputs
  Key-tile kernel: two slots of row statistics.  A warp passes p_full of tile i - 1 before it
  reads slot i & 1, and writes slot (i + 1) & 1 with its share of tile i's operands.
Forward: K and V tiles travel in rings of their own (one or two stages).
  producer   per key tile j: k_empty[s] parity ((j / n) & 1) ^ 1, K; then v_empty[s], V
  MMA        q_full; scores(0); per tile: s_free parity j & 1, scores(j + 1) (k_full; commit
             s_full, k_empty), p_full parity j & 1, v_full, P V (commit v_empty, o_done)
  4 warps    s_full parity j & 1; read S; arrive s_free; for j > 0 o_done parity (j - 1) & 1
             (rescale O); write P; arrive p_full; at the end o_done parity (n - 1) & 1."""
import random

import pytest

from test_gemm_persist_protocol import Bar, Deadlock


def _schedule(actors, events, on_event, rnd, limit=20000):
    steps = 0
    while actors or events:
        c = rnd.randrange(len(actors) + (1 if events else 0))
        if c == len(actors):
            commits = [k for k, e in enumerate(events) if e[0] != "tx"]
            tx = [k for k, e in enumerate(events) if e[0] == "tx"]
            idx = commits[0] if commits and (not tx or rnd.random() < 0.5) else rnd.choice(tx)
            on_event(events.pop(idx))
            continue
        try:
            next(actors[c])
        except StopIteration:
            actors.pop(c)
        steps += 1
        if steps > limit:
            raise Deadlock()


def run_backward(ntile, seed, ew=8, stages=2, s_free_count=None, ew_o_done_flip=0,
                 early_scores=False, slots=0):
    """One CTA of the tcgen05 attention backward over ntile streamed tiles (slots: the
    key-tile kernel's row statistics)."""
    rnd = random.Random(seed)
    res_full = Bar(1)
    st_full = [Bar(1) for _ in range(stages)]
    st_empty = [Bar(1) for _ in range(stages)]
    s_full, o_done = Bar(1), Bar(1)
    s_free, p_full = Bar(s_free_count or ew), Bar(ew)
    st = {"stage": [None] * stages, "stage_readers": [set() for _ in range(stages)],
          "S_issued": None, "S_done": None, "op": [None] * ew, "op_reading": None,
          "acc_done": -1, "outputs": 0}
    slot = [[0] * ew] + [[None] * ew for _ in range(slots - 1)]   # slot 0 before the loop
    events = []

    def producer():
        events.append(("tx", "res"))
        res_full.arrive_expect_tx(1)
        yield
        for i in range(ntile):
            s, ph = i % stages, (i // stages) & 1
            while not st_empty[s].try_wait(ph ^ 1):
                yield
            assert not st["stage_readers"][s], "stage refilled while an MMA may read it"
            st_full[s].arrive_expect_tx(1)
            st["stage"][s] = i
            events.append(("tx", s))
            yield

    def scores(i):
        s = i % stages
        while not st_full[s].try_wait((i // stages) & 1):
            yield
        assert st["stage"][s] == i, "scores read the wrong stage"
        st["S_issued"] = i
        st["stage_readers"][s].add(("S", i))
        events.append(("commit", "s_full", i))
        yield

    def mma():
        while not res_full.try_wait(0):
            yield
        yield from scores(0)
        for i in range(ntile):
            if early_scores and i + 1 < ntile:
                yield from scores(i + 1)
            while not s_free.try_wait(i & 1):
                yield
            if not early_scores and i + 1 < ntile:
                yield from scores(i + 1)
            while not p_full.try_wait(i & 1):
                yield
            assert all(o == i for o in st["op"]), "products read A operands of another tile"
            s = i % stages
            assert st["stage"][s] == i, "products read the wrong stage"
            st["stage_readers"][s].add(("acc", i))
            st["op_reading"] = i
            events.append(("commit", "st_empty", i))
            events.append(("commit", "o_done", i))
            yield

    def ew_warp(w):
        for i in range(ntile):
            while slots and i > 0 and not p_full.try_wait((i - 1) & 1):
                yield
            while not s_full.try_wait(i & 1):
                yield
            assert st["S_done"] == i and st["S_issued"] == i, "scores read before written"
            yield
            assert st["S_issued"] == i, "scores overwritten while being read"
            s_free.arrive()
            yield
            assert not slots or slot[i % slots] == [i] * ew, "row statistics of another tile"
            yield
            if i > 0:
                while not o_done.try_wait(((i - 1) & 1) ^ ew_o_done_flip):
                    yield
            assert st["op_reading"] is None, "A operands rewritten while the products read them"
            st["op"][w] = i
            if slots:
                slot[(i + 1) % slots][w] = i + 1
            p_full.arrive()
            yield
        while not o_done.try_wait((ntile - 1) & 1):
            yield
        assert st["acc_done"] == ntile - 1, "outputs read before the last products"
        st["outputs"] += 1

    def on_event(ev):
        if ev[0] == "tx":
            (res_full if ev[1] == "res" else st_full[ev[1]]).complete_tx(1)
        elif ev[1] == "s_full":
            st["S_done"] = ev[2]
            st["stage_readers"][ev[2] % stages].discard(("S", ev[2]))
            s_full.arrive()
        elif ev[1] == "st_empty":
            st["stage_readers"][ev[2] % stages].discard(("acc", ev[2]))
            st_empty[ev[2] % stages].arrive()
        else:
            st["op_reading"] = None
            st["acc_done"] = ev[2]
            o_done.arrive()

    _schedule([producer(), mma()] + [ew_warp(w) for w in range(ew)], events, on_event, rnd)
    return st["outputs"]


def run_forward(n, seed, stages, warps=4, early_release=False, no_s_free=False, o_done_flip=0,
                p_full_count=None):
    """One CTA's forward over n key tiles.  Mistakes to plant: K's stage freed before its commit
    (early_release), the next scores issued without s_free, a flipped parity, a wrong count."""
    rnd = random.Random(seed)
    q_full, s_full, o_done = Bar(1), Bar(1), Bar(1)
    full = {r: [Bar(1) for _ in range(stages)] for r in "kv"}
    empty = {r: [Bar(1) for _ in range(stages)] for r in "kv"}
    s_free, p_full = Bar(warps), Bar(p_full_count or warps)
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
            if not no_s_free:
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
            assert st["S_issued"] == j, "scores overwritten while being read"
            s_free.arrive()
            yield
            if j > 0:
                yield from wait(o_done, ((j - 1) & 1) ^ o_done_flip)
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


@pytest.mark.parametrize("stages,slots", [(2, 2), (3, 2), (3, 0), (4, 0)])
def test_backward_protocol_completes(stages, slots):
    """The rings of the primal and dual kernels: key tiles (with statistics), query tiles."""
    rnd = random.Random(7)
    for seed in range(200):
        n = rnd.randint(1, 11)
        assert run_backward(n, seed, stages=stages, slots=slots) == 8, (n, seed)


@pytest.mark.parametrize("stages", [1, 2])
def test_forward_protocol_completes(stages):
    rnd = random.Random(11)
    for seed in range(300):
        n = rnd.randint(1, 9)
        assert run_forward(n, seed, stages=stages) == 4, (n, seed)


@pytest.mark.parametrize("mistake", ["s_free_count", "o_done_parity", "early_scores", "one_slot"])
def test_backward_model_catches_planted_mistakes(mistake):
    """A wrong arrival count, a flipped parity, the next tile's scores issued before the warps
    have read this tile's, or one slot of statistics are caught in nearly every run with
    several tiles."""
    caught = runs = 0
    rnd = random.Random(3)
    for seed in range(80):
        n = rnd.randint(3, 9)
        kw = {"s_free_count": 9} if mistake == "s_free_count" else \
             {"ew_o_done_flip": 1} if mistake == "o_done_parity" else \
             {"early_scores": True} if mistake == "early_scores" else {"slots": 1}
        runs += 1
        try:
            run_backward(n, seed, **kw)
        except (AssertionError, Deadlock):
            caught += 1
    assert caught >= 0.9 * runs, (mistake, caught, runs)


@pytest.mark.parametrize("mistake", ["o_done_parity", "p_full_count", "no_s_free"])
def test_forward_model_catches_planted_mistakes(mistake):
    caught = runs = 0
    rnd = random.Random(5)
    for seed in range(80):
        n = rnd.randint(3, 9)
        kw = {"o_done_flip": 1} if mistake == "o_done_parity" else \
             {"p_full_count": 5} if mistake == "p_full_count" else {"no_s_free": True}
        runs += 1
        try:
            run_forward(n, seed, stages=2, **kw)
        except (AssertionError, Deadlock):
            caught += 1
    assert caught >= 0.9 * runs, (mistake, caught, runs)


@pytest.mark.parametrize("stages", [1, 2])
def test_forward_model_catches_an_early_release(stages):
    caught = 0
    for seed in range(60):
        try:
            run_forward(9, seed, stages, early_release=True)
        except (AssertionError, Deadlock):
            caught += 1
    assert caught > 15   # the orders in which the refill beats the product
