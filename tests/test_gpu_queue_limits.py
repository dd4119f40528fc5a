"""The limits of a candidate's event queue (sim_opts_t.queue_cap): up to 32 +
queue_cap ops that became ready may wait, and a call beyond that answers
GMG_SIM_QUEUE; within it every result is the oracle's.  Ops without
predecessors do not count before they start, and the log of HBM events has room
for what one generation adds.  (With at most 32 accelerators and in the arbitrated
kernels one op more may wait, where a root's successor took the root's place.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import compare, torch_place  # noqa: E402
from helpers import mk  # noqa: E402
from oracle import oracle as O  # noqa: E402
from paper_2608_15762_gb300 import gmgsim as G  # noqa: E402
from paper_2608_15762_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2608_15762_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _rows(seed, K, n, D):
    rows = np.zeros((K, W.placement_ld(n)), np.uint8)
    rows[:, :n] = np.random.default_rng(seed).integers(0, D, (K, n))
    rows[-1, :n] = 0
    return rows


def _run(d, queue_cap, arb):
    """Two warps per candidate or (warps_per_block) one; each result against the oracle."""
    rows = _rows(1, 4, d.n_ops, d.n_dev)
    g = G.gmg_create(d)
    outs = [G.sim_batch(g, torch_place(rows), req_done=True, queue_cap=queue_cap, arbitrated=arb, warps_per_block=w)
            for w in (0, 4)]
    torch.cuda.synchronize()
    want = O.simulate_batch(d, rows, arbitrated=arb)
    return [(o.to_numpy(), want) for o in outs]


@pytest.mark.parametrize("arb", [False, True])
@pytest.mark.parametrize("D,preds,lat", [
    # 33 ops feed the same seven: 297 events at once, pending ops at the limit
    (8, [[]] * 33 + [list(range(33))] * 7, 5),
    (32, [[]] * 33 + [list(range(33))] * 7, 5),
    # 24 pairs across slow links: 144 events
    (33, [[]] * 24 + [[i] for i in range(24)], 1000),
    (256, [[]] * 24 + [[i] for i in range(24)], 1000),
])
def test_the_log_holds_what_a_generation_adds(D, preds, lat, arb):
    n = len(preds)
    d = mk(preds, [1 + i % 3 for i in range(n)], [64 + i for i in range(n)], n_dev=D, bw=100, lat=lat)
    for got, want in _run(d, 1, arb):
        compare(got, *want)


@pytest.mark.parametrize("arb", [False, True])
@pytest.mark.parametrize("D", [1, 8, 33, 256])
@pytest.mark.parametrize("roots,gap,succ", [
    (40, 10 ** 6, 5),    # roots far in the future
    (40, 10 ** 6, 33),   # as many pending ops as may wait beside them
    (90, 0, 0),          # more roots at once than ops may wait
    (90, 0, 20),
    (40, 3, 20),         # roots that come in while others run
])
def test_ops_without_predecessors_do_not_count_before_they_start(D, roots, gap, succ, arb):
    preds = [[] for _ in range(roots)] + [[0]] * succ
    n = len(preds)
    d = mk(preds, [5] * n, [1] * n, n_dev=D, bw=1, lat=1, release=[i * gap for i in range(roots)] + [0] * succ)
    for got, want in _run(d, 1, arb):
        compare(got, *want)


@pytest.mark.parametrize("D", [1, 8, 32])
def test_resumed_where_roots_start(D):
    """Arbitrated bases take checkpoints right before ops without predecessors
    start; moves of ops on both sides of them, with the base's queue_cap."""
    preds = [[] for _ in range(40)] + [[i] for i in range(40)]
    n = len(preds)
    d = mk(preds, [5] * n, [3] * n, n_dev=D, bw=1, lat=1, release=[i * 4 for i in range(40)] + [0] * 40)
    base = np.arange(n, dtype=np.uint8) % D
    mv = W.random_moves(3, 40, base, D, max_moves=3)
    g = G.gmg_create(d)
    for arb in (False, True):
        b = G.base_create(g, torch.from_numpy(base).cuda(), queue_cap=40, arbitrated=arb)
        inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True, queue_cap=40, arbitrated=arb)
        torch.cuda.synchronize()
        compare(inc.to_numpy(), *O.incremental_batch(d, base, mv, arbitrated=arb, resumed=arb))


def _late(queue_cap, late, D, successor=True):
    """32 ops at time 0, the first with as many successors as may wait, all
    released at 1e6; then `late` ops without predecessors, each with one more
    such successor (or none)."""
    preds = [[] for _ in range(32)] + [[0]] * (32 + queue_cap)
    rel = [0] * 32 + [10 ** 6] * (32 + queue_cap)
    for t in range(late):
        preds.append([])
        rel.append(1000 + 10 * t)
        if successor:
            preds.append([len(preds) - 1])
            rel.append(10 ** 6)
    n = len(preds)
    return mk(preds, [1] * n, [1] * n, n_dev=D, bw=1, lat=1, release=rel)


@pytest.mark.parametrize("arb", [False, True])
@pytest.mark.parametrize("D", [1, 8, 32, 33, 256])
@pytest.mark.parametrize("queue_cap", [1, 3, 100, 200])
@pytest.mark.parametrize("late,successor", [(0, True), (3, False), (1, True), (2, True), (40, True)])
def test_pending_ops_beyond_the_limit_are_never_dropped(D, queue_cap, late, successor, arb):
    """Ops that wait outside while all places are taken change places with the
    last pending one; none is lost."""
    d = _late(queue_cap, late, D, successor)
    spare = 1 if D <= 32 or arb else 0
    for got, want in _run(d, queue_cap, arb):
        if successor and late > spare:
            assert (got["status"] == G.SIM_QUEUE).all()
        elif successor and late:
            ok = got["status"] == 0
            assert ((got["status"] == G.SIM_QUEUE) | ok).all()
            if ok.any():
                compare(got, *(w[ok] for w in want), ks=np.flatnonzero(ok))
        else:
            compare(got, *want)
    for got, want in _run(d, queue_cap + late, arb):
        compare(got, *want)


@pytest.mark.parametrize("arb", [False, True])
@pytest.mark.parametrize("D", [1, 8, 33])
@pytest.mark.parametrize("late", [0, 1, 3])
def test_resumed_candidates_at_the_limit(D, late, arb):
    """The same against a base with room: moves of the late ops' successors, of
    the first op's and of the first op itself."""
    if arb and D > 32:
        pytest.skip("candidates of an arbitrated base: at most 32 accelerators")
    q = 100
    d = _late(q, late, D)
    n = d.n_ops
    base = np.arange(n, dtype=np.uint8) % D
    ops = [0, 40, n - 1]
    mv = W.Moves(np.arange(len(ops) + 1, dtype=np.int32), np.array(ops, np.int32),
                 ((base[ops] + 1) % D).astype(np.uint8))
    g = G.gmg_create(d)
    b = G.base_create(g, torch.from_numpy(base).cuda(), arbitrated=arb)
    dev = G.moves_to_device(mv, "cuda")
    at, room = [G.sim_incremental(g, b, *dev, queue_cap=c, arbitrated=arb) for c in (q, q + 50)]
    torch.cuda.synchronize()
    want = O.incremental_batch(d, base, mv, arbitrated=arb, resumed=arb)
    compare(room.to_numpy(), *want[:2])
    st = at.to_numpy()["status"]
    if D == 1:                            # no move has an effect: the base's results
        assert (st == 0).all()
    elif late == 0:
        assert st[0] == 0
    elif late > 1 or D > 32:
        assert (st == G.SIM_QUEUE).all()
    ok = st == 0
    for f in ("makespan", "score", "events"):
        assert (at.to_numpy()[f][ok] == want[0][f][ok]).all()
