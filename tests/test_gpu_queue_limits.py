"""The limits of a candidate's event queue (sim_opts_t.queue_cap): up to 32 +
queue_cap ops that became ready may wait, and a call beyond that answers
GMG_SIM_QUEUE; within it every result is the oracle's.  Ops without
predecessors do not count before they start, and the log of HBM events has room
for what one generation adds."""
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
