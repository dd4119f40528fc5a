"""GPU parity of the sweep of pending READY ops and of the HBM accounting where
they can go wrong: more pending ops than lanes or pool slots, more startable ops
than lanes, equal times, batches that share accelerators, capacities that bind,
sizes beyond 48 bits, 64-bit times; against the oracle, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import compare, oracle_rows, torch_place  # noqa: E402
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


def _chains(seed, chains, length, D, dur_hi=20, bytes_lo=1, bytes_hi=1 << 20, cap=None, release_hi=0, fan=1):
    """Independent chains; with fan > 1 every op feeds `fan` ops of the next
    level of its chain and one op joins them."""
    g = np.random.default_rng(seed)
    preds, rel = [], []
    for c in range(chains):
        last = []
        r = int(g.integers(0, release_hi + 1))
        for _ in range(length):
            first = len(preds)
            preds.append(last)
            rel.append(r if not last else 0)
            if fan > 1:
                for _ in range(fan):
                    preds.append([first])
                    rel.append(0)
                preds.append(list(range(first + 1, first + 1 + fan)))
                rel.append(0)
            last = [len(preds) - 1]
    n = len(preds)
    return mk(preds, g.integers(1, dur_hi + 1, n), g.integers(bytes_lo, bytes_hi + 1, n), n_dev=D, bw=1000, lat=2,
              release=rel, req_id=[0] * n, deadline=[1000], cap=None if cap is None else [cap] * D)


def _rows(seed, K, n, D):
    rows = np.zeros((K, W.placement_ld(n)), np.uint8)
    rows[:, :n] = np.random.default_rng(seed).integers(0, D, (K, n))
    rows[-1, :n] = 0
    return rows


@pytest.mark.parametrize("D", [1, 2, 8, 32, 33, 256])
@pytest.mark.parametrize("kw", [
    dict(chains=33, length=6),                                   # one more chain than lanes
    dict(chains=161, length=4),                                  # one more than pool slots
    dict(chains=400, length=2, dur_hi=1),                        # lockstep: every op startable at once
    dict(chains=70, length=5, release_hi=60, dur_hi=4),          # roots that come in while the pool is full
    dict(chains=9, length=4, fan=5),                             # joins, long lists
    dict(chains=20, length=6, bytes_lo=1 << 18, cap=6 << 20),    # capacities that bind
    dict(chains=5, length=5, bytes_lo=1 << 48, bytes_hi=1 << 50),  # sizes beyond 48 bits
    dict(chains=30, length=6, dur_hi=1 << 29),                   # 64-bit times
    dict(chains=30, length=6, release_hi=3_900_000_000),         # 32-bit times beyond 2^31
])
def test_pending_ops_and_accounting(D, kw):
    d = _chains(7, D=D, **kw)
    rows = _rows(8, 13, d.n_ops, D)
    g = G.gmg_create(d)
    tk = torch.tensor([0, 12], dtype=torch.int32, device="cuda")
    out = G.sim_batch(g, torch_place(rows), req_done=True, trace_k=tk)
    base = rows[0, :d.n_ops].copy()
    mv = W.random_moves(9, 40, base, D, max_moves=5)
    b = G.base_create(g, torch.from_numpy(base).cuda())
    inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True)
    torch.cuda.synchronize()
    got = out.to_numpy()
    compare(got, *oracle_rows(d, rows))
    for slot, k in enumerate((0, 12)):
        r = O.simulate(d, rows[k])
        assert np.array_equal(got["trace_start"][slot], r["start"])
        assert np.array_equal(got["trace_finish"][slot], r["finish"])
    compare(inc.to_numpy(), *O.incremental_batch(d, base, mv))


@pytest.mark.parametrize("K", [1, 130])
def test_two_warps_one_warp_and_staged_give_the_same(K):
    """Two warps per candidate (the default for few), one warp and the staged copy."""
    wl = W.config2()
    rows = wl.full_rows(range(K))
    g = G.gmg_create(wl.desc)
    place = torch_place(rows)
    outs = [G.sim_batch(g, place, req_done=True, **kw)
            for kw in ({}, dict(warps_per_block=4), dict(gmg_staging=G.GMG_STAGING_SHARED))]
    torch.cuda.synchronize()
    for o in outs:
        compare(o.to_numpy(), *oracle_rows(wl.desc, rows))


@pytest.mark.parametrize("D", [2, 32, 33, 256])
@pytest.mark.parametrize("kw", [
    dict(chains=300, length=3, dur_hi=1, bytes_lo=4096, bytes_hi=4096),  # transfers that complete together
    dict(chains=80, length=4, dur_hi=1, release_hi=2, bytes_lo=0, bytes_hi=1 << 12),
    dict(chains=9, length=4, fan=5),                                       # several destinations per op
    dict(chains=40, length=4, dur_hi=1 << 29),                             # 64-bit times
    dict(chains=40, length=4, release_hi=3_900_000_000),                   # 32-bit times beyond 2^31
])
def test_arbitrated_events_at_one_time(D, kw):
    """More pending ops than lanes, and more completions and intents at one time
    than are looked up at once."""
    d = _chains(17, D=D, **kw)
    rows = _rows(18, 9, d.n_ops, D)
    g = G.gmg_create(d)
    out = G.sim_batch(g, torch_place(rows), req_done=True, arbitrated=True)
    base = rows[0, :d.n_ops].copy()
    mv = W.random_moves(19, 24, base, D, max_moves=5)
    b = G.base_create(g, torch.from_numpy(base).cuda(), arbitrated=D <= 32)
    inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True, arbitrated=True)
    torch.cuda.synchronize()
    compare(out.to_numpy(), *O.simulate_batch(d, rows, arbitrated=True))
    compare(inc.to_numpy(), *O.incremental_batch(d, base, mv, arbitrated=True), check_events=D > 32)


@pytest.mark.parametrize("D", [8, 64])
@pytest.mark.parametrize("more", [0, 1])
def test_both_sides_of_the_two_warp_line(D, more):
    """As many candidates as fit with two warps each, and one more."""
    d = _chains(27, D=D, chains=5, length=4, fan=2, bytes_lo=1 << 18, cap=6 << 20)
    g = G.gmg_create(d)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K = 14 * sms + more
    rows = _rows(28, K, d.n_ops, D)
    out = G.sim_batch(g, torch_place(rows), req_done=True)
    base = rows[0, :d.n_ops].copy()
    mv = W.random_moves(29, K, base, D, max_moves=4)
    mv.dev[mv.off[2]:mv.off[3]] = D               # written without the second warp
    b = G.base_create(g, torch.from_numpy(base).cuda())
    inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True)
    torch.cuda.synchronize()
    compare(out.to_numpy(), *oracle_rows(d, rows))
    compare(inc.to_numpy(), *O.incremental_batch(d, base, mv))


@pytest.mark.parametrize("more", [0, 1])
def test_both_sides_of_the_wide_arbitrated_line(more):
    """As many candidates as the instance with four blocks per SM holds, and one more."""
    d = _chains(30, D=33, chains=5, length=4, fan=2, bytes_lo=1 << 18, cap=6 << 20)
    g = G.gmg_create(d)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K = 16 * sms + more
    rows = _rows(31, K, d.n_ops, 33)
    out = G.sim_batch(g, torch_place(rows), req_done=True, arbitrated=True)
    torch.cuda.synchronize()
    compare(out.to_numpy(), *O.simulate_batch(d, rows, arbitrated=True))


@pytest.mark.parametrize("K", [1, 32, 33, 1024, 1025, 4096, 4097])
def test_select_best_on_both_sides_of_one_block(K):
    g = np.random.default_rng(K)
    out = G.SimOut.empty(K, 1, 1, "cuda")
    st = (g.random(K) < 0.2).astype(np.int32)
    vf = (g.random(K) < 0.3).astype(np.int32)
    sc, ms = g.integers(0, max(2, K // 2), K), g.integers(0, 3, K).astype(np.int32)
    for t, a in ((out.status, st), (out.viol_flag, vf), (out.score, sc), (out.sla_miss, ms)):
        t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    for mode in (0, 1):
        ok = [(int(ms[k]) if mode else 0, int(sc[k]), k) for k in range(K) if st[k] == 0 and vf[k] == 0]
        want = [min(ok)[2], min(ok)[1]] if ok else [-1, np.iinfo(np.int64).max]
        assert G.select_best(out, score_mode=mode).cpu().tolist() == want


@pytest.mark.parametrize("D", [33, 64, 256])
@pytest.mark.parametrize("kw", [
    dict(chains=40, length=5),
    dict(chains=170, length=2),                                   # more pending ops than pool slots
    dict(chains=9, length=4, fan=5, bytes_lo=1 << 18, cap=6 << 20),  # joins, capacities that bind
    dict(chains=30, length=5, release_hi=1 << 41),
])
def test_wide_graphs_whose_keys_leave_no_room_for_the_accelerator(D, kw):
    """Times so wide that an HBM event's accelerator is kept beside its key:
    the pool with events applied one at a time, full placements and moves."""
    d = _chains(41, D=D, dur_hi=1 << 40, **kw)
    rows = _rows(42, 9, d.n_ops, D)
    g = G.gmg_create(d)
    assert g.info["batched_sweep"] == 0 and g.info["t32"] == 0
    tk = torch.tensor([0, 8], dtype=torch.int32, device="cuda")
    out = G.sim_batch(g, torch_place(rows), req_done=True, trace_k=tk)
    base = rows[0, :d.n_ops].copy()
    mv = W.random_moves(43, 24, base, D, max_moves=5)
    b = G.base_create(g, torch.from_numpy(base).cuda())
    inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True)
    torch.cuda.synchronize()
    got = out.to_numpy()
    compare(got, *oracle_rows(d, rows))
    for slot, k in enumerate((0, 8)):
        r = O.simulate(d, rows[k])
        assert np.array_equal(got["trace_start"][slot], r["start"])
        assert np.array_equal(got["trace_finish"][slot], r["finish"])
    compare(inc.to_numpy(), *O.incremental_batch(d, base, mv))
    with pytest.raises(G.GmgError) as e:
        G.sim_batch(g, torch_place(rows), arbitrated=True)
    assert e.value.code == G.GMG_ERANGE


@pytest.mark.parametrize("K", [2048, 2049])
def test_select_best_at_the_line(K):
    test_select_best_on_both_sides_of_one_block(K)


@pytest.mark.parametrize("D", [1, 2, 3, 32])
@pytest.mark.parametrize("kw", [
    dict(chains=1, length=40),                                    # one op at a time
    dict(chains=1, length=12, fan=40),                            # one op with more successors than lanes
    dict(chains=3, length=10, fan=3, bytes_lo=1 << 18, cap=6 << 20),  # capacities that bind
    dict(chains=33, length=6),
])
def test_staged_and_one_warp_on_few_accelerators(D, kw):
    """One warp per candidate, staged and through L1: batches of one op, and drains
    ordered without sums on one or two accelerators."""
    d = _chains(34, D=D, **kw)
    rows = _rows(35, 40, d.n_ops, D)
    g = G.gmg_create(d)
    place = torch_place(rows)
    outs = [G.sim_batch(g, place, req_done=True, **o)
            for o in (dict(warps_per_block=4), dict(gmg_staging=G.GMG_STAGING_SHARED))]
    torch.cuda.synchronize()
    for o in outs:
        compare(o.to_numpy(), *oracle_rows(d, rows))


@pytest.mark.parametrize("D", [2, 8])
@pytest.mark.parametrize("blocks,more", [(5, 0), (5, 1), (6, 0), (6, 1), (7, 0), (7, 1)])
def test_both_sides_of_the_arbitrated_lines(D, blocks, more):
    """As many candidates as the instances with 5, 6 and 7 blocks per SM hold, and
    one more."""
    d = _chains(32, D=D, chains=3, length=4, fan=2)
    g = G.gmg_create(d)
    K = 4 * blocks * torch.cuda.get_device_properties(0).multi_processor_count + more
    rows = _rows(33, K, d.n_ops, D)
    out = G.sim_batch(g, torch_place(rows), req_done=True, arbitrated=True)
    torch.cuda.synchronize()
    compare(out.to_numpy(), *O.simulate_batch(d, rows, arbitrated=True))


@pytest.mark.parametrize("D", [16, 17, 32])
@pytest.mark.parametrize("kw", [dict(n_types=2), dict(link_hetero=True), dict(n_types=2, dur_hi=1 << 30)])
def test_drains_summed_in_one_part_and_in_four(D, kw):
    """Graphs without compact records on both sides of 16 accelerators, with a
    capacity that binds."""
    d = W.random_desc(51, 400, D, window=80, **kw)
    rows = _rows(52, 24, d.n_ops, D)
    d.cap[:] = int(np.median(oracle_rows(d, rows)[1].max(axis=1)))   # half of the placements exceed it
    g = G.gmg_create(d)
    outs = [G.sim_batch(g, torch_place(rows), req_done=True, warps_per_block=w) for w in (0, 4)]
    base = rows[0, :d.n_ops].copy()
    mv = W.random_moves(53, 24, base, D, max_moves=5)
    b = G.base_create(g, torch.from_numpy(base).cuda())
    inc = G.sim_incremental(g, b, *G.moves_to_device(mv, "cuda"), req_done=True)
    torch.cuda.synchronize()
    want = oracle_rows(d, rows)
    for o in outs:
        compare(o.to_numpy(), *want)
    compare(inc.to_numpy(), *O.incremental_batch(d, base, mv))
