"""GPU parity of the list rebuild at the sizes where its grid, its per-thread rows and its index
segments have edges: lists against the oracle's, decisions and load state through a few windows."""
import numpy as np
import pytest

from oracle import OracleCatalog
from paper_1905_13348_b200 import workloads as W
from tests.helpers import rows_from
from tests.test_gpu_parity import assert_state_equal, run_both
from tests.test_gpu_stateful import _states, run_stateful

pytestmark = pytest.mark.gpu

# rows and columns of the grid hold 16 variants up to 1024 variants, 32 up to 2048 and so on; a
# thread has one variant up to 1024; 8192 is the limit
SIZES = [1, 15, 17, 31, 33, 255, 257, 512, 1023, 1025, 2049, 8192]


def _workload(V, kind, n=6000, window=1999):
    rng = np.random.default_rng([V, len(kind)])
    sizes = [V, 0, max(1, V // 3)]
    task = np.repeat(np.arange(3), sizes)
    N = task.size
    lat = np.exp(rng.uniform(np.log(500.0), np.log(2e6), N)).astype(np.int64)
    batch = rng.choice([1, 2, 7, 64, 65535], N)
    if kind == "ties":                    # few costs, accuracies and latencies: runs of equal (cost, accuracy)
        cost, acc = rng.integers(1, 4, N), 7000 + 30 * rng.integers(0, 5, N)
        lat = rng.choice([1000, 4000, 20_000, 20_001], N)
        queued = rng.choice([0, 0, 5], N)
    elif kind == "one":                   # a single cost and accuracy
        cost, acc, queued = np.full(N, 9), np.full(N, 8000), rng.integers(0, 3, N)
    elif kind == "saturated":             # predicted latencies of 2^32-2 and 2^32-1 among ordinary ones
        cost, acc = rng.integers(1, 500, N), rng.integers(0, 10001, N)
        pick = rng.random(N)
        lat = np.where(pick < 0.4, 2**32 - 2, np.where(pick < 0.8, 2**32 - 1, lat))
        queued = rng.choice([0, 0, 0, 2**32 - 1], N)
    else:                                 # a trade-off: long lists
        cost = (4e7 / lat**0.6 * np.exp(0.2 * rng.standard_normal(N))).astype(np.int64) + 1
        acc = np.clip(3000 + 900 * np.log10(lat) + 150 * rng.standard_normal(N), 0, 10000).astype(np.int64)
        queued = np.zeros(N, np.int64)
    rows = rows_from(task, batch, lat, acc, cost, queued)
    rows = rows[rng.permutation(N)].copy()
    q_task = rng.choice([0, 0, 0, 1, 2, 3], n).astype(np.uint16)
    q_slo = np.exp(rng.uniform(np.log(300.0), np.log(4.2e9), n)).astype(np.uint64).clip(0, 2**32 - 1).astype(np.uint32)
    q_slo[::97] = 2**32 - 2
    q_acc = rng.choice(np.concatenate([rows["acc_bp"], [0, 9999]]), n).astype(np.uint16)
    return W.Workload(f"{kind}{V}", 3, rows, q_task, q_slo, q_acc, window, 3_000, "edges of the rebuild")


@pytest.mark.parametrize("kind", ["ties", "one", "saturated", "tradeoff"])
@pytest.mark.parametrize("V", SIZES)
def test_lists_and_decisions_at_the_edges(V, kind):
    import paper_1905_13348_b200 as P
    w = _workload(V, kind)
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    try:
        assert_state_equal(cat, o)
        for t in range(w.n_tasks):
            assert np.array_equal(P.infaas_catalog_get_frontier(cat, t), o.frontier(t)), t
    finally:
        cat.free()
    run_both(w)


@pytest.mark.parametrize("kind", ["ties", "saturated", "tradeoff"])
@pytest.mark.parametrize("V", [17, 257, 1025, 8192])
def test_two_lists_at_the_edges(V, kind):
    w = _workload(V, kind)
    rng = np.random.default_rng(V)
    load = rng.choice(np.array([0, 1, 5000, 2**32 - 1], np.uint32), w.n_variants)
    run_stateful(w, _states(rng, w.n_variants, (0.45, 0.45, 0.05, 0.05)), load)


# A thread per variant up to 256 and up to 512 variants per task: the sizes on either side, lists of one and of
# two segments (248 entries), equal costs and accuracies across the groups of 32, both kinds of catalog
@pytest.mark.parametrize("kind", ["ties", "saturated", "tradeoff"])
@pytest.mark.parametrize("V", [32, 248, 249, 256, 511, 513])
def test_a_thread_per_variant(V, kind):
    w = _workload(V, kind)
    run_both(w)
    rng = np.random.default_rng(V)
    load = rng.choice(np.array([0, 1, 5000, 2**32 - 1], np.uint32), w.n_variants)
    run_stateful(w, _states(rng, w.n_variants, (0.45, 0.45, 0.05, 0.05)), load)


# Lists of every variant: 7 and 34 segments, so that with four CTAs per task (3 tasks; 33 is the last
# number of tasks for which all clusters run at once) a CTA indexes several of them, and with one (34) all
@pytest.mark.parametrize("states", [False, True])
@pytest.mark.parametrize("V,n_tasks", [(1500, 3), (1500, 33), (1500, 34), (8192, 3)])
def test_lists_of_many_segments(V, n_tasks, states):
    import paper_1905_13348_b200 as P
    rng = np.random.default_rng([V, n_tasks])
    i = np.concatenate([np.arange(V), np.arange(V)] + [np.arange(3)] * (n_tasks - 2))
    task = np.concatenate([np.zeros(V), np.ones(V), np.repeat(np.arange(2, n_tasks), 3)]).astype(np.int64)
    # slower is cheaper and more accurate: nothing is dominated
    rows = rows_from(task, np.full(i.size, 64), 1000 + 37 * i, 1 + i * 9998 // V, 5 + 11 * (V - i), None)
    rows = rows[rng.permutation(rows.size)].copy()
    n = 4000
    q_task = rng.choice([0, 0, 1, 1, 2, n_tasks], n).astype(np.uint16)
    q_slo = np.exp(rng.uniform(np.log(500.0), np.log(80.0 * V), n)).astype(np.uint32)
    q_acc = rng.integers(0, 10_001, n).astype(np.uint16)
    w = W.Workload(f"segments{V}", n_tasks, rows, q_task, q_slo, q_acc, 1333, 3_000, "lists of many segments")
    cat = P.infaas_catalog_load(rows, n_tasks)
    try:
        assert P.infaas_catalog_get_info(cat)["longest_list"] == V
        if states:
            state = _states(rng, rows.size, (0.45, 0.45, 0.05, 0.05))
            load = np.zeros(rows.size, np.uint32)
            P.infaas_catalog_set_states(cat, state, load)
            assert P.infaas_catalog_get_info(cat)["longest_list"] > 0.85 * V > 1000
    finally:
        cat.free()
    if states:
        run_stateful(w, state, load)
    else:
        run_both(w)


# Beside a task of more than 1024 variants, which brings four CTAs for every task, tasks so small that some of
# the four have no variants: every list after every window, with and without states.
SMALL = [1, 3, 10, 31, 33, 37, 63, 70, 95, 100, 130, 255, 260, 287]


def _lists(o, state, load):
    """Every task's list at the oracle's present load: Active variants, then (with states) Inactive ones."""
    if state is None:
        return [o.frontier(t) for t in range(o.n_tasks)]
    active = np.flatnonzero(state == 1)
    a = OracleCatalog(o.rows[active], o.n_tasks)
    a.queued = o.queued[active].copy()
    eff = np.minimum(o.pred_lat().astype(np.int64) + load, 2**32 - 1)
    out = []
    for t in range(o.n_tasks):
        ids, best = list(active[a.frontier(t)]) if active.size else [], -1
        rest = np.flatnonzero((o.rows["task"] == t) & (state == 0))
        for v in rest[np.lexsort((rest, -o.rows["acc_bp"][rest].astype(np.int64), eff[rest]))]:
            if int(o.rows["acc_bp"][v]) > best:
                best = int(o.rows["acc_bp"][v])
                ids.append(v)
        out.append(np.array(ids, np.uint32))
    return out


@pytest.mark.parametrize("states", [False, True])
@pytest.mark.parametrize("kind", ["ties", "tradeoff"])
@pytest.mark.parametrize("V", [1025, 1999])
def test_small_tasks_beside_large_ones(V, kind, states):
    import torch

    import paper_1905_13348_b200 as P
    from oracle import StatefulOracleCatalog
    from tests.test_gpu_parity import _to_dev, _to_host_u32
    rng = np.random.default_rng([V, len(kind), states])
    sizes = [V] + SMALL
    T, task = len(sizes), np.repeat(np.arange(len(sizes)), sizes)
    N, windows, n = task.size, 120, 1500
    lat = np.exp(rng.uniform(np.log(500.0), np.log(2e6), N)).astype(np.int64)
    if kind == "ties":
        cost, acc, lat = rng.integers(1, 4, N), 7000 + 30 * rng.integers(0, 5, N), rng.choice([1000, 4000, 20_000, 20_001], N)
    else:
        cost = (4e7 / lat**0.6 * np.exp(0.2 * rng.standard_normal(N))).astype(np.int64) + 1
        acc = np.clip(3000 + 900 * np.log10(lat) + 150 * rng.standard_normal(N), 0, 10000).astype(np.int64)
    rows = rows_from(task, rng.choice([1, 2, 7, 64], N), lat, acc, cost, None)
    rows = rows[rng.permutation(N)].copy()
    load = rng.choice(np.array([0, 1, 5000, 2**32 - 1], np.uint32), N)
    state = _states(rng, N, (0.45, 0.45, 0.05, 0.05)) if states else None
    cat = P.infaas_catalog_load(rows, T)
    o = StatefulOracleCatalog(rows, T, state, load) if states else OracleCatalog(rows, T)
    if states:
        P.infaas_catalog_set_states(cat, state, load)
    d = torch.empty(n, dtype=torch.int32, device="cuda")
    try:
        for w in range(windows):
            for t, want in enumerate(_lists(o, o.state if states else None, load)):
                got = P.infaas_catalog_get_frontier(cat, t)
                assert np.array_equal(got, want), (w, t, sizes[t], got[:5], want[:5])
            q = (rng.integers(0, T, n).astype(np.uint16),
                 np.exp(rng.uniform(np.log(300.0), np.log(4e6), n)).astype(np.uint32),
                 rng.choice(rows["acc_bp"], n).astype(np.uint16))
            P.infaas_select_update(cat, *map(_to_dev, q), d, 3000)
            want = o.select(*q, 8)
            assert np.array_equal(_to_host_u32(d), want), w
            o.load_update(want, 3000)
    finally:
        cat.free()


def _image_bytes(rows, lists, lat, n_buckets):
    """Size of the image for these lists (layout in common.cuh): no block is larger than its tables."""
    T, up = len(lists), lambda x, a: -(-x // a) * a
    lo, hi = int(rows["acc_bp"].min()) // 24 * 24, int(rows["acc_bp"].max())
    nbw = (hi + 1 - lo) // 24 + 1
    size = up(up(64 + 4 * (T + 1), 128) + 4 * (n_buckets + 1) * (T + 1) + 4 * (nbw | 1) * (T + 1), 64)
    for ids in lists:
        for at in range(0, len(ids), 248):
            seg = ids[at:at + 248]
            F, Ks, Ka = len(seg), len(set(lat[seg].tolist())), len(set(rows["acc_bp"][seg].tolist()))
            slow = up(8 * F + 8 * (Ka + 1) + 4 * Ks + 4 * (Ks + 1) + Ks + 1, 8)
            block = up(4 * (F + 1) + (Ks + 3) * (Ka + 1), 4) + (4 * nbw if at else 0)
            size += up(up(block, 8) + slow, 16)
    return size


# Few distinct latencies, as a profile in whole milliseconds has them, and nothing dominated (cheaper is less
# accurate): lists of 2, 3, 5 and 9 segments.  One CTA of 256, 512 and 1024 threads per task, and four
@pytest.mark.parametrize("n_tasks,V", [(40, 256), (20, 512), (8, 1000), (3, 1999)])
def test_blocks_of_the_image_are_as_large_as_their_tables(n_tasks, V):
    import paper_1905_13348_b200 as P
    rng = np.random.default_rng(V)
    i, task = np.tile(np.arange(V), n_tasks), np.repeat(np.arange(n_tasks), V)
    rows = rows_from(task, np.full(i.size, 8), 1000 * rng.integers(1, 40, i.size), 7000 + i, 5 + 11 * i, None)
    cat, o = P.infaas_catalog_load(rows, n_tasks), OracleCatalog(rows, n_tasks)
    try:
        lists = [o.frontier(t) for t in range(n_tasks)]
        assert [len(x) for x in lists] == [V] * n_tasks
        info = P.infaas_catalog_get_info(cat)
        assert info["image_bytes"] == _image_bytes(rows, lists, o.pred_lat(), info["slo_buckets"])
    finally:
        cat.free()
