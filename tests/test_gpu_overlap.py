"""Order between overlapping kernels: every launch of the library may start while its predecessor in
the stream still runs, so what a kernel reads -- queries written by a kernel just before it, decisions,
tables, the image of the last rebuild -- has to be waited for.  Side streams, hand-overs between
streams, catalogs interleaved on one stream, replayed graphs and repeated loads, against the oracle."""
import numpy as np
import pytest

from oracle import OracleCatalog, StatefulOracleCatalog, assign_workers, autoscale_step
from paper_1905_13348_b200 import workloads as W
from tests.test_gpu_parity import _to_dev, _to_host_u32, assert_state_equal, gpu_select

pytestmark = pytest.mark.gpu

# one query per thread with fused tallies; the staging kernel with fused tallies; separate tallies
WINDOWS = [4_099, 120_001, 200_003]


def _torch():
    import torch
    return torch


class Feed:
    """A workload's windows on the GPU; `next` writes one into the same three arrays with kernels of the
    current stream, right behind a fill that would give other decisions."""

    def __init__(self, w, n):
        torch = _torch()
        self.src = [(_to_dev(w.task[k:k + n]), _to_dev(w.slo_us[k:k + n]), _to_dev(w.min_acc_bp[k:k + n]))
                    for k in range(0, w.n_queries - n + 1, n)]
        self.buf = [torch.empty_like(a) for a in self.src[0]]

    def next(self, k):
        for b, a in zip(self.buf, self.src[k % len(self.src)]):
            b.fill_(-1)
            b.copy_(a)
        return self.buf


def _tables(rng, rows):
    nv = rows.size
    iv = rng.integers(0, nv, nv).astype(np.uint32)
    return (iv, rng.integers(0, 50, nv).astype(np.uint32), rng.integers(0, 99, nv).astype(np.uint32),
            rng.integers(0, 4, 50).astype(np.uint8), rng.integers(0, 99, 50).astype(np.uint32))


@pytest.mark.parametrize("n", WINDOWS)
def test_side_stream_behind_torch_kernels(n):
    import paper_1905_13348_b200 as P
    torch = _torch()
    w = W.make("C3", n_queries=4 * n, window=n)
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    tables = _tables(np.random.default_rng(n), w.rows)
    side = torch.cuda.Stream()
    try:
        with torch.cuda.stream(side):
            feed = Feed(w, n)
            P.infaas_workers_config(cat, *tables)
            dec, wrk = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
            got = []
            for k in range(4):
                t, s, a = feed.next(k)
                dec.fill_(0)
                if k % 2:
                    P.infaas_select_update(cat, t, s, a, dec, w.window_us)
                else:
                    P.infaas_select_batch(cat, t, s, a, dec)
                    P.infaas_load_update(cat, dec, w.window_us)
                wrk.fill_(0)
                P.infaas_assign_workers(cat, dec, wrk)
                got.append((dec.clone(), wrk.clone()))
        side.synchronize()
        for k in range(4):
            s = slice(k * n, (k + 1) * n)
            want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
            o.load_update(want, w.window_us)
            assert np.array_equal(_to_host_u32(got[k][0]), want), k
            assert np.array_equal(_to_host_u32(got[k][1]), assign_workers(w.rows, *tables, want)), k
        assert_state_equal(cat, o)
    finally:
        cat.free()


@pytest.mark.parametrize("n", WINDOWS)
def test_two_catalogs_interleaved_on_one_stream(n):
    import paper_1905_13348_b200 as P
    torch = _torch()
    ws = [W.make("C3", n_queries=3 * n, window=n), W.make("C5", n_windows=3, window=n)]
    cats = [P.infaas_catalog_load(w.rows, w.n_tasks) for w in ws]
    oracles = [OracleCatalog(w.rows, w.n_tasks) for w in ws]
    try:
        feeds = [Feed(w, n) for w in ws]
        dec = torch.empty(n, dtype=torch.int32, device="cuda")      # shared: the next catalog's call overwrites it
        got = []
        for k in range(3):
            for cat, feed, w in zip(cats, feeds, ws):
                P.infaas_select_update(cat, *feed.next(k), dec, w.window_us)
                got.append(dec.clone())
        torch.cuda.synchronize()
        for k in range(3):
            for i, (o, w) in enumerate(zip(oracles, ws)):
                s = slice(k * n, (k + 1) * n)
                want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
                o.load_update(want, w.window_us)
                assert np.array_equal(_to_host_u32(got[2 * k + i]), want), (k, i)
        for cat, o in zip(cats, oracles):
            assert_state_equal(cat, o)
    finally:
        for cat in cats:
            cat.free()


@pytest.mark.parametrize("n", WINDOWS)
def test_hand_over_between_streams(n):
    """Selection on one stream, tallies and the load advance on another, joined by events only."""
    import paper_1905_13348_b200 as P
    torch = _torch()
    w = W.make("C3", n_queries=4 * n, window=n)
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        feed = Feed(w, n)
        dec = torch.empty(n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        got = []
        for k in range(4):
            with torch.cuda.stream(a):
                a.wait_stream(b)
                P.infaas_select_batch(cat, *feed.next(k), dec)
            with torch.cuda.stream(b):
                b.wait_stream(a)
                P.infaas_tally(cat, dec)
                P.infaas_advance(cat, w.window_us)
                got.append(dec.clone())
        torch.cuda.synchronize()
        for k in range(4):
            s = slice(k * n, (k + 1) * n)
            want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
            o.load_update(want, w.window_us)
            assert np.array_equal(_to_host_u32(got[k]), want), k
        assert_state_equal(cat, o)
    finally:
        cat.free()


@pytest.mark.parametrize("n", WINDOWS)
@pytest.mark.parametrize("fork", [False, True])
def test_captured_window_replayed(n, fork):
    """A window of the control loop as a graph, behind fills and copies; with `fork` the worker choice
    runs on a second stream of the capture and the load advance waits for it."""
    import paper_1905_13348_b200 as P
    torch = _torch()
    w = W.make("C3", n_queries=4 * n, window=n)
    rng = np.random.default_rng(n)
    state, load = W.variant_states(w.n_variants)
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), StatefulOracleCatalog(w.rows, w.n_tasks, state, load)
    tables = _tables(rng, w.rows)
    inst, slo = rng.integers(0, 2, w.n_variants).astype(np.uint32), rng.integers(20_000, 200_000, w.n_tasks).astype(np.uint32)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    try:
        P.infaas_catalog_set_states(cat, state, load)
        P.infaas_autoscale_config(cat, inst, slo)
        P.infaas_workers_config(cat, *tables)
        feed = Feed(w, n)
        inputs = [torch.empty_like(x) for x in feed.buf]
        dec, wrk = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
        act = [torch.empty(w.n_tasks, dtype=torch.int32, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=main):
            for b, x in zip(inputs, feed.buf):
                b.zero_()
                b.copy_(x)
            dec.zero_()
            P.infaas_select_batch(cat, *inputs, dec)
            if fork:
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    P.infaas_assign_workers(cat, dec, wrk)
            P.infaas_tally(cat, dec)
            P.infaas_autoscale_step(cat, w.window_us, 105, 100, *act)
            if fork:
                main.wait_stream(side)
            else:
                P.infaas_assign_workers(cat, dec, wrk)
            P.infaas_advance(cat, w.window_us)
        got = []
        for k in range(4):
            feed.next(k)
            graph.replay()
            got.append([x.clone() for x in (dec, wrk, *act)])
        torch.cuda.synchronize()
        for k in range(4):
            s = slice(k * n, (k + 1) * n)
            want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
            assert np.array_equal(_to_host_u32(got[k][0]), want), k
            assert np.array_equal(_to_host_u32(got[k][1]), assign_workers(w.rows, *tables, want)), k
            counts = np.bincount(want[want < w.n_variants], minlength=w.n_variants).astype(np.uint32)
            var, delta = autoscale_step(w.rows, w.n_tasks, counts, inst, load, slo, w.window_us, 105, 100)
            assert np.array_equal(_to_host_u32(got[k][2]), var) and np.array_equal(_to_host_u32(got[k][3]), delta), k
            o.load_update(want, w.window_us)
        assert_state_equal(cat, o)
        assert np.array_equal(P.infaas_catalog_get_states(cat), o.state)
    finally:
        del graph
        cat.free()


@pytest.mark.parametrize("n", WINDOWS)
def test_bucket_scale_that_changes_between_windows(n):
    """Larger SLOs from window to window: each rebuild publishes another bucket scale, and the selection
    right behind it must not see the one before."""
    import paper_1905_13348_b200 as P
    torch = _torch()
    w = W.make("C3", n_queries=6 * n, window=n)
    rng = np.random.default_rng(n)
    for k in range(6):
        s = slice(k * n, (k + 1) * n)
        w.slo_us[s][::7] = rng.integers(1000, 1 << (18 + 2 * k), w.slo_us[s][::7].size)
        w.slo_us[s][0] = (1 << (20 + 2 * k)) + 1
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    try:
        feed = Feed(w, n)
        dec = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(6)]
        torch.cuda.synchronize()
        for k in range(6):                       # nothing but the library's kernels on the stream
            P.infaas_select_update(cat, *feed.src[k], dec[k], w.window_us)
        torch.cuda.synchronize()
        for k in range(6):
            s = slice(k * n, (k + 1) * n)
            want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
            o.load_update(want, w.window_us)
            assert np.array_equal(_to_host_u32(dec[k]), want), k
        assert_state_equal(cat, o)
    finally:
        cat.free()


def test_select_right_behind_many_loads():
    """The first lists are built from a layout made by a kernel just before."""
    import paper_1905_13348_b200 as P
    rng = np.random.default_rng(4)
    n = 3000
    for k in range(60):
        T = int(rng.integers(1, 40))
        rows = W.structured_catalog(rng, T, int(rng.integers(1, 9)), 4, [1, 2, 4, 8], queued_hi=3) if k % 3 else \
            W.tradeoff_catalog(rng, T, int(rng.integers(1, 300)))
        task = rng.integers(0, T, n).astype(np.uint16)
        slo = np.exp(rng.uniform(np.log(1e3), np.log(1e6), n)).astype(np.uint32)
        acc = rng.choice(rows["acc_bp"], n).astype(np.uint16)
        cat = P.infaas_catalog_load(rows, T)
        try:
            want = OracleCatalog(rows, T).select(task, slo, acc, 8)
            assert np.array_equal(_to_host_u32(gpu_select(cat, task, slo, acc)), want), k
        finally:
            cat.free()
