"""GPU parity of the selection at the batch sizes where the library changes kernels, and of the SLO
buckets' edges on catalogs whose bucket count differs."""
import numpy as np
import pytest

from oracle import OracleCatalog
from paper_1905_13348_b200 import workloads as W
from tests.test_gpu_parity import _to_dev, _to_host_u32, assert_state_equal, gpu_select

pytestmark = pytest.mark.gpu


# 96 K queries: one query per thread up to here where the image fits in shared memory; 192 K where it
# does not, and below it the fused window call tallies in the selection kernel; 160 K: tally by
# shared-memory histograms on these catalogs
@pytest.mark.parametrize("name,kw", [("C3", {}), ("C4", {}), ("C5", {"n_windows": 5})])
@pytest.mark.parametrize("n", [255, 257, 96 * 1024, 96 * 1024 + 1, 163839, 163840, 192 * 1024 - 1, 192 * 1024 + 1])
def test_batch_sizes_around_the_kernels_limits(name, kw, n):
    import paper_1905_13348_b200 as P
    import torch
    w = W.make(name, **(kw or {"n_queries": 2**18}))
    t, s, a = w.task[:n].copy(), w.slo_us[:n].copy(), w.min_acc_bp[:n].copy()
    t[:: max(1, n // 50)] = 65535                       # invalid ones among them
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    try:
        for _ in range(2):                              # the second window sees the first one's load
            want = o.select(t, s, a, 8)
            assert np.array_equal(_to_host_u32(gpu_select(cat, t, s, a)), want)
            dec = torch.empty(n, dtype=torch.int32, device="cuda")
            P.infaas_select_update(cat, _to_dev(t), _to_dev(s), _to_dev(a), dec, 40_000)
            torch.cuda.synchronize()
            assert np.array_equal(_to_host_u32(dec), want)
            o.load_update(want, 40_000)
            assert_state_equal(cat, o)
    finally:
        cat.free()


# both sides of every line where the bucket count changes: 48 KB of records at 4 / 5, 10 / 11 and 22 / 23
# tasks, 256 variants per task
@pytest.mark.parametrize("n_tasks,per_task,buckets", [
    (1, 1100, 2048), (4, 1100, 2048), (5, 1100, 1024), (10, 600, 1024), (11, 600, 512), (22, 300, 512), (23, 300, 256),
    (2, 300, 512), (24, 300, 256), (2, 257, 512), (2, 256, 256)])
def test_slos_at_every_latency_and_bucket_edge(n_tasks, per_task, buckets):
    import paper_1905_13348_b200 as P
    rng = np.random.default_rng(n_tasks)
    rows = W.tradeoff_catalog(rng, n_tasks, per_task)
    cat, o = P.infaas_catalog_load(rows, n_tasks), OracleCatalog(rows, n_tasks)
    try:
        assert P.infaas_catalog_get_info(cat)["slo_buckets"] == buckets
        edges = np.arange(0x3F800000 >> 16, 0x4F80, dtype=np.uint32) << 16     # every possible bucket's start
        edge = np.floor(edges.view(np.float32).astype(np.float64)).astype(np.uint64)
        v = np.unique(np.concatenate([edge, rows["lat_us"].astype(np.uint64), np.array([0, 1, 2**24, 2**32 - 1], np.uint64)]))
        v = np.unique(np.concatenate([v, v + np.uint64(1), v - np.minimum(v, np.uint64(1))])).clip(0, 2**32 - 1)
        slo = np.repeat(v.astype(np.uint32), 2)
        task = rng.integers(0, n_tasks, slo.size).astype(np.uint16)
        acc = rng.choice(np.concatenate([rows["acc_bp"], np.array([0], np.uint16)]), slo.size).astype(np.uint16)
        for _ in range(2):                              # the second rebuild's buckets cover the largest SLO
            want = o.select(task, slo, acc, 8)
            dec = gpu_select(cat, task, slo, acc)
            assert np.array_equal(_to_host_u32(dec), want)
            big = np.tile(np.arange(slo.size), 2**18 // slo.size + 1)              # the staging kernel too
            assert np.array_equal(_to_host_u32(gpu_select(cat, task[big], slo[big], acc[big])), want[big])
            P.infaas_load_update(cat, dec, 2_000)
            o.load_update(want, 2_000)
    finally:
        cat.free()


def test_image_that_outgrows_what_the_host_last_saw():
    """The staging kernel copies what the host expects the image to need and fetches the rest: windows
    that let the lists grow, without a look at the state in between."""
    import paper_1905_13348_b200 as P
    win, n_win = 120_000, 12
    w = W.make("C3", n_queries=n_win * win, window=win)
    cat, o = P.infaas_catalog_load(w.rows, w.n_tasks), OracleCatalog(w.rows, w.n_tasks)
    try:
        first = P.infaas_catalog_get_info(cat)["image_bytes"]
        grown = 0
        for k in range(n_win):
            s = slice(k * win, (k + 1) * win)
            want = o.select(w.task[s], w.slo_us[s], w.min_acc_bp[s], 8)
            dec = gpu_select(cat, w.task[s], w.slo_us[s], w.min_acc_bp[s])
            assert np.array_equal(_to_host_u32(dec), want), k
            info = P.infaas_catalog_get_info(cat)
            grown += first * 1.25 + 4096 < info["image_bytes"] <= info["image_smem"]
            P.infaas_load_update(cat, dec, 70_000)
            o.load_update(want, 70_000)
        print("grown", grown, first, info)
        assert grown > 0, (first, info)
    finally:
        cat.free()


# the small-batch kernel's two builds: 5 of its CTAs of 256 queries per SM, and one query more
@pytest.mark.parametrize("name,kw", [("C4", {}), ("C5", {"n_windows": 5})])
@pytest.mark.parametrize("over", [0, 1])
def test_small_batches_that_fill_the_chip(name, kw, over):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * 5 * 256 + over
    test_batch_sizes_around_the_kernels_limits(name, kw, n)
