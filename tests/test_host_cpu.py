"""The host side of the C ABI without a GPU: csrc/api.cu compiled as plain C++ against a stand-in for
the CUDA runtime and the kernel launchers (host_runtime.cpp) that writes down what is called."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_1905_13348_b200 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1905_13348_b200", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "host.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-x", "c++",
                           "-I", "/usr/local/cuda/include", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           os.path.join(CSRC, "api.cu"), os.path.join(HERE, "host_runtime.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    lib.host_log.restype = ctypes.c_char_p
    lib.host_allocation_limit.argtypes = [ctypes.c_size_t]
    return lib


def _load(host, rows, n_tasks):
    host.host_log_clear()
    out = ctypes.c_void_p(None)
    host.infaas_catalog_load.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int, ctypes.c_void_p]
    assert host.infaas_catalog_load(rows.ctypes.data, rows.shape[0], n_tasks, 0, ctypes.byref(out)) == 0
    return out


def _log(host):
    return host.host_log().decode().split()


def test_load_waits_for_the_layout_before_the_first_rebuild(host):
    """Kernels are launched as programmatic dependents and read the layout before they wait for their
    predecessor, so the layout has to be complete when the first of them is launched."""
    w = W.make("C2", n_queries=16)
    c = _load(host, w.rows, w.n_tasks)
    log = _log(host)
    assert log.count("layout") == 1 and log.count("rebuild") == 1
    assert "wait" in log[log.index("layout"):log.index("rebuild")], log
    host.infaas_catalog_free(c)


def test_overlapping_kernels_do_not_read_through_the_read_only_path():
    """A kernel launched as a programmatic dependent runs while its predecessor still writes: loads that
    promise constant data (__ldg, const __restrict__) or that the compiler may move over the wait are
    allowed for the layout's arrays alone, which no kernel writes once the catalog is loaded."""
    fixed = ("c.task_off", "c.reg_off")
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        if not name.endswith(".cu") or "chain_wait()" not in text:
            continue
        seen += 1
        assert not re.search(r"const[^;,()]*\*\s*__restrict__", text), name
        bad = [m.group(0) for m in re.finditer(r"__ld[a-z]+\(([^\n]{0,20})", text) if not m.group(1).startswith(fixed)]
        assert not bad, (name, bad)
    assert seen >= 5


def _workers_config(host, c, tables):
    host.infaas_workers_config.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_uint32] + [ctypes.c_void_p] * 2 + [ctypes.c_uint32,
                                                                                                          ctypes.c_void_p]
    iv, iw, il, hw, ut = tables
    host.host_log_clear()
    rc = host.infaas_workers_config(c, iv.ctypes.data, iw.ctypes.data, il.ctypes.data, iv.size, hw.ctypes.data, ut.ctypes.data,
                                    hw.size, None)
    host.host_workers_table.restype = ctypes.c_void_p
    got = [np.ctypeslib.as_array(ctypes.cast(host.host_workers_table(i), ctypes.POINTER(ctypes.c_uint8)), (a.nbytes,))
           for i, a in enumerate(tables)]
    return rc, all(np.array_equal(g, a.view(np.uint8)) for g, a in zip(got, tables))


@pytest.mark.parametrize("n_inst,n_workers", [(1, 1), (1000, 17), (40_001, 5_003)])
def test_host_tables_without_host_memory(host, n_inst, n_workers):
    """The header promises that no function throws and asks for no host memory: a table call goes on
    without the buffer it would pass its tables through, and no table is copied on the host that is
    larger than the catalog's own."""
    w = W.make("C1", n_queries=16)
    rng = np.random.default_rng(n_inst)
    tables = [rng.integers(0, 2**31, n, np.uint32) for n in (n_inst, n_inst, n_inst)] + \
        [rng.integers(0, 256, n_workers, np.uint8), rng.integers(0, 2**31, n_workers, np.uint32)]
    # a catalog's own buffers: 32 bytes per variant, 4 per task and 32 KB
    own = 32 * w.n_variants + 4 * w.n_tasks + 32768
    for limit, grown in ((64, False), (own, False), (2**62, False), (64, True)):
        c = _load(host, w.rows, w.n_tasks)
        if grown:                                     # buffers as an earlier, larger call leaves them
            big = [np.repeat(a, 3) for a in tables]
            assert _workers_config(host, c, big) == (0, True)
        host.host_allocation_limit(limit)
        try:
            rc, same = _workers_config(host, c, tables)
            log = _log(host)
            state = np.ones(w.n_variants, np.uint8)
            queued, served = np.empty(w.n_variants, np.uint32), np.empty(w.n_variants, np.uint64)
            host.infaas_catalog_set_states.argtypes = host.infaas_autoscale_config.argtypes = [ctypes.c_void_p] * 4
            host.infaas_catalog_get_state.argtypes = [ctypes.c_void_p] * 6
            rcs = [host.infaas_catalog_set_states(c, state.ctypes.data, queued.ctypes.data, None),
                   host.infaas_autoscale_config(c, queued.ctypes.data, np.zeros(w.n_tasks, np.uint32).ctypes.data, None),
                   host.infaas_catalog_get_state(c, queued.ctypes.data, None, served.ctypes.data, None, None)]
        finally:
            host.host_allocation_limit(2**64 - 1)
        assert rc == 0 and same and rcs == [0, 0, 0]
        assert log.count("malloc") == (12 * n_inst + 5 * n_workers > own and not grown)
        host.infaas_catalog_free(c)


def test_no_exception_leaves_the_c_entries(host):
    """Host memory that runs out inside a call is an error code, not a C++ exception."""
    w = W.make("C2", n_queries=16)
    c = _load(host, w.rows, w.n_tasks)
    out, info = ctypes.c_void_p(None), np.zeros(8, np.uint32)
    host.infaas_catalog_get_info.argtypes = [ctypes.c_void_p] * 3
    rcs = []
    for limit in (0, 64, 200, 4 * w.n_tasks, 4 * w.n_variants - 1):
        host.host_allocation_limit(limit)
        rcs.append(host.infaas_catalog_load(w.rows.ctypes.data, w.rows.shape[0], w.n_tasks, 0, ctypes.byref(out)))
        assert out.value is None
        if limit < 4 * w.n_tasks:
            rcs.append(host.infaas_catalog_get_info(c, info.ctypes.data, None))
    host.host_device_error(1)
    host.host_allocation_limit(0)                        # (no room for the error's text either)
    failed = host.infaas_catalog_get_info(c, info.ctypes.data, None)
    host.host_device_error(0)
    host.host_allocation_limit(2**64 - 1)
    assert set(rcs) == {-6} and failed == -7
    assert host.infaas_catalog_get_info(c, info.ctypes.data, None) == 0
    host.infaas_catalog_free(c)


@pytest.mark.parametrize("n_tasks,per_task,clusters", [(1, 1024, False), (1, 1025, True), (33, 1025, True), (34, 1025, False),
                                                       (37, 1025, False), (5, 8192, True), (7, 8192, False)])
def test_clusters_only_where_all_run_at_once(host, n_tasks, per_task, clusters):
    """Four CTAs per large task only while a second wave is not needed (the stand-in's device runs 33
    clusters at once), and while every block is in reach of the task word (7 x 8192 variants are not)."""
    rows = np.zeros(n_tasks * per_task, W.VARIANT_DTYPE)
    rows["task"] = np.arange(rows.size) % n_tasks
    rows["batch"] = rows["lat_us"] = rows["cost"] = 1
    c = _load(host, rows, n_tasks)
    assert [x for x in _log(host) if x.startswith("rebuild")] == ["rebuild_by_clusters" if clusters else "rebuild"]
    host.infaas_catalog_free(c)


@pytest.mark.parametrize("K", [1, 4])
def test_every_word_of_a_tasks_bit_sets_has_one_writer(host, K):
    """The CTAs of a task share its variants out, and the words of the bit sets over them: a CTA behind the
    last variant has no word either (it would overwrite another's)."""
    out = (ctypes.c_uint32 * 8)()
    empty = 0
    for V in range(8193):
        writers, at = [0] * ((V + 31) // 32), 0
        for share in range(K):
            host.host_task_share(V, K, share, out)
            cs, ng, rows, y0, lo, hi, w0, w1 = out
            assert ng <= 64 and y0 == share * rows and at == lo <= hi <= V, (V, share)
            assert lo == hi or (lo % 32 == 0 and lo == y0 << cs and w0 == lo // 32 and w1 == (hi + 31) // 32), (V, share)
            at = hi
            empty += lo == hi and V > 0
            for w in range(w0, w1):
                writers[w] += 1
        assert at == V and writers == [1] * len(writers), (V, writers)
    assert empty > 100 or K == 1


def test_small_split_only_where_the_rebuild_fits_into_it(host):
    """Kernels ask for 32 KB of shared memory per SM only around a rebuild whose CTA fits into that; -1 = the
    driver's choice."""
    src = open(os.path.join(CSRC, "rebuild.cu")).read()
    assert "c.max_task_variants <= REBUILD_THREAD_MAX" in src
    assert [host.host_split(n) for n in (0, 1, 256, 257, 512, 513, 1024, 8192)] == [14] * 5 + [-1] * 3
