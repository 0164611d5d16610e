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
