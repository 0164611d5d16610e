"""No-GPU checks of the C-ABI library: it builds, loads, exports every symbol the header
declares, and rejects bad catalogs on the host before any CUDA call."""
import ctypes
import os
import re

import numpy as np
import pytest

from paper_1905_13348_b200 import build as B
from paper_1905_13348_b200 import workloads as W
from tests.helpers import rows_from

ROOT = os.path.join(os.path.dirname(__file__), "..")


@pytest.fixture(scope="module")
def lib():
    return ctypes.CDLL(B.build())


def declared_functions():
    text = open(os.path.join(ROOT, "include", "infaas.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(infaas_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert {"infaas_catalog_load", "infaas_select_batch", "infaas_load_update"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def test_row_struct_is_24_bytes_and_matches_generator_dtype():
    assert W.VARIANT_DTYPE.itemsize == 24
    offs = {k: W.VARIANT_DTYPE.fields[k][1] for k in W.VARIANT_DTYPE.names}
    assert offs == {"task": 0, "arch": 2, "hw": 4, "opt": 5, "batch": 6, "lat_us": 8,
                    "acc_bp": 12, "reserved": 14, "cost": 16, "queued": 20}


def _load(lib, rows, n_tasks):
    out = ctypes.c_void_p(None)
    lib.infaas_catalog_load.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint32,
                                        ctypes.c_int, ctypes.POINTER(ctypes.c_void_p)]
    rc = lib.infaas_catalog_load(rows.ctypes.data if rows is not None else None,
                                 0 if rows is None else rows.shape[0], n_tasks, 0, ctypes.byref(out))
    assert rc != 0 and out.value is None
    return rc


def test_host_side_validation_codes(lib):
    good = rows_from([0, 1], [1, 1], [10, 10], [7000, 7000], [1, 1])
    assert _load(lib, None, 1) == -1
    assert _load(lib, good, 0) == -2 and _load(lib, good, 70000) == -2
    assert _load(lib, good, 1) == -2                        # row task 1 >= n_tasks 1
    for field, value, code in (("batch", 0, -3), ("lat_us", 0, -4), ("acc_bp", 10001, -5),
                               ("reserved", 1, -5)):
        bad = good.copy(); bad[field][1] = value
        assert _load(lib, bad, 2) == code, field
    big = rows_from([0] * 8193, [1] * 8193, [10] * 8193, [7000] * 8193, [1] * 8193)
    assert _load(lib, big, 1) == -6                         # above the per-task limit
    lib.infaas_strerror.restype = ctypes.c_char_p
    for code in range(-10, 1):
        assert lib.infaas_strerror(code)
    lib.infaas_catalog_free(None)                           # NULL is allowed


def test_binding_fails_loudly_without_device():
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present")
    import paper_1905_13348_b200 as P
    with pytest.raises(P.InfaasError):
        P.infaas_catalog_load(W.make("C1").rows, 1)


def test_binding_constants_match_the_header():
    text = open(os.path.join(ROOT, "include", "infaas.h")).read()
    defs = {m.group(1): int(m.group(2).rstrip("u"), 0)
            for m in re.finditer(r"#define\s+(INFAAS_[A-Z_]+)\s+\(?(-?(?:0x[0-9A-Fa-f]+|\d+)u?)\)?", text)}
    from paper_1905_13348_b200 import binding as b
    assert defs["INFAAS_NO_FEASIBLE"] == b.NO_FEASIBLE and defs["INFAAS_INVALID"] == b.INVALID
    assert [defs[f"INFAAS_STATE_{n}"] for n in ("INACTIVE", "ACTIVE", "OVERLOADED", "INTERFERED")] == \
        [b.STATE_INACTIVE, b.STATE_ACTIVE, b.STATE_OVERLOADED, b.STATE_INTERFERED]
    assert defs["INFAAS_AUTOSCALE_NONE"] == b.AUTOSCALE_NONE and defs["INFAAS_AUTOSCALE_ESCALATE"] == b.AUTOSCALE_ESCALATE
    assert sorted(b.EXPORTS) == sorted(n for n in declared_functions())
    codes = sorted(v for k, v in defs.items() if k.startswith("INFAAS_E_"))
    assert codes == list(range(-11, 0))


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_torchs_private_getters(monkeypatch, missing):
    import types

    import torch

    from paper_1905_13348_b200 import binding as b
    monkeypatch.delattr(torch._C, missing)
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: types.SimpleNamespace(cuda_stream=4000 + device))
    monkeypatch.setattr(b, "_raw_stream", None)
    monkeypatch.setattr(b, "_current_device", None)
    assert b._stream_ptr(None) == 4003
    assert b._stream_ptr(types.SimpleNamespace(cuda_stream=5)) == 5


def test_per_window_calls_convert_arguments_as_before():
    """The extension module's calls: errors and conversions of the Python they stand for."""
    import types

    import torch

    import paper_1905_13348_b200 as P
    s = types.SimpleNamespace(cuda_stream=0)
    cat = types.SimpleNamespace(handle=ctypes.c_void_p(None), n_tasks=1, n_variants=1)
    t32 = torch.zeros(4, dtype=torch.int32)

    class Like:                              # not a tensor, but it answers what is asked of one
        is_cuda, dtype, device, shape = True, torch.int32, "cuda", (4,)
        numel = staticmethod(lambda: 4)
        is_contiguous = staticmethod(lambda: True)
        data_ptr = staticmethod(lambda: 4096)

    calls = [lambda d, **k: P.infaas_tally(cat, d, stream=s, **k),
             lambda d, **k: P.infaas_load_update(cat, d, 1000, stream=s, **k),
             lambda d, **k: P.infaas_assign_workers(cat, d, d, stream=s, **k),
             lambda d, **k: P.infaas_select_batch(cat, None, d, None, d, stream=s, **{"n": 4, **k}),
             lambda d, **k: P.infaas_select_update(cat, None, d, None, d, 1000, stream=s, **{"n": 4, **k})]
    for call in calls:
        with pytest.raises(TypeError, match="expected a contiguous CUDA tensor of u32, got torch.int32 on cpu"):
            call(t32)
        for d, n in ((Like(), 3), (Like(), 3.7), (Like(), True), (None, 0)):
            with pytest.raises(P.InfaasError, match="NULL"):             # the catalog's handle
                call(d, n=n)
        with pytest.raises((TypeError, ValueError)):
            call(Like(), n="many")
    with pytest.raises(TypeError, match="u16, got torch.int32"):
        P.infaas_select_batch(cat, t32, None, None, None, stream=s)
    with pytest.raises(AttributeError):
        P.infaas_select_batch(cat, None, None, None, None, stream=s)     # no length to be had
    with pytest.raises(IndexError):
        P.infaas_tally(cat, torch.zeros((), dtype=torch.int32), stream=s)
    with pytest.raises(P.InfaasError, match="NULL"):
        P.infaas_advance(cat, 1000, stream=s)
    with pytest.raises(P.InfaasError, match="NULL"):
        P.infaas_autoscale_step(cat, 1000, 105, 100, Like(), Like(), stream=s)
    with pytest.raises((TypeError, ValueError)):
        P.infaas_advance(cat, None, stream=s)
    with pytest.raises(AttributeError):
        P.infaas_advance(object(), 1000, stream=s)


def test_extension_module_of_another_torch_is_not_used(monkeypatch):
    """The module reads tensors by the layout of the torch it was built against: after an upgrade it has to be
    built again, not loaded."""
    import torch

    import paper_1905_13348_b200 as P
    from paper_1905_13348_b200 import binding as b, build
    build.build()
    monkeypatch.setattr(b, "_calls", None)
    assert not build._stale() and b._load_calls() is not None
    monkeypatch.setattr(torch, "__version__", "99.0.0+other")
    monkeypatch.setattr(b, "_calls", None)
    assert build._stale()
    with pytest.raises(RuntimeError, match="not built for this torch"):
        P.infaas_advance(object(), 1000)
    assert b._calls is None
