"""The per-micro-batch calls of the binding, through the CPython module and through ctypes, take the same objects and hand
on the same addresses.  A recording stub takes the library's place; no call touches a GPU."""
import ctypes as C
import os
import subprocess
import sysconfig
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2604_19654_b200 import build as B
from paper_2604_19654_b200 import feplb as F

# parameters of every call that the module resolves; the last but one of moe_backward is an int
ARITY = {"feplb_moe_forward": 18, "feplb_moe_backward": 21, "feplb_route_topk": 5, "feplb_route_hist": 5,
         "feplb_dispatch": 8, "feplb_combine": 6}
BUF = ["counts", "rank_load", "x_perm", "h_scratch", "y_perm", "slot_to_row", "row_to_token", "out"]
BWD = ["ab", "d_y_perm", "d_ab", "d_x_perm", "d_x", "d_gates"]


@pytest.fixture(scope="module")
def stub_path(tmp_path_factory):
    B.build()
    src = tmp_path_factory.mktemp("stub") / "stub.cpp"
    text = "extern \"C\" { unsigned long long seen[32];\n"
    for name, n in ARITY.items():
        types = ["int" if name == "feplb_moe_backward" and i == 19 else "void*" for i in range(n)]
        text += f"int {name}({', '.join(f'{t} a{i}' for i, t in enumerate(types))}) {{"
        text += "".join(f" seen[{i}] = (unsigned long long)a{i};" for i in range(n)) + " return 0; }\n"
    src.write_text(text + "}\n")
    lib = str(src.with_suffix(".so"))
    subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, str(src)], check=True)
    return lib


@pytest.fixture(params=["module", "ctypes"])
def calls(stub_path, request):
    """(module, function that returns what the stub was given last)"""
    stub = C.CDLL(stub_path)
    for name in ARITY:
        getattr(stub, name).argtypes = getattr(F.lib(), name).argtypes
    seen = (C.c_ulonglong * 32).in_dll(stub, "seen")
    read = lambda name: [v or None for v in seen[:ARITY[name]]]       # noqa: E731
    if request.param == "module":
        mod = F._fast()
        assert not isinstance(mod, F._CtypesCalls)
        mod.load(stub_path)
        yield mod, read
        mod.load(F.LIB_PATH)
    else:
        with pytest.MonkeyPatch.context() as m:
            m.setattr(F, "lib", lambda: stub)
            yield F._CtypesCalls(), read


def _objects(n, kind):
    if kind == "tensor":
        return [torch.zeros(4 + i) for i in range(n)]
    if kind == "array":
        return [np.zeros(4 + i, np.float32) for i in range(n)]
    return [1 << 40 | 16 * i for i in range(1, n + 1)]


@pytest.mark.parametrize("kind", ["tensor", "array", "address"])
def test_same_addresses_as_the_ctypes_route(calls, kind):
    mod, seen = calls
    o = _objects(20, kind)
    p = [F._ptr(x) for x in o]
    buf = SimpleNamespace(**dict(zip(BUF, o[6:14])))
    mod.moe_forward(7, *o[:6], None, buf, None, 9)
    assert seen("feplb_moe_forward") == [7, *p[:6], None, *p[6:14], None, 9]
    bwd = SimpleNamespace(**dict(zip(BWD, o[14:20])))
    mod.moe_backward(7, *o[:5], buf, bwd, o[5], None, o[0], 1, None)
    assert seen("feplb_moe_backward") == [7, *p[:5], p[8], p[14], p[9], p[10], p[11], *p[15:20], p[5], None, p[0], 1, None]
    for name, n in (("route_topk", 3), ("route_hist", 3), ("dispatch", 6), ("combine", 4)):
        getattr(mod, name)(7, *o[:n], 9)
        assert seen("feplb_" + name) == [7, *p[:n], 9]


def test_backward_reads_only_the_buffers_it_needs(calls):
    """The forward's buffers that the backward pass has no use for may be gone, or be anything."""
    mod, seen = calls
    o = _objects(10, "tensor")
    buf = SimpleNamespace(**{k: o[i] for i, k in enumerate(("x_perm", "h_scratch", "y_perm", "slot_to_row"))},
                          out=torch.zeros(4, 4).t()[:2])
    mod.moe_backward(7, *o[:5], buf, SimpleNamespace(**dict(zip(BWD, o[4:10]))), None, None, None, 0, None)
    assert seen("feplb_moe_backward")[9] == o[2].data_ptr()


def test_refused_objects(calls):
    mod, _ = calls
    a = torch.zeros(8)
    with pytest.raises(AssertionError):
        mod.combine(7, torch.zeros(4, 4).t(), a, a, a, None)
    with pytest.raises(AttributeError, match="is_contiguous"):
        mod.combine(7, "text", a, a, a, None)


@pytest.mark.parametrize("stream,handle", [(0, None), (12, 12), (C.c_void_p(12), 12), (C.c_void_p(), None),
                                           (SimpleNamespace(cuda_stream=12), 12), (SimpleNamespace(cuda_stream=0), None)])
def test_stream_handles(stream, handle):
    assert F.Context._stream(stream) == handle


def test_interpreter_without_the_module(monkeypatch, tmp_path):
    """The module's file name carries the interpreter's ABI; without that file the calls go through ctypes, and without
    Python headers the library alone makes the build complete."""
    B.build()
    assert F.PY_LIB_PATH == B.PY_LIB and F.PY_LIB_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    monkeypatch.setattr(F, "_fast_mod", None)
    monkeypatch.setattr(F, "PY_LIB_PATH", str(tmp_path / "none.so"))
    assert isinstance(F._fast(), F._CtypesCalls) and F._fast().combine(None, None, None, None, None, None) == F.E_INVALID
    monkeypatch.setattr(B, "PY_LIB", str(tmp_path / "none.so"))
    assert B.needs_build()
    monkeypatch.setattr(B, "_python_include", lambda: None)
    assert not B.needs_build() and os.path.exists(B.LIB)
