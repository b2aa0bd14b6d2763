"""The binding without a GPU: what is built again after which change, what a tree that is not built says, and that a decode step's
calls do the same through the extension as through ctypes."""
import ctypes as C
import importlib.machinery
import importlib.util
import os
import shutil
import types

import numpy as np
import pytest
import torch

from paper_2608_23599_b200 import binding as B
from paper_2608_23599_b200 import build as _build


@pytest.mark.parametrize("changed,stale", [
    (None, False), ("gkv_call.cpp", True), ("gkv.h", True), ("gkv_decode.cu", True), ("gkv_exchange.h", True)])
@pytest.mark.parametrize("fresh", [_build.LIB, _build.CALL_LIB])
def test_either_library_is_built_again_after_a_change_of_its_sources(monkeypatch, changed, stale, fresh):
    """One of the two libraries is newer than the change, as an interrupted build leaves it."""
    monkeypatch.setattr(_build.os.path, "exists", lambda p: True)
    when = {_build.LIB: 2.0, _build.CALL_LIB: 2.0, changed: 3.0, fresh: 4.0}
    monkeypatch.setattr(_build.os.path, "getmtime", lambda p: when.get(p, when.get(os.path.basename(p), 1.0)))
    concerns_both = changed == "gkv.h"
    only_fresh_concerned = {"gkv_call.cpp": _build.CALL_LIB}.get(changed, _build.LIB) == fresh and not concerns_both
    assert _build.needs_build() == (stale and not only_fresh_concerned)


def test_a_tree_without_the_extension_says_what_to_do(monkeypatch, tmp_path):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(_build, "CALL_LIB", str(tmp_path / "_gkv_call.so"))
    with pytest.raises(FileNotFoundError, match="_gkv_call.so is missing: run `python -m paper_2608_23599_b200.build`"):
        B.load()


class Address:
    def __init__(self, value):
        self.value = value

    def data_ptr(self):
        if isinstance(self.value, Exception):
            raise self.value
        return self.value


TENSOR = torch.arange(8, dtype=torch.float32)
CALLS = {
    "gkv_append_demote": lambda c, layer, n, p: c.gkv_append_demote(layer, p, p, token_mass=p, level_plan=np.ones(3, dtype=np.int64), n_new=n),
    "gkv_decode_attn": lambda c, layer, n, p: c.gkv_decode_attn(layer, p, p, lse=p, page_idx=p, n_sel=n),
    "gkv_decode_attn_observe": lambda c, layer, n, p: c.gkv_decode_attn_observe(layer, p, p, p, p, p),
    "gkv_quest_select": lambda c, layer, n, p: c.gkv_quest_select(layer, p, n, p),
}


@pytest.fixture
def extension(tmp_path):
    """A second copy of the extension, to be bound to fakes."""
    B.load()
    path = shutil.copy(_build.CALL_LIB, tmp_path)
    spec = importlib.util.spec_from_file_location("_gkv_call", path, loader=importlib.machinery.ExtensionFileLoader("_gkv_call", path))
    return importlib.util.module_from_spec(spec)


@pytest.mark.parametrize("name", CALLS)
def test_the_extension_and_ctypes_do_the_same(extension, monkeypatch, name):
    """The library's four entry points replaced by fakes that note what reaches them: arguments of every type that either road
    takes or refuses, and every kind of status, give the same call and the same result or exception on both."""
    real, seen, status = B.load(), [], [0]

    def fake(entry):
        def note(*args):
            args = list(args)
            if entry == "gkv_quest_select":
                args[5][0] = 7                       # pages selected
                args[5] = None
            seen.append((entry, args))
            return status[0]
        return C.CFUNCTYPE(C.c_int, *getattr(real, entry).argtypes)(note)

    fakes = {entry: fake(entry) for entry in CALLS}
    extension.bind(*(C.cast(fakes[entry], C.c_void_p).value for entry in CALLS), C.c_void_p)
    through_ctypes = types.SimpleNamespace(**{f: lambda *a: NotImplemented for f in ("append", "decode", "observe", "select")})
    monkeypatch.setattr(B, "_lib", types.SimpleNamespace(gkv_strerror=real.gkv_strerror, **fakes))

    class Bare(B.Cache):
        def __init__(self):
            pass

        def close(self):                             # (the handle is no cache)
            pass

    cache = Bare()

    def outcome(road, handle, stream, layer, n, p):
        monkeypatch.setattr(B, "_call", road)
        cache.handle, cache.stream_handle = handle, stream
        seen.clear()
        try:
            got = CALLS[name](cache, layer, n, p)
        except Exception as e:      # noqa: BLE001
            got = type(e), str(e)
        if name == "gkv_append_demote":              # the plan is copied for the call
            seen[:] = [(e, a[:6] + [bool(a[6])] + a[7:]) for e, a in seen]
        return got, list(seen)

    plain = dict(handle=C.c_void_p(0x1230), stream=0x77, layer=3, n=64, p=TENSOR)
    unusual = [
        dict(handle=v) for v in (None, 0x1230, True, C.c_void_p(), C.c_int(5), Address(5), 1.5)
    ] + [
        dict(stream=v) for v in (0, -1, 2 ** 64 + 5, C.c_void_p(0x88), Address(5), np.int64(5), 1.5)
    ] + [
        {key: v} for key in ("layer", "n") for v in (np.int32(2), np.int64(2), True, -1, 2 ** 32 + 3, 2 ** 70, 1.0, None, "2", TENSOR)
    ] + [
        dict(p=v) for v in (None, 0x5000, -1, 2 ** 64 + 9, Address(0x5000), Address(None), Address(np.int64(5)), Address(1.5),
                            Address(RuntimeError("no storage")), np.int64(5), np.zeros(3), "x", 1.5, C.c_void_p(5))
    ]
    made = 0
    for change in [{}] + unusual:
        args = {**plain, **change}
        want = outcome(through_ctypes, **args)
        got = outcome(extension, **args)
        assert got == want, (name, change)
        made += len(got[1])
    assert made > 20                                 # (most of them are calls)
    for code in (B.OK, B.ERR_RANGE, B.ERR_BUDGET, B.ERR_INVALID_ARG, B.ERR_CUDA, -77):
        status[0] = code
        assert outcome(extension, **plain) == outcome(through_ctypes, **plain), (name, code)


def test_the_extension_lets_an_interrupt_through(extension):
    extension.bind(0, 0, 0, 0, C.c_void_p)

    class Interrupted:
        def data_ptr(self):
            raise KeyboardInterrupt

    with pytest.raises(KeyboardInterrupt):
        extension.decode(None, 0, Interrupted(), None, 0, None, None, None)
    with pytest.raises(TypeError):
        extension.decode(None, 0)
