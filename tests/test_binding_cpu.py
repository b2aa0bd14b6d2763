"""The binding without a GPU: what is built again after which change, and what a tree that is not built says."""
import os

import pytest

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
