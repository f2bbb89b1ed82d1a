"""The binding loads the call module built for this interpreter and no other file like it."""
import os
import shutil

import pytest

from paper_cs_9809105_gb300 import build as B
from paper_cs_9809105_gb300 import hsmm as H


@pytest.fixture
def empty(tmp_path, monkeypatch):
    """A build folder without a call module for this interpreter."""
    B.build()
    H.lib()
    monkeypatch.setattr(H, "LIB_PATH", str(tmp_path / "libhsmm.so"))
    monkeypatch.setattr(H, "CALL_PATH", str(tmp_path / os.path.basename(B.CALL)), raising=False)
    monkeypatch.setattr(H, "_call", None)
    return tmp_path


def test_the_path_is_the_one_built():
    assert H.CALL_PATH == B.CALL


@pytest.mark.parametrize("name", ["_hsmmcall.cpython-399-other.so", "_hsmmcall.so.so"])
def test_other_modules_are_not_loaded(empty, name):
    if not os.path.exists(B.CALL):
        pytest.skip("no Python headers: the binding uses ctypes")
    shutil.copy(B.CALL, empty / name)
    H._bind_calls(H.lib())
    assert H._call is None
    shutil.copy(B.CALL, empty / os.path.basename(B.CALL))
    H._bind_calls(H.lib())
    assert H._call is not None and H._call.__file__ == str(empty / os.path.basename(B.CALL))


def test_a_file_that_is_no_module_is_passed_over(empty):
    (empty / os.path.basename(B.CALL)).write_bytes(b"not a module")
    H._bind_calls(H.lib())
    assert H._call is None
