"""$CC may carry options or a launcher, and may be empty, as build tools have it."""
import os
import sysconfig

import pytest

from paper_cs_9809105_gb300 import build as B


@pytest.mark.parametrize("cc", ["gcc -pthread", "env gcc", ""])
def test_cc_with_words(tmp_path, monkeypatch, cc):
    headers = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(headers, "Python.h")):
        pytest.skip("no Python headers: the binding uses ctypes")
    monkeypatch.setenv("CC", cc)
    B.compile_call(headers, str(tmp_path / "m.so"))
    assert (tmp_path / "m.so").stat().st_size > 0
