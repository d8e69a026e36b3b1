"""build() compiles again when any file that goes into the library is newer than
it, headers included. No GPU and no compiler needed."""
import os

import pytest

from paper_2106_02159_gb300 import binding as B

FILES = sorted(os.listdir(B.CSRC)) + ["euler_hyp.h"]


@pytest.mark.parametrize("changed", [None, *FILES])
def test_a_changed_file_is_compiled(changed, tmp_path, monkeypatch):
    csrc, include, out = (tmp_path / d for d in ("csrc", "include", "_build"))
    for d in (csrc, include, out):
        d.mkdir()
    for name in FILES:
        f = (include if name == "euler_hyp.h" else csrc) / name
        f.write_text("")
        age = 100 if name == changed else -100
        os.utime(f, (1e9 + age, 1e9 + age))
    lib = out / "lib.so"
    lib.write_text("old")
    os.utime(lib, (1e9, 1e9))
    calls = []

    def compiler(cmd, check):
        calls.append(cmd)
        (out / "lib.so.tmp").write_text("new")

    monkeypatch.setattr(B, "CSRC", str(csrc))
    monkeypatch.setattr(B, "_ROOT", str(tmp_path))
    monkeypatch.setattr(B, "BUILD_DIR", str(out))
    monkeypatch.setattr(B, "LIB_PATH", str(lib))
    monkeypatch.setattr(B.subprocess, "run", compiler)
    B.build()
    assert len(calls) == (0 if changed is None else 1)
    assert lib.read_text() == ("old" if changed is None else "new")
