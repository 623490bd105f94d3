"""The build step compiles again what has changed: sources, headers and the
included tables (a stand-in for nvcc writes the files it is asked for)."""
import os

import pytest

from paper_2607_23354_gb300 import build as B

NVCC = """#!/bin/sh
echo "$@" >> "$LOG"
while [ $# -gt 0 ]; do
  if [ "$1" = "-o" ]; then shift; touch "$1"; fi
  shift
done
"""


@pytest.mark.parametrize("changed,objects", [(None, 0), ("csrc/a.cu", 1), ("csrc/h.cuh", 2), ("csrc/table.inc", 2),
                                             ("include/api.h", 2)])
def test_changed_files_are_compiled_again(tmp_path, monkeypatch, changed, objects):
    for d in ("csrc", "include", "_build"):
        (tmp_path / d).mkdir()
    for f in ("csrc/a.cu", "csrc/b.cu", "csrc/h.cuh", "csrc/table.inc", "include/api.h"):
        (tmp_path / f).write_text("")
        os.utime(tmp_path / f, (1e9, 1e9))
    nvcc, log = tmp_path / "nvcc", tmp_path / "log"
    nvcc.write_text(NVCC)
    nvcc.chmod(0o755)
    monkeypatch.setenv("LOG", str(log))
    monkeypatch.setattr(B, "_nvcc", lambda: str(nvcc))
    for name, value in (("CSRC", "csrc"), ("INCLUDE", "include"), ("BUILD", "_build"), ("LIB", "_build/lib.so")):
        monkeypatch.setattr(B, name, str(tmp_path / value))
    B.build()
    assert log.read_text().count(" -c ") == 2
    for f in (tmp_path / "_build").iterdir():
        os.utime(f, (1.1e9, 1.1e9))
    log.write_text("")
    if changed:
        os.utime(tmp_path / changed, (1.2e9, 1.2e9))
    B.build()
    assert log.read_text().count(" -c ") == objects
    assert log.read_text().count("-shared") == (1 if objects else 0)
