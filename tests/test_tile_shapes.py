"""The launch shapes that the kernels' constants allow (CPU only: kernels.cuh
compiles as host code without its device part): a CTA's threads must copy a
whole tile and fit their kernel's launch bound."""
import os
import subprocess

import pytest

from paper_2607_26566_gb300 import build as b


@pytest.mark.parametrize("threads,ok", [(None, True), (256, True), (320, True), (384, True), (512, True), (1024, True),
                                        (128, False), (224, False), (400, False), (416, False), (448, False),
                                        (1056, False), (500, False)])
def test_threads_of_a_tile(tmp_path, threads, ok):
    src = tmp_path / "k.cpp"
    src.write_text('#include "kernels.cuh"\n')
    r = subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-fsyntax-only", "-I" + b.CSRC, str(src)]
                       + ([f"-DT2I_TUNE_TILE_THREADS={threads}"] if threads else []), capture_output=True, text=True)
    assert (r.returncode == 0) == ok, r.stderr
    assert ok or "does not cover a tile" in r.stderr
