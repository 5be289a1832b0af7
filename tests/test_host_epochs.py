"""The barrier epochs of the small-lattice kernels over a long-lived engine's
launches (csrc/epochs.h), compiled for the host (no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_word_left_in_an_inbox_passes_a_later_barrier(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "epochs"
    subprocess.run([cxx, "-std=c++17", "-O2", os.path.join(HERE, "host", "epochs.cc"), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout
    launches, clearings = (int(v) for v in out.stdout.split())
    assert launches > 1 << 21 and clearings > 0  # (2^21 launches: twice 2^32 epochs)
