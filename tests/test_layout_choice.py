"""Which streams store colour words beside their entries, and streams that have to do without them after all:
a pool that 32-bit offsets do not span with the words, or that the memory does not hold."""
import os
import subprocess
import sys

import pytest

from paper_1811_09136_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_choice_of_layout(tmp_path):
    exe = str(tmp_path / "layout_choice_check")
    subprocess.check_call([_build._nvcc(), "-O2", "-std=c++17", "-I", _build.CSRC, "-I", _build.INCLUDE, "-o", exe,
                           os.path.join(HERE, "native", "layout_choice_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.gpu
def test_streams_that_give_up_their_words():
    path = _build.build(debug_bounds=True)
    out = subprocess.run([sys.executable, os.path.join(HERE, "layout_change_run.py")],
                         env=dict(os.environ, REPT_LIBRARY=path), capture_output=True, text=True, timeout=900)
    assert out.returncode == 0 and "layout change ok" in out.stdout, out.stdout[-3000:] + out.stderr[-3000:]
    assert "index check" not in out.stderr, out.stderr[-3000:]
