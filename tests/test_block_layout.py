"""The parts of a node's block stay inside it at every table size (host build)."""
import os
import subprocess

from paper_1811_09136_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_parts_of_a_block_do_not_overlap(tmp_path):
    exe = str(tmp_path / "block_layout_check")
    subprocess.check_call([_build._nvcc(), "-O2", "-std=c++17", "-I", _build.CSRC, "-I", _build.INCLUDE, "-o", exe,
                           os.path.join(HERE, "native", "block_layout_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
