"""The block-wide reservation of the batch kernels, also where a block's requests together pass 2^32."""
import os
import subprocess

import pytest

from paper_1811_09136_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def compile_check(tmp_path):
    exe = str(tmp_path / "block_reserve_check")
    subprocess.check_call([_build._nvcc(), *_build.NVCC_FLAGS, "-I", _build.CSRC, "-I", _build.INCLUDE, "-o", exe,
                           os.path.join(HERE, "native", "block_reserve_check.cu")])
    return exe


@pytest.mark.gpu
def test_reservations_follow_one_another(tmp_path):
    out = subprocess.run([compile_check(tmp_path)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr


def test_pool_requests_are_summed_in_64_bits():
    """k_plan's requests are whole block sizes: their sum over a thread block may pass 2^32 quads, and a
    wrapped sum would pass the check of the pool's capacity."""
    with open(os.path.join(_build.CSRC, "rept_kernels.cuh")) as f:
        source = f.read()
    plan = source[source.index("void k_plan_body("):source.index("void k_commit_body(")]
    assert "BlockReserve<unsigned long long> part[2];" in plan
