"""What admission and the batched path reckon a stream's state to take is what the library allocates."""
import os
import subprocess

import numpy as np
import pytest

from paper_1811_09136_gb300 import _build, batched

HERE = os.path.dirname(os.path.abspath(__file__))

CONFIGS = [(m, c, n, edges) for m in (1, 2, 3, 10, 20, 100, 128, 129, 256, 257, 300, 65_536, 65_537)
           for c in (1, 2, 7, 10, 32, 33, 100, 140, 500, 4096) for n in (1000, 1 << 24, (1 << 24) + 1)
           for edges in (1000, 357_913_935, 357_913_936, 600_000_000)]


def test_pool_bytes_per_edge(tmp_path):
    exe = str(tmp_path / "edge_bytes_table")
    subprocess.check_call([_build._nvcc(), "-O2", "-std=c++17", "-I", _build.CSRC, "-I", _build.INCLUDE, "-o", exe,
                           os.path.join(HERE, "native", "edge_bytes_table.cu")])
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % x for x in CONFIGS), capture_output=True, text=True,
                         timeout=300, check=True)
    want = [int(x) for x in out.stdout.split()]
    assert len(want) == len(CONFIGS) and set(want) == {256, 384}
    got = [batched._edge_bytes(n, edges, m, c) for m, c, n, edges in CONFIGS]
    assert [x for x, a, b in zip(CONFIGS, got, want) if a != b] == []


def test_waves_reckon_with_colour_words():
    from paper_1811_09136_gb300.graphgen import EdgeStream
    streams = [EdgeStream(np.zeros(50_000, np.uint32), np.zeros(50_000, np.uint32), 1000) for _ in range(6)]
    plain = batched._state_bytes(1000, 50_000, 64, 20, 20) + 8 * 50_000
    assert plain == batched._state_bytes(1000, 50_000, 64) + 8 * 50_000
    words = batched._state_bytes(1000, 50_000, 64, 20, 100) + 8 * 50_000
    assert words - plain == 128 * 50_000
    assert [len(w) for w in batched._waves(streams, 64, 3 * plain, [(20, 20, 1)] * 6)] == [3, 3]
    assert [len(w) for w in batched._waves(streams, 64, 3 * plain, [(20, 100, 1)] * 6)] == [2, 2, 2]


@pytest.mark.gpu
@pytest.mark.parametrize("m,c", [(10, 10), (300, 300), (20, 100), (3, 3), (100, 500)])
def test_reckoned_bytes_cover_a_handle(m, c):
    from paper_1811_09136_gb300.rept import ReptStream
    with ReptStream(30_000, m, c, 1, expected_edges=400_000, max_batch=1 << 14) as h:
        held = h.stats()["device_bytes"]
    reckoned = batched._state_bytes(30_000, 400_000, 1 << 14, m, c)
    assert held <= reckoned <= held + (3 << 20)
