"""Edges grouped by a larger endpoint whose list is too long for a filter to pay (filter_pays): their lists are
tested by hashing, or looked up at once, in the same units.  Both sides of every line, at the edges of rows
(128 entries), pieces (1,024) and of the short lists of warp units, in every colour layout, against the CPU
oracle."""
import os
import subprocess

import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_counts_equal, gpu_run
from paper_1811_09136_gb300 import _build
from paper_1811_09136_gb300 import graphgen as gg

HERE = os.path.dirname(os.path.abspath(__file__))
LAYOUTS = [(2, 2), (10, 7), (300, 300), (3, 7), (20, 100), (1, 3), (100, 500)]


def test_the_rule(tmp_path):
    exe = str(tmp_path / "filter_rule_check")
    subprocess.check_call([_build._nvcc(), "-O2", "-std=c++17", "-I", _build.CSRC, "-I", _build.INCLUDE, "-o", exe,
                           os.path.join(HERE, "native", "filter_rule_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr


def pairs_stream(pairs, leaves, seed):
    """For every (L, lists): an endpoint with L entries and one node per length in `lists` with that many
    entries, at least half of them shared, in random order among 40,000 other edges; then the edges between."""
    r = np.random.default_rng(seed)
    ids = sum(1 + len(lists) for _, lists in pairs)
    e, last, node = [], [], 0
    for n_l, lists in pairs:
        l, near = node, ids + r.permutation(leaves)[:n_l]
        e.append(np.stack([np.full(n_l, l), near], 1))
        node += 1
        for k in lists:
            own = np.unique(np.concatenate([r.permutation(near)[:(k + 1) // 2], ids + r.permutation(leaves)[:k]]))
            own = r.permutation(own)[:k]
            e.append(np.stack([np.full(len(own), node), own], 1))
            last.append((node, l))
            node += 1
    a, b = ids + r.integers(leaves, size=40_000), ids + r.integers(leaves, size=40_000)
    key = np.unique((np.minimum(a, b) * (1 << 32) + np.maximum(a, b))[a != b])
    e = np.concatenate([*e, np.stack([key >> 32, key & 0xFFFFFFFF], 1)])
    e = np.concatenate([e[r.permutation(len(e))], np.array(last)])
    flip = r.random(len(e)) < 0.5
    return gg.EdgeStream(np.where(flip, e[:, 1], e[:, 0]).astype(np.uint32),
                         np.where(flip, e[:, 0], e[:, 1]).astype(np.uint32), ids + leaves)


def check(s, m, c):
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 7, pair_counters=c > m and c % m != 0)
    for batch in (len(s), 1 << 15):
        proc, local, _, _, _ = gpu_run(s, m, c, 7, batch=batch, expected_edges=len(s))
        assert_counts_equal(proc, local, ref.tau_proc, ref.local1 + ref.local2, f"batch={batch}")


LISTS = [33, 64, 127, 128, 129, 130, 255, 257, 1023, 1024, 1025, 2049, 5000]


@pytest.mark.gpu
@pytest.mark.parametrize("m,c", LAYOUTS)
def test_long_lists_of_the_larger_endpoint(m, c):
    # (the edge between the two counts as well)
    check(pairs_stream([(24_576 - len(LISTS), LISTS), (24_577 - len(LISTS), LISTS), (30_000, LISTS)], 31_000, m), m, c)


@pytest.mark.gpu
@pytest.mark.parametrize("m,c", [(3, 7), (20, 100), (1, 3), (100, 500)])
def test_longer_ones_without_single_colours(m, c):
    lists = [40, 129, 1025, 16_500]  # (the edges between the two count as well)
    check(pairs_stream([(262_140, lists), (262_141, lists)], 263_000, m), m, c)


@pytest.mark.gpu
@pytest.mark.parametrize("m,c", LAYOUTS)
def test_few_scanned_entries_beside_the_larger_list(m, c):
    # on both sides of four (sixteen) times the scanned entries; larger endpoints of warp units (up to 1,024
    # entries), which always have their filter, and of block units
    pairs = [(times * (k + 1) + more, [k]) for k in (32, 33, 40, 127, 128, 129, 130, 255, 400) for times in (4, 16)
             for more in (-2, -1, 0, 60)]
    check(pairs_stream(pairs, 12_000, m + 1), m, c)
