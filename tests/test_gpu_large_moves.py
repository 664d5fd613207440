"""Moves of the largest blocks, which many thread blocks share, against the CPU oracle: hubs whose tables
grow past the sizes that one warp, one thread block or several move, in every colour layout, in small
and large batches; and two of them in a batch of one edge."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_counts_equal, gpu_run
from paper_1811_09136_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

LAYOUTS = [(2, 2), (10, 7), (300, 300), (20, 100), (1, 3)]


def hubs_stream(sizes, seed):
    """Hubs 0 .. len(sizes) - 1 with sizes[i] common leaves in random order, then the edges between hubs."""
    r = np.random.default_rng(seed)
    k, n = len(sizes), len(sizes) + max(sizes)
    e = np.concatenate([np.stack([np.full(s, i), k + r.permutation(max(sizes))[:s]], 1) for i, s in enumerate(sizes)])
    e = e[r.permutation(len(e))]
    e = np.concatenate([e, [(i, j) for i in range(k) for j in range(i)]])
    flip = r.random(len(e)) < 0.5
    return gg.EdgeStream(np.where(flip, e[:, 1], e[:, 0]).astype(np.uint32),
                         np.where(flip, e[:, 0], e[:, 1]).astype(np.uint32), n)


@pytest.mark.parametrize("m,c", LAYOUTS)
def test_hubs_grow_past_every_kind_of_move(m, c):
    # tables of twice as many slots, rounded up to a power of two
    s = hubs_stream([30, 250, 4096, 4097, 8200, 16_500, 33_000], seed=m)
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 7, pair_counters=False)
    for batch, sized in ((len(s), 1), (20_000, 0), (3000, 1)):  # from nothing; step by step; in small batches
        proc, local, _, _, _ = gpu_run(s, m, c, 7, batch=batch, expected_edges=sized * len(s))
        assert_counts_equal(proc, local, ref.tau_proc, ref.local1 + ref.local2, f"batch={batch}")


@pytest.mark.parametrize("m,c", [(2, 2), (20, 100)])
def test_two_hubs_in_a_batch_of_one_edge(m, c):
    s = hubs_stream([4096, 4096], seed=3)  # the last edge takes both from 8,192 to 16,384 slots
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 7, pair_counters=False)
    proc, local, _, _, _ = gpu_run(s, m, c, 7, batch=1, expected_edges=len(s))
    assert_counts_equal(proc, local, ref.tau_proc, ref.local1 + ref.local2)
