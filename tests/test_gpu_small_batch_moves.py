"""Small batches in which the tables of several hubs outgrow, at the same time, what one thread block moves:
16,384 to 131,072 new slots, emptied and filled by all blocks of the kernel that runs a small batch's
steps.  The handle is reused, so that the new tables lie on the keys of an earlier stream.  Counts against
the CPU oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_counts_equal, device_edges
from paper_1811_09136_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

# entries before the small batch: each is what half a table of 8,192 to 131,072 slots holds
SIZES = [4096, 4096, 4096, 8192, 8192, 16_384, 16_384, 32_768, 65_536]
PAST = 700  # entries that the small batch adds to each


def stream(seed):
    """(stream, edges before the small batch): every hub's first edges, then PAST more of each in random
    order, then the edges between the hubs, whose wedges are looked up in those tables."""
    r = np.random.default_rng(seed)
    k, leaves = len(SIZES), max(SIZES) + PAST
    first, more = [], []
    for i, size in enumerate(SIZES):
        own = k + r.permutation(leaves)[:size + PAST]
        first.append(np.stack([np.full(size, i), own[:size]], 1))
        more.append(np.stack([np.full(PAST, i), own[size:]], 1))
    first, more = np.concatenate(first), np.concatenate(more)
    hubs = np.array([(i, j) for i in range(k) for j in range(i)])
    e = np.concatenate([r.permutation(first), r.permutation(more), hubs])
    flip = r.random(len(e)) < 0.5
    return gg.EdgeStream(np.where(flip, e[:, 1], e[:, 0]).astype(np.uint32),
                         np.where(flip, e[:, 0], e[:, 1]).astype(np.uint32), k + leaves), len(first)


@pytest.mark.parametrize("m,c", [(2, 2), (300, 300), (20, 100), (1, 3)])
def test_hubs_outgrow_a_block_move_together(m, c):
    from paper_1811_09136_gb300.rept import ReptStream
    n, edges = stream(0)[0].n_nodes, len(stream(0)[0])
    with ReptStream(n, m, c, 7, expected_edges=edges, max_batch=edges) as h:
        for seed in range(4):
            s, before = stream(seed)
            src, dst = device_edges(s)
            h.reset()
            h.ingest(src[:before], dst[:before])
            for off in range(before, edges, 8192):
                h.ingest(src[off:off + 8192], dst[off:off + 8192])
            proc, local = h.counts()
            ref = O.rept_stream(s.src, s.dst, n, m, c, 7, pair_counters=False)
            assert_counts_equal(proc, local.cpu().numpy().view(np.uint64), ref.tau_proc, ref.local1 + ref.local2,
                                f"seed={seed}")
