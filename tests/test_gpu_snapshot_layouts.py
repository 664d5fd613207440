"""Snapshots whose header names a layout of the blocks that the handle's configuration cannot have are refused,
and leave the handle as it was."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_counts_equal, device_edges
from paper_1811_09136_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

COLOURS_AT = 14 * 8  # of the header


@pytest.mark.parametrize("m,c,others", [(10, 10, (0, 2, 3, 4, 1 + (1 << 32))), (300, 300, (0, 1, 3, 7)),
                                        (20, 100, (1, 2, 4, 8, 3 + (1 << 32), (1 << 64) - 1)), (20, 140, (1, 2, 3, 5))])
def test_unknown_layouts_are_refused(m, c, others):
    from paper_1811_09136_gb300.rept import ReptError, ReptStream
    s = gg.chung_lu(2000, 2.2, 9000, graph_seed=m, order_seed=c)
    src, dst = device_edges(s)
    with ReptStream(s.n_nodes, m, c, 3, max_batch=4096) as h:
        h.ingest(src[:5000], dst[:5000])
        snap = h.snapshot()
        for other in others:
            bad = np.array(snap, copy=True)
            bad[COLOURS_AT:COLOURS_AT + 8] = np.frombuffer(np.uint64(other).tobytes(), dtype=np.uint8)
            with pytest.raises(ReptError):
                h.restore(bad)
        h.ingest(src[5000:], dst[5000:])
        proc, local = h.counts()
        ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 3, pair_counters=False)
        assert_counts_equal(proc, local.cpu().numpy().view(np.uint64), ref.tau_proc, ref.local1 + ref.local2)
