"""The filtered list scans of the intersection and the block layouts they read, against the CPU oracle.

Lists and larger endpoints at the edges of the scan's rows, pieces and units (32-entry small edges,
128-entry rows, 1,024-entry pieces and warp units, 4,096-entry units, filters with several entries per
word), in every colour layout; and snapshots of the older layout (lists of {entry, stream index} pairs).
"""
import struct

import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_counts_equal, device_edges, gpu_run
from paper_1811_09136_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu

# (m, c): colour in the entry, a word beside it, several groups in one word, one bit per group, no words
LAYOUTS = [(2, 2), (10, 7), (300, 300), (3, 7), (20, 100), (1, 3), (100, 500)]


def hub_stream(n_l, lists, seed):
    """A hub of n_l neighbours and one node per length in `lists` with that many of them, those edges in
    random order among 40,000 others, then an edge from each such node to the hub."""
    r = np.random.default_rng(seed)
    n = 30_000
    first = 1 + len(lists)
    near = first + r.permutation(n - first)[:n_l]
    pairs = [(0, int(x)) for x in near]
    for i, k in enumerate(lists):
        own = r.permutation(near)[:min(k, n_l)] if i % 2 else first + r.permutation(n - first)[:k]
        pairs += [(1 + i, int(x)) for x in own]
    key = {(min(a, b), max(a, b)) for a, b in pairs}
    a, b = first + r.integers(n - first, size=40_000), first + r.integers(n - first, size=40_000)
    key |= {(int(min(x, y)), int(max(x, y))) for x, y in zip(a, b) if x != y}
    e = np.array(sorted(key), dtype=np.uint32)
    e = e[r.permutation(len(e))]
    e = np.concatenate([e, np.array([(1 + i, 0) for i in range(len(lists))], dtype=np.uint32)])
    flip = r.random(len(e)) < 0.5
    return gg.EdgeStream(np.where(flip, e[:, 1], e[:, 0]).astype(np.uint32),
                         np.where(flip, e[:, 0], e[:, 1]).astype(np.uint32), n)


@pytest.mark.parametrize("m,c", LAYOUTS)
@pytest.mark.parametrize("n_l", [33, 1024, 1025, 4097, 17_000])
def test_lists_and_hubs_at_the_scan_edges(n_l, m, c):
    s = hub_stream(n_l, [31, 32, 33, 127, 128, 129, 257, 1023, 1024, 1025, 1153], seed=n_l + m)
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 9, pair_counters=False)
    for batch in (len(s), (1 << 15) - 1, 1000):  # grouped; nearly all edges small (below 2^15)
        proc, local, _, _, _ = gpu_run(s, m, c, 9, batch=batch)
        assert_counts_equal(proc, local, ref.tau_proc, ref.local1 + ref.local2, f"batch={batch}")


def pair_list_snapshot(snap):
    """A snapshot rewritten in the older format (version 3): lists of {entry word, stream index} pairs,
    no colour words beside the stream indices, a header without the layout field."""
    h = list(struct.unpack_from("<15Q", snap.tobytes()))
    n, c, colours = h[5], h[3], h[14]
    raw = snap.tobytes()[15 * 8:]
    meta = np.frombuffer(raw, dtype="<u4", count=4 * n).reshape(n, 4).copy()
    at = 16 * n
    tallies = raw[at:at + 8 * n + 8 * c]
    at += 8 * n + 8 * c
    pool = np.frombuffer(raw, dtype="<u4", count=8 * h[9], offset=at)
    rest = raw[at + 32 * h[9]:]
    assert not meta[:, 2:].any()  # no batch in progress
    out, top = [], 0
    for x in range(n):
        cnt = int(meta[x, 1])
        if not cnt:
            continue
        lg = max(2, (2 * cnt - 1).bit_length())
        cap, slots = 1 << lg, max(4, 1 << (lg - 1))
        b = pool[8 * int(meta[x, 0]):]
        table = cap * (3 if colours == 3 else 2)
        words = b[table:table + cnt]
        aux = table + slots
        if colours in (1, 2):  # stream indices from the interleaved table
            buckets = b[:2 * cap].reshape(-1, 2, 4)
            index = dict(zip(buckets[:, 0].ravel().tolist(), buckets[:, 1].ravel().tolist()))
            t = [index[int(w) & (0xFFFFFF if colours == 1 else 0xFFFFFFFF)] for w in words]
        else:
            t = b[aux:aux + cnt * (2 if colours == 3 else 1)][::2 if colours == 3 else 1]
        quads = (cap + slots + (max(4, cap // 4) if colours == 2 else 0)) // 4
        block = np.zeros(8 * quads, dtype="<u4")
        block[2 * cap:2 * cap + 2 * cnt:2] = words
        block[2 * cap + 1:2 * cap + 1 + 2 * cnt:2] = t
        if colours == 2:
            block[2 * (cap + slots):2 * (cap + slots) + cnt] = b[2 * (cap + slots):2 * (cap + slots) + cnt]
        meta[x, 0] = top
        top += quads
        out.append(block)
    h[1], h[9] = 3, top
    return np.frombuffer(struct.pack("<14Q", *h[:14]) + meta.tobytes() + tallies + np.concatenate(out).tobytes() + rest,
                         dtype=np.uint8)


@pytest.mark.parametrize("m,c", LAYOUTS)
def test_older_snapshots_resume_exactly(m, c):
    from paper_1811_09136_gb300.rept import ReptStream, ReptError
    s = gg.chung_lu(3000, 2.2, 25_000, graph_seed=m + c, order_seed=8)
    src, dst = device_edges(s)
    half = 12_345
    with ReptStream(s.n_nodes, m, c, 9, max_batch=4096) as a:
        a.ingest(src[:half], dst[:half])
        snap = pair_list_snapshot(a.snapshot())
    with ReptStream(s.n_nodes, m, c, 9, max_batch=64) as b:  # (a small pool, which the restore grows)
        with pytest.raises(ReptError):
            b.restore(snap[:-1])
        b.restore(snap)
        b.ingest(src[half:], dst[half:])
        proc, local = b.counts()
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 9)
    assert_counts_equal(proc, local.cpu().numpy().view(np.uint64), ref.tau_proc, ref.local1 + ref.local2)
