"""Run in a child process with REPT_LIBRARY naming the bounds-checked build, whose limits on a pool's quads
and a handle's bytes can be lowered (REPT_DEBUG_MAX_QUADS, REPT_DEBUG_MAX_BYTES): streams of several hash
groups that fit only without their colour words, or outgrow the limits with them, against the CPU oracle.
Prints "layout change ok" at the end."""
import os
import struct
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

import oracle as O  # noqa: E402
from paper_1811_09136_gb300 import rept  # noqa: E402
from paper_1811_09136_gb300 import graphgen as gg  # noqa: E402
from paper_1811_09136_gb300.batched import ReptGroup  # noqa: E402
from gpu_helpers import assert_counts_equal, device_edges  # noqa: E402

WORDS, PLAIN = 3, 0  # layouts in a snapshot's header


def limits(quads=None, size=None):
    for name, v in (("REPT_DEBUG_MAX_QUADS", quads), ("REPT_DEBUG_MAX_BYTES", size)):
        if v is None:
            os.environ.pop(name, None)
        else:
            os.environ[name] = str(v)


def layout(handle):
    return struct.unpack_from("<Q", handle.snapshot().tobytes(), 14 * 8)[0]


def reference(s, m, c, flags=0):
    if flags & rept.FLAG_MASCOT:
        ref = O.mascot_stream(s.src, s.dst, s.n_nodes, m, c, 7)
        return ref.tau_proc, ref.local1
    ref = O.rept_stream(s.src, s.dst, s.n_nodes, m, c, 7)
    return ref.tau_proc, ref.local1 + ref.local2


def ingest(handle, s, batch, at=0):
    src, dst = device_edges(s)
    for off in range(at, len(s), batch):
        handle.ingest(src[off:off + batch], dst[off:off + batch])


def check(handle, ref, what):
    proc, local = handle.counts()
    assert_counts_equal(proc, local.cpu().numpy().view(np.uint64), *ref, what)


def main():
    assert os.path.basename(rept.library_path()) == "librept_debug.so", rept.library_path()
    s = gg.cached("powerlaw_20k")
    E = len(s)
    for m, c, flags in [(20, 100, 0), (3, 7, 0), (1, 3, 0), (10, 32, rept.FLAG_MASCOT)]:
        ref = reference(s, m, c, flags)
        what = f"m={m} c={c}"

        def make(edges, batch):
            return rept.ReptStream(s.n_nodes, m, c, 7, expected_edges=edges, max_batch=batch, flags=flags)

        # sized: with room for the words; with a pool that offsets do not span; without the memory for them
        limits()
        with make(E, 1 << 14) as h:
            ingest(h, s, 1 << 14)
            assert layout(h) == WORDS
            size, room = h.stats()["device_bytes"], 32 * 4 * E
            check(h, ref, what + ", words")
        for cap in ({"quads": 12 * E}, {"size": size - 1}, {"size": size - room}):
            limits(**cap)
            with make(E, 1 << 14) as h:
                ingest(h, s, 1 << 14)
                assert layout(h) == PLAIN, cap
                check(h, ref, f"{what}, {cap}")
        # grown: the words go when the pool would pass a limit with them, in whichever batch that is
        for batch in (1000, 30_000, E):
            limits()
            with make(0, 1000) as h:
                ingest(h, s, batch)
                assert layout(h) == WORDS
                words = h.stats()
            pool = words["pool_slots"] // 4  # as the last growth made it
            for cap in ({"quads": pool - 1}, {"size": words["device_bytes"] + 16 * pool}):
                limits(**cap)
                with make(0, 1000) as h:
                    ingest(h, s, batch)
                    assert layout(h) == PLAIN, (cap, batch)
                    assert h.stats()["pool_slots"] // 4 <= cap.get("quads", 1 << 40)
                    check(h, ref, f"{what}, batches of {batch}, {cap}")
                    # the handle's next stream, and its state taken over by one with room
                    h.reset()
                    ingest(h, gg.EdgeStream(s.src[:E // 2], s.dst[:E // 2], s.n_nodes), batch)
                    half = h.snapshot()
                for room, after in ((None, WORDS), (struct.unpack_from("<Q", half.tobytes(), 9 * 8)[0], PLAIN)):
                    limits(quads=room)
                    with make(0, 1000) as h:
                        h.restore(half)
                        assert layout(h) == after
                        limits()
                        ingest(h, s, batch, E // 2)
                        check(h, ref, f"{what}, restored")
    # a group: streams that change their layout beside ones that do not
    streams = [s, gg.chung_lu(3000, 2.2, 9000, graph_seed=1, order_seed=2),
               gg.chung_lu(9000, 2.1, 70_000, graph_seed=3, order_seed=4)]
    params = [(20, 100), (20, 60), (10, 10)]
    for batch in (7000, 1 << 16):
        limits()
        with rept.ReptStream(s.n_nodes, 20, 100, 7, max_batch=1000) as h:
            ingest(h, s, batch)
            pool = h.stats()["pool_slots"] // 4
        limits(quads=pool - 1)
        hs = [rept.ReptStream(x.n_nodes, m, c, 7, max_batch=1000) for x, (m, c) in zip(streams, params)]
        group = ReptGroup(len(hs), graph=False)
        dev = [device_edges(x) for x in streams]
        for off in range(0, E, batch):
            live = [i for i, x in enumerate(streams) if off < len(x)]
            group.ingest([hs[i] for i in live], [dev[i][0][off:off + batch] for i in live],
                         [dev[i][1][off:off + batch] for i in live])
        assert [layout(h) for h in hs[:2]] == [PLAIN, WORDS]
        for h, x, (m, c) in zip(hs, streams, params):
            check(h, reference(x, m, c), f"group, m={m} c={c}")
            h.close()
        group.close()
    limits()
    print("layout change ok")


if __name__ == "__main__":
    main()
