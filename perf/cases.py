"""Timed cases of the REPT counting path, through the package's public entry points.

A pass counts one edge stream (or a set of them) from empty to its estimates, the way the callers in this
repository do: reset the handle, append the edges batch by batch, read the estimates and counters.
Graphs are made on the GPU from the seed: distinct undirected edges, no self-loops, random
orientation, scrambled node ids, random stream order (heavy-tailed Chung-Lu and R-MAT graphs, the two
families of paper_1811_09136_gb300.graphgen).  The sizes are those of the repository's workloads,
accuracy sweeps and tests.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1811_09136_gb300 import batched, rept

GOLDEN = 0x9E3779B97F4A7C15
MASK64 = (1 << 64) - 1


# ---------------------------------------------------------------------------------------- cases
def _stream(name, kind, n_nodes, edges, m, c, batch, gamma=2.1, cap=0.0, entry="device", sized=True, mascot=False):
    """One stream.  entry: "device" (edges in device memory) or "host" (pinned host arrays).  sized: the
    handle is created with the stream's length (expected_edges), else its pool grows as needed."""
    return {"name": name, "kind": kind, "n_nodes": n_nodes, "edges": edges, "gamma": gamma, "cap": cap, "m": m, "c": c,
            "batch": batch, "entry": entry, "sized": sized, "mascot": mascot, "streams": 1}


def _mix(name, streams, n_min, n_max, epn_min, epn_max, batch, persistent=False, spec_seed=1000):
    """Many independent streams through one group, half R-MAT and half Chung-Lu, p in {0.1, 0.05, 0.01};
    their sizes and p come from spec_seed."""
    return {"name": name, "kind": "mix", "streams": streams, "spec_seed": spec_seed, "n_min": n_min, "n_max": n_max, "epn_min": epn_min,
            "epn_max": epn_max, "batch": batch, "persistent": persistent}


def listed():
    return [
        # the shortest call: a window of a thousand edges counted at once (latency of a whole pass)
        _stream("short_window", "chung_lu", 300, 1000, 5, 5, 1 << 20, gamma=2.3),
        # edges arriving in small batches: per-batch latency decides
        _stream("small_batches", "chung_lu", 20_000, 200_000, 10, 10, 4096, gamma=2.3),
        # the 20,000-node power-law workload, one batch
        _stream("powerlaw_20k", "chung_lu", 20_000, 200_000, 10, 10, 1 << 20, gamma=2.3),
        # a handle made without a length hint: the pool is checked and grown batch by batch
        _stream("unsized", "chung_lu", 100_003, 1_500_001, 20, 20, 1 << 16, gamma=2.2, sized=False),
        # the R-MAT scale-20 workload at c = m (every edge stored once) ...
        _stream("rmat_s20", "rmat", 1 << 20, 15_700_820, 100, 100, 1 << 20),
        # ... and with c < m processors (30 % of the edges stored)
        _stream("rmat_s20_c30", "rmat", 1 << 20, 15_700_820, 100, 30, 1 << 20),
        # the same family from pinned host memory, estimates back to the host (end to end)
        _stream("host_edges", "rmat", 1 << 18, 3_900_000, 100, 100, 1 << 18, entry="host"),
        # the accuracy sweeps' 200,000-node graph with more colours than an entry's spare bits hold
        _stream("many_colours", "chung_lu", 200_000, 2_000_000, 300, 300, 1 << 18),
        # ... with a partial last group (Algorithm 2, pair counters)
        _stream("partial_group", "chung_lu", 200_000, 2_000_000, 100, 160, 1 << 20),
        # parallel MASCOT, the accuracy sweeps' other arm
        _stream("mascot", "chung_lu", 20_000, 200_000, 10, 32, 1 << 20, gamma=2.3, mascot=True),
        # the 4M-node workload: hub-heavy, five hash groups; the largest stream
        _stream("five_groups", "chung_lu", 1 << 22, 64 << 20, 20, 100, 1 << 20, cap=50_000.0),
        # many tenants' streams side by side, fed chunk by chunk through one group (batched path, serving)
        _mix("many_streams", 48, 1e4, 1e5, 10.0, 40.0, 1 << 16),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if rng.random() < 0.25:
        return _mix("", rng.randint(2, 60), 1e4, math.exp(rng.uniform(math.log(2e4), math.log(3e5))), 10.0,
                    rng.uniform(12.0, 40.0), log_int(1 << 14, 1 << 20), persistent=rng.random() < 0.3,
                    spec_seed=rng.randrange(1 << 20))
    n = log_int(300, 2_000_000)
    edges = min(int(n * rng.uniform(3.0, 32.0)), n * (n - 1) // 8, 20_000_000)
    m, c, mascot = rng.choice([(2, 2, False), (5, 5, False), (10, 10, False), (20, 20, False), (100, 100, False),
                               (100, 30, False), (10, 3, False), (300, 300, False), (300, 120, False),
                               (20, 100, False), (10, 20, False), (10, 32, False), (100, 160, False), (10, 8, True),
                               (10, 32, True), (100, 20, True)])
    if m < 20 or c > m:  # dense colours and several groups close many more wedges
        edges = min(edges, 2_500_000)
    batch = max(log_int(512, 1 << 20), edges // 400)
    return _stream("", rng.choice(["chung_lu", "rmat"]), n, edges, m, c, batch, gamma=rng.uniform(2.1, 2.5),
                   entry=rng.choice(["device", "device", "host"]), sized=rng.random() < 0.7, mascot=mascot)


# ---------------------------------------------------------------------------------------- inputs
def _distinct(draw_pairs, n, want, gen):
    """Up to `want` distinct undirected edges from repeated draws, in random order and orientation."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    for _ in range(12):
        missing = want - keys.numel()
        if missing <= 0:
            break
        a, b = draw_pairs(int(missing * 1.15) + 64)
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        new = (lo * n + hi)[lo != hi]
        keys = torch.unique(torch.cat([keys, new]))
    keys = keys[torch.randperm(keys.numel(), generator=gen, device="cuda")][:want]
    perm = torch.randperm(n, generator=gen, device="cuda")
    a, b = perm[keys // n], perm[keys % n]
    flip = torch.rand(keys.numel(), generator=gen, device="cuda") < 0.5
    return torch.where(flip, b, a).to(torch.int32), torch.where(flip, a, b).to(torch.int32)


def _chung_lu(n, gamma, edges, cap, gen):
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    w *= 2.0 * edges / w.sum()
    if cap > 0:
        for _ in range(50):
            over = w >= cap
            rest = w[~over].sum()
            scale = (2.0 * edges - cap * over.sum()) / rest
            if scale <= 1.0 + 1e-12:
                break
            w = torch.where(over, torch.full_like(w, cap), w * scale).clamp_(max=cap)
    cdf = torch.cumsum(w, 0)

    def pairs(k):
        x = torch.rand((2, k), dtype=torch.float64, device="cuda", generator=gen) * cdf[-1]
        e = torch.searchsorted(cdf, x, right=True).clamp_(max=n - 1)
        return e[0], e[1]

    return _distinct(pairs, n, edges, gen)


def _rmat(n, edges, gen, a=0.57, b=0.19, c=0.19):
    scale = max(1, math.ceil(math.log2(n)))

    def pairs(k):
        x = torch.zeros(k, dtype=torch.int64, device="cuda")
        y = torch.zeros(k, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            r = torch.rand(k, device="cuda", generator=gen)
            x = (x << 1) | (r >= a + b)
            y = (y << 1) | (((r >= a) & (r < a + b)) | (r >= a + b + c))
        return x, y

    return _distinct(pairs, 1 << scale, edges, gen), 1 << scale


def _graph(kind, n, edges, gamma, cap, seed):
    """(src, dst, number of node ids)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "rmat":
        (src, dst), n = _rmat(n, edges, gen)
    else:
        src, dst = _chung_lu(n, gamma, edges, cap, gen)
    return src, dst, n


def _mix_specs(case, seed):
    r = np.random.default_rng(case["spec_seed"])
    specs = []
    for i in range(case["streams"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        edges = int(n * r.uniform(case["epn_min"], case["epn_max"]))
        m = int(r.choice([10, 20, 100]))
        specs.append((("rmat", "chung_lu")[int(r.integers(2))], n, edges, float(r.uniform(2.1, 2.5)), m,
                      _hash_seed(seed * 1009 + i), seed * 1009 + i))
    return specs


def _hash_seed(seed):
    return (seed * GOLDEN + 1) & (MASK64 >> 1)


def _pinned(t):
    return t.cpu().pin_memory().numpy().view(np.uint32)


def prepare(case, seed):
    if case["kind"] == "mix":
        handles, srcs, dsts = [], [], []
        for kind, n, edges, gamma, m, hseed, gseed in _mix_specs(case, seed):
            src, dst, n = _graph(kind, n, edges, gamma, 0.0, gseed)
            handles.append(rept.ReptStream(n, m, m, hseed, expected_edges=src.numel(),
                                           max_batch=min(case["batch"], max(1, src.numel()))))
            srcs.append(src)
            dsts.append(dst)
        group = batched.ReptGroup(len(handles), graph=True, persistent=case["persistent"])
        return {"case": case, "handles": handles, "srcs": srcs, "dsts": dsts, "group": group}
    src, dst, n = _graph(case["kind"], case["n_nodes"], case["edges"], case["gamma"], case["cap"], seed)
    edges = src.numel()
    handle = rept.ReptStream(n, case["m"], case["c"], _hash_seed(seed),
                             expected_edges=edges if case["sized"] else 0,
                             max_batch=min(case["batch"], max(1, edges)),
                             flags=rept.FLAG_MASCOT if case["mascot"] else 0)
    state = {"case": case, "handle": handle}
    if case["entry"] == "host":
        state["src"], state["dst"] = _pinned(src), _pinned(dst)
        state["out"] = torch.empty(n, dtype=torch.float64).pin_memory().numpy()
    else:
        state["src"], state["dst"] = src, dst
    return state


# ---------------------------------------------------------------------------------------- a pass
def _run_mix(state):
    batch, group = state["case"]["batch"], state["group"]
    handles, srcs, dsts = state["handles"], state["srcs"], state["dsts"]
    for h in handles:
        h.reset()
    rounds = max((s.numel() + batch - 1) // batch for s in srcs)
    for r in range(rounds):
        live = [j for j, s in enumerate(srcs) if r * batch < s.numel()]
        group.ingest([handles[j] for j in live], [srcs[j][r * batch:(r + 1) * batch] for j in live],
                     [dsts[j][r * batch:(r + 1) * batch] for j in live])
    tau_hat, tau_i, tau_v = [], [], []
    for h in handles:
        i, v = h.counts()
        tau_i.append(i)
        tau_v.append(v)
        tau_hat.append(h.estimates(local=False)[0])
    return {"tau_hat": np.array(tau_hat), "tau_i": np.concatenate(tau_i), "tau_v": tau_v}


def run(state):
    case = state["case"]
    if case["kind"] == "mix":
        return _run_mix(state)
    h, src, dst, batch = state["handle"], state["src"], state["dst"], state["case"]["batch"]
    h.reset()
    if case["entry"] == "host":
        h.ingest_host(src, dst, batch=batch)
        tau_hat, tau_hat_v = h.estimates_host(out=state["out"])
    else:
        for off in range(0, src.numel(), batch):
            h.ingest(src[off:off + batch], dst[off:off + batch])
        tau_hat, tau_hat_v = h.estimates()
    tau_i, tau_v = h.counts()
    out = {"tau_hat": tau_hat, "tau_hat_v": tau_hat_v, "tau_i": tau_i, "tau_v": tau_v}
    if case["c"] > case["m"] and case["c"] % case["m"] and not case["mascot"]:
        out["eta_i"], out["eta_v"], out["tau_v_full"], out["tau_v_part"] = h.pair_counts()
    return out


def work(case):
    """One pass has to read the edges and write the estimates and counters; for every edge it needs the
    smaller endpoint's kept neighbours once.  The neighbour reads depend on the graph: they are not
    known from the sizes alone, so only the streams and results are counted as bytes, and one hash
    (about 31 integer operations) per edge and hash group as operations."""
    if case["kind"] == "mix":
        n = math.sqrt(case["n_min"] * case["n_max"]) * case["streams"]
        edges = n * 0.5 * (case["epn_min"] + case["epn_max"])
        return {"bytes": int(8 * edges + 8 * n), "flops": int(31 * edges)}
    n, e = case["n_nodes"], case["edges"]
    groups = case["c"] if case["mascot"] else -(-case["c"] // case["m"])
    return {"bytes": 8 * e + 16 * n + 8 * case["c"] + 8, "flops": 31 * groups * e}


# ---------------------------------------------------------------------------------------- 64-bit values
def _i64(x):
    x &= MASK64
    return x - (1 << 64) if x >> 63 else x


def _shr(x, s):
    return (x >> s) & ((1 << (64 - s)) - 1)


def _colour(lo, hi, seed, k, m):
    """h_k of the edges {lo, hi} (lo < hi): SplitMix64((lo << 32 | hi) xor s_k) mod m."""
    z = (((lo << 32) | hi) ^ _i64(seed + k * GOLDEN)) + _i64(GOLDEN)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    return (_shr(z, 32) * ((1 << 32) % m) + (z & 0xFFFFFFFF) % m) % m


def _exact_counts(src, dst, n, m, c, seed, mascot, budget=1 << 30):
    """(tau^(i), sum_i tau_v^(i)) by enumerating, per hash group and kept colour, every pair of stored
    edges that share a node and looking up the edge that closes it; None if there are too many pairs."""
    a, b = src.to(torch.int64), dst.to(torch.int64)
    lo, hi = torch.minimum(a, b), torch.maximum(a, b)
    keys, order = torch.sort(lo * n + hi)
    tau_i = torch.zeros(c, dtype=torch.int64, device="cuda")
    tau_v = torch.zeros(n, dtype=torch.int64, device="cuda")
    t = torch.arange(a.numel(), device="cuda")
    groups = c if mascot else -(-c // m)
    for k in range(groups):
        col = _colour(lo, hi, seed, k, m)
        proc = torch.where(col == 0, k, c) if mascot else k * m + col
        keep = proc < c
        p2, t2 = proc[keep].repeat(2), t[keep].repeat(2)
        x2, y2 = torch.cat([a[keep], b[keep]]), torch.cat([b[keep], a[keep]])
        o = torch.argsort((x2 * c + p2) * (a.numel() + 1) + t2)  # runs of one node and processor, oldest first
        p2, t2, x2, y2 = p2[o], t2[o], x2[o], y2[o]
        run = x2 * c + p2
        if run.numel() == 0:
            continue
        new = torch.ones_like(run, dtype=torch.bool)
        new[1:] = run[1:] != run[:-1]
        pos = torch.arange(run.numel(), device="cuda")
        rank = pos - torch.cummax(torch.where(new, pos, torch.zeros_like(pos)), 0).values
        ends = torch.cumsum(rank, 0)
        budget -= int(ends[-1])
        if budget < 0:
            return None
        step, at, total = 1 << 26, 0, int(ends[-1])
        while at < total:  # pairs at .. at + step - 1: the later entry q and an earlier one of its run
            q = torch.arange(at, min(at + step, total), device="cuda")
            e = torch.searchsorted(ends, q, right=True)
            first = pos[e] - 1 - (q - (ends[e] - rank[e]))
            u, v = torch.minimum(y2[e], y2[first]), torch.maximum(y2[e], y2[first])
            want = u * n + v
            f = torch.searchsorted(keys, want).clamp_(max=keys.numel() - 1)
            hit = (keys[f] == want) & (order[f] > t2[e])
            e, u, v = e[hit], u[hit], v[hit]
            tau_i += torch.bincount(p2[e], minlength=c)
            for nodes in (u, v, x2[e]):
                tau_v += torch.bincount(nodes, minlength=n)
            at += step
    return tau_i, tau_v


def _factor(m, c, mascot):
    return float(m) * m / c if mascot or c <= m else float(m) / (c // m)


def exact(case, seed):
    if case["kind"] == "mix":
        tau_hat, tau_i, tau_v = [], [], []
        for kind, n, edges, gamma, m, hseed, gseed in _mix_specs(case, seed):
            src, dst, n = _graph(kind, n, edges, gamma, 0.0, gseed)
            got = _exact_counts(src, dst, n, m, m, hseed, False, budget=1 << 31)
            if got is None:
                return None
            tau_hat.append(float(got[0].sum()) * _factor(m, m, False))
            tau_i.append(got[0].cpu().numpy().view(np.uint64))
            tau_v.append(got[1])
        return {"tau_hat": np.array(tau_hat), "tau_i": np.concatenate(tau_i), "tau_v": tau_v}
    m, c, mascot = case["m"], case["c"], case["mascot"]
    if c > m and c % m and not mascot or case["edges"] > 20_000_000:
        return None
    src, dst, n = _graph(case["kind"], case["n_nodes"], case["edges"], case["gamma"], case["cap"], seed)
    got = _exact_counts(src, dst, n, m, c, _hash_seed(seed), mascot)
    if got is None:
        return None
    f = _factor(m, c, mascot)
    tau_hat_v = got[1].to(torch.float64) * f
    return {"tau_hat": float(got[0].sum()) * f,
            "tau_hat_v": tau_hat_v.cpu().numpy() if case["entry"] == "host" else tau_hat_v,
            "tau_i": got[0].cpu().numpy().view(np.uint64), "tau_v": got[1]}
