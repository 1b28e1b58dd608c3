"""Timed cases of the SF-sketch library: what a user has it do, through its public entry points.

A monitoring node fills a sketch (one at a time or in chunks, insertions, deletions or a mixed
stream, keys on the device or in pinned host memory), exports its Slim, and a collector answers point
queries on it; many nodes' sketches are updated in one batch, and many Slims are served at once.

Every input is drawn on the GPU from the seed: Zipf ranks by inverting the continuous power law, ranks
to keys by a seeded 64-bit mixing bijection, deletions of occurrences inserted before (strict
turnstile).  exact() restates the insertion, deletion and query rules in numpy.
"""
import math

import numpy as np
import torch

import paper_1701_04148_gb300 as sf


def listed():
    return [
        # a dashboard asks a small exported Slim for a thousand items: launch latency and host calls
        {"name": "query_small", "kind": "query", "d": 4, "w": 4096, "kb": 4, "n": 1000, "ids": 10_000, "zipf": 1.0},
        # all 10^6 flows of a link are read back from its 4 MiB Slim (13-byte 5-tuples)
        {"name": "query_flows", "kind": "query", "d": 4, "w": 1 << 18, "kb": 13, "n": 1_000_000, "ids": 1_000_000,
         "zipf": 0.0},
        # an offline scan of 2^24 64-bit ids on a 64 MiB Slim
        {"name": "query_large", "kind": "query", "d": 4, "w": 1 << 22, "kb": 8, "n": 1 << 24, "ids": 1 << 26,
         "zipf": 1.2},
        # a node's short measurement interval: two chunks of 1,024 items, then its Slim is exported
        {"name": "node_small", "kind": "update", "mode": "insert", "d": 4, "w": 4096, "z": 16, "kb": 4, "chunk": 1024,
         "n": 2048, "ids": 10_000, "zipf": 1.0, "del": 0.0, "host": False, "export": True},
        # the paper's one-at-a-time insertion rule on 100,000 u32 items
        {"name": "one_at_a_time_insert", "kind": "update", "mode": "insert", "d": 4, "w": 4096, "z": 16, "kb": 4,
         "chunk": 1, "n": 100_000, "ids": 10_000, "zipf": 1.0, "del": 0.0, "host": False, "export": False},
        # the same rule on a turnstile stream, a tenth of it deletions
        {"name": "one_at_a_time_mixed", "kind": "update", "mode": "mixed", "d": 4, "w": 4096, "z": 16, "kb": 4,
         "chunk": 1, "n": 100_000, "ids": 10_000, "zipf": 1.0, "del": 0.1, "host": False, "export": False},
        # a link's flows counted without skew, every key of a chunk distinct or nearly so
        {"name": "flows_uniform_insert", "kind": "update", "mode": "insert", "d": 4, "w": 1 << 18, "z": 16, "kb": 13,
         "chunk": 65_536, "n": 1 << 23, "ids": 1_000_000, "zipf": 0.0, "del": 0.0, "host": False, "export": False},
        # a link's skewed flows counted, then a tenth of the counted packets taken back
        {"name": "flows_insert_delete", "kind": "update", "mode": "insert_delete", "d": 4, "w": 1 << 18, "z": 16,
         "kb": 13, "chunk": 65_536, "n": 1 << 23, "ids": 1_000_000, "zipf": 1.0, "del": 0.1, "host": False,
         "export": False},
        # the same from pinned host memory, as packets arrive, the keys moved inside the call
        {"name": "flows_host_insert", "kind": "update", "mode": "insert", "d": 4, "w": 1 << 18, "z": 16, "kb": 13,
         "chunk": 65_536, "n": 1 << 23, "ids": 1_000_000, "zipf": 1.0, "del": 0.0, "host": True, "export": False},
        # a backbone node: 1 GiB of Fat counters, large chunks, a fifth of the stream deletions
        {"name": "backbone_mixed", "kind": "update", "mode": "mixed", "d": 4, "w": 1 << 22, "z": 16, "kb": 8,
         "chunk": 1 << 20, "n": 1 << 24, "ids": 1 << 26, "zipf": 1.2, "del": 0.2, "host": False, "export": False},
        # many nodes' sketches updated by one call, each in four chunks
        {"name": "batch_nodes", "kind": "batch", "sketches": 32, "d": 4, "z": 16, "kb": 4, "rounds": 4,
         "w_lo": 10.0, "w_hi": 16.0, "n_lo": 4.0, "n_hi": 7.0, "del": 0.1},
        # a burst of requests of all sizes against the collector's resident Slims, host to host
        {"name": "collector_burst", "kind": "collector", "sketches": 128, "d": 4, "kb": 4, "requests": 192,
         "w_lo": 10.0, "w_hi": 18.0, "n_lo": 0.0, "n_hi": 16.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: row counts 1 to 8, key widths 3 to 15 bytes, bucket sizes that
    are and are not multiples of four, ragged lengths and widths, chunks from one update to 2^20."""
    what = rng.choice(["query", "query", "one", "small", "flows", "flows", "flows", "backbone", "batch", "collector"])
    d = rng.choice([1, 2, 3, 4, 4, 4, 5, 6, 8])
    kb = rng.choice([3, 4, 4, 5, 8, 8, 13, 13, 15])
    zipf = round(rng.choice([0.0, rng.uniform(0.3, 1.5)]), 3)
    if what == "query":
        n = _log_int(rng, 300, 1 << 23)
        return {"kind": "query", "d": d, "w": _log_int(rng, 1000, 1 << 21), "kb": kb, "n": n,
                "ids": _log_int(rng, 1000, 1 << 22), "zipf": zipf}
    if what == "batch":
        n_lo = rng.uniform(3.0, 5.0)
        return {"kind": "batch", "sketches": rng.randint(2, 32), "d": rng.choice([3, 4, 5]), "z": rng.choice([4, 7, 16]),
                "kb": rng.choice([4, 8, 13]), "rounds": rng.choice([2, 4, 8, 16, 32]), "w_lo": 10.0,
                "w_hi": round(rng.uniform(11.0, 16.0), 2), "n_lo": round(n_lo, 2), "n_hi": round(n_lo + 1.7, 2),
                "del": rng.choice([0.0, 0.1, 0.2])}
    if what == "collector":
        return {"kind": "collector", "sketches": rng.randint(8, 128), "d": rng.choice([3, 4, 5]),
                "kb": rng.choice([4, 8, 13]), "requests": _log_int(rng, 8, 192), "w_lo": 10.0,
                "w_hi": round(rng.uniform(11.0, 17.0), 2), "n_lo": 0.0, "n_hi": round(rng.uniform(8.0, 16.0), 2)}
    case = {"kind": "update", "mode": rng.choice(["insert", "insert_delete", "mixed"]), "d": d, "zipf": zipf,
            "host": False, "export": False}
    if what == "one":
        case.update(w=_log_int(rng, 256, 50_000), z=rng.choice([1, 3, 4, 7, 16]), kb=kb, chunk=1,
                    n=_log_int(rng, 1000, 60_000), ids=_log_int(rng, 1000, 100_000))
    elif what == "small":
        case.update(w=_log_int(rng, 1000, 40_000), z=rng.choice([3, 4, 8, 16]), kb=kb, chunk=_log_int(rng, 64, 8192),
                    n=_log_int(rng, 500, 50_000), ids=_log_int(rng, 1000, 100_000), export=rng.random() < 0.5)
    elif what == "flows":
        case.update(w=_log_int(rng, 4096, 1 << 18), z=rng.choice([3, 7, 8, 16, 16]), kb=kb,
                    chunk=_log_int(rng, 2000, 200_000), n=_log_int(rng, 100_000, 1 << 22),
                    ids=_log_int(rng, 10_000, 1_000_000), host=rng.random() < 0.25)
    else:
        case.update(w=_log_int(rng, 1 << 18, 1 << 22), z=rng.choice([8, 16]), d=rng.choice([3, 4]), kb=rng.choice([4, 8, 13]),
                    chunk=_log_int(rng, 1 << 17, 1 << 20), n=_log_int(rng, 1 << 20, 1 << 23), ids=1 << 24)
    case["del"] = 0.0 if case["mode"] == "insert" else round(rng.uniform(0.05, 0.3), 3)
    return case


# ---- inputs ------------------------------------------------------------------------------------

def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt * 7919 + 17) & 0x7FFF_FFFF_FFFF)
    return g


def _ranks(n, ids, s, g):
    """int64 ranks in [0, ids), rank r with a frequency near (r + 1)^-s (uniform at s = 0)."""
    u = torch.rand(n, dtype=torch.float64, generator=g, device="cuda")
    if s == 0.0:
        x = u * ids
    elif abs(s - 1.0) < 1e-9:
        x = torch.exp(u * math.log(ids + 1.0)) - 1.0
    else:
        x = (u * ((ids + 1.0) ** (1.0 - s) - 1.0) + 1.0).pow(1.0 / (1.0 - s)) - 1.0
    return x.to(torch.int64).clamp_(0, ids - 1)


def _mix(x):
    """A 64-bit bijection (xor-shifts and odd multipliers; int64 arithmetic wraps)."""
    x = (x ^ ((x >> 31) & 0x1FFFFFFFF)) * 0x7FB5D329728EA185
    x = (x ^ ((x >> 27) & 0x1FFFFFFFFF)) * -0x7E25210B43D22BB3
    return x ^ ((x >> 33) & 0x7FFFFFFF)


def _keys(ranks, kb, seed):
    """(n, kb) uint8 keys of the ranks; ranks below 2^64 give distinct keys when kb >= 8.  13-byte
    keys end in a protocol byte (TCP, UDP or ICMP)."""
    lo = _mix(ranks + ((int(seed) & 0xFFFFF) << 40))
    out = torch.empty((ranks.numel(), kb), dtype=torch.uint8, device="cuda")
    out[:, :min(kb, 8)] = lo.view(torch.uint8).view(-1, 8)[:, :min(kb, 8)]
    if kb > 8:
        hi = _mix(lo + 0x1234567)
        out[:, 8:] = hi.view(torch.uint8).view(-1, 8)[:, :kb - 8]
        if kb == 13:
            proto = torch.tensor([6, 17, 1, 6], dtype=torch.uint8, device="cuda")
            out[:, 12] = proto[(hi >> 40) & 3]
    return out


def _stream(mode, n, ids, s, frac, kb, seed, salt=0):
    """insert: (keys, None); insert_delete: (inserted keys, deleted keys), a random `frac` of the
    occurrences deleted in random order; mixed: (keys, int8 operations), n in all, each deletion
    placed uniformly after the insertion it removes."""
    g = _generator(seed, salt)
    if mode == "insert":
        return _keys(_ranks(n, ids, s, g), kb, seed), None
    if mode == "insert_delete":
        ranks = _ranks(n, ids, s, g)
        gone = torch.randperm(n, generator=g, device="cuda")[:max(1, int(n * frac))]
        return _keys(ranks, kb, seed), _keys(ranks[gone], kb, seed)
    n_del = int(n * frac)
    n_ins = n - n_del
    ranks = _ranks(n_ins, ids, s, g)
    gone = torch.randperm(n_ins, generator=g, device="cuda")[:n_del]
    at = gone.to(torch.float64)
    u = torch.rand(n_del, dtype=torch.float64, generator=g, device="cuda")
    place = torch.cat([torch.arange(n_ins, dtype=torch.float64, device="cuda"), at + 0.5 + u * (n_ins - at - 0.5)])
    order = torch.argsort(place, stable=True)
    keys = _keys(torch.cat([ranks, ranks[gone]])[order], kb, seed)
    ops = torch.where(order >= n_ins, -1, 1).to(torch.int8)
    return keys, ops


def _nodes(case, seed):
    """Widths and stream lengths of a batch's or a collector's sketches, log-uniform; they belong to
    the case, so every seed has the same ones."""
    r = np.random.RandomState(case["sketches"] * 131 + case["d"])
    w = [int(round(2.0 ** x)) for x in r.uniform(case["w_lo"], case["w_hi"], case["sketches"])]
    if case["kind"] == "batch":
        n = [int(round(10.0 ** x)) for x in r.uniform(case["n_lo"], case["n_hi"], case["sketches"])]
    else:
        n = [2 * x for x in w]
    return w, n, [float(x) for x in r.uniform(0.5, 1.5, case["sketches"])]


def _requests(case):
    r = np.random.RandomState(case["requests"] * 17 + case["sketches"])
    n = [max(1, int(2.0 ** x)) for x in r.uniform(case["n_lo"], case["n_hi"], case["requests"])]
    return n, [int(x) for x in r.randint(0, case["sketches"], case["requests"])]


def _node_stream(case, k, n, w, s, seed):
    """Node k's stream: a turnstile in a batch, insertions of Zipf(1) items at a collector's node."""
    if case["kind"] == "batch":
        return _stream("mixed" if case["del"] else "insert", n, 10 * w, s, case["del"], case["kb"], seed, 1 + k)
    return _stream("insert", n, w, 1.0, 0.0, case["kb"], seed, 1 + k)


def _request_keys(case, w, seed):
    """The keys of all requests: Zipf-hot ids of the asked node, most of them present in its Slim."""
    n, which = _requests(case)
    return [_keys(_ranks(n[q], 4 * w[which[q]], 1.0, _generator(seed, 5000 + q)), case["kb"], seed).cpu().numpy()
            for q in range(case["requests"])]


def _query_inputs(case, seed):
    fill, _ = _stream("insert", min(1 << 21, 4 * case["w"]), case["ids"], 1.0, 0.0, case["kb"], seed, 1)
    asked = _keys(_ranks(case["n"], case["ids"], case["zipf"], _generator(seed, 2)), case["kb"], seed)
    return fill, asked


def _typed(keys, kb):
    """4- and 8-byte keys as a program holds them, in integers."""
    return keys.view(torch.int32).reshape(-1) if kb == 4 else keys.view(torch.int64).reshape(-1) if kb == 8 else keys


def prepare(case, seed):
    kind = case["kind"]
    if kind == "query":
        fill, asked = _query_inputs(case, seed)
        node = sf.Sketch(case["d"], case["w"], 4, case["kb"], seed=11, chunk=16_384)
        node.insert(fill)
        slim, hdr = node.export_slim()
        node.sync()
        return {"kind": kind, "slim": slim, "hdr": hdr, "keys": _typed(asked, case["kb"])}
    if kind == "update":
        keys, other = _stream(case["mode"], case["n"], case["ids"], case["zipf"], case["del"], case["kb"], seed)
        node = sf.Sketch(case["d"], case["w"], case["z"], case["kb"], seed=5, chunk=case["chunk"])
        node.sync()
        keys = _typed(keys, case["kb"])
        if case["mode"] == "insert_delete":
            other = _typed(other, case["kb"])
        if case["host"]:
            keys = keys.cpu().pin_memory()
            other = other.cpu().pin_memory() if other is not None else None
        return {"kind": kind, "mode": case["mode"], "node": node, "keys": keys, "other": other, "export": case["export"]}
    w, n, s = _nodes(case, seed)
    if kind == "batch":
        items, slots, dict_bytes = [], 0, 0
        for k in range(case["sketches"]):
            chunk = max(2, min(1 << 20, -(-n[k] // case["rounds"])))
            keys, ops = _node_stream(case, k, n[k], w[k], s[k], seed)
            node = sf.Sketch(case["d"], w[k], case["z"], case["kb"], seed=k, chunk=chunk, shared_dict=True)
            items.append((node, _typed(keys, case["kb"]), ops))
            slots += (chunk + 31) // 32 * 32
            dict_bytes += sf.dictionary_bytes(case["d"], w[k], case["z"], case["kb"], k, chunk)
        batch = sf.Batch(case["sketches"], max_round_slots=slots, dict_arena_bytes=dict_bytes)
        batch.sync()
        return {"kind": kind, "batch": batch, "items": items}
    collector = sf.Collector(4 * sum(case["d"] * x + 64 for x in w), case["sketches"])
    for k in range(case["sketches"]):
        keys, _ = _node_stream(case, k, n[k], w[k], 1.0, seed)
        node = sf.Sketch(case["d"], w[k], 4, case["kb"], seed=k, chunk=2048)
        node.insert(keys)
        slim, hdr = node.export_slim()
        node.sync()
        sf.check(collector.upload(k, slim, hdr), "upload")
    asked = _request_keys(case, w, seed)
    answers = np.zeros(sum(len(a) for a in asked), np.int32)
    ends = np.cumsum([len(a) for a in asked])
    requests = [(k, a, answers[e - len(a):e]) for k, a, e in zip(_requests(case)[1], asked, ends)]
    return {"kind": kind, "collector": collector, "requests": requests, "answers": answers}


def run(state):
    kind = state["kind"]
    if kind == "query":
        return sf.query(state["slim"], state["hdr"], state["keys"])
    if kind == "update":
        node, mode = state["node"], state["mode"]
        if mode == "mixed":
            node.update(state["keys"], state["other"])
        else:
            node.insert(state["keys"])
            if mode == "insert_delete":
                node.delete(state["other"])
        out = {"fat": node.fat_view(), "slim": node.slim_view()}
        if state["export"]:
            out["exported"] = node.export_slim()[0]
        return out
    if kind == "batch":
        state["batch"].update(state["items"])
        return [[node.fat, node.slim] for node, _, _ in state["items"]]
    collector = state["collector"]
    tickets = [collector.submit(k, keys, out) for k, keys, out in state["requests"]]
    for t in tickets:
        sf.check(collector.wait(t), "wait")
    return state["answers"]


def _update_work(n, kb, ops, d, w, z):
    """Keys and operations read once; the Slim and Fat counters that n updates can touch read and written
    once.  The arithmetic of a row (hash, two reductions, comparisons) is about 20 operations."""
    fat, slim = min(n * d, d * w * z), min(n * d, d * w)
    return n * (kb + ops) + 8 * (fat + slim), 20 * n * d


def work(case):
    kind, d, kb = case["kind"], case["d"], case["kb"]
    if kind == "query":
        n = case["n"]
        return {"bytes": n * (kb + 4) + 4 * min(n * d, d * case["w"]), "flops": 20 * n * d}
    if kind == "update":
        n = case["n"] + (max(1, int(case["n"] * case["del"])) if case["mode"] == "insert_delete" else 0)
        b, f = _update_work(n, kb, 1 if case["mode"] == "mixed" else 0, d, case["w"], case["z"])
        return {"bytes": b + (8 * d * case["w"] if case["export"] else 0), "flops": f}
    w, n, _ = _nodes(case, 0)
    if kind == "batch":
        each = [_update_work(n[k], kb, 1 if case["del"] else 0, d, w[k], case["z"]) for k in range(case["sketches"])]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    asked = sum(_requests(case)[0])
    return {"bytes": asked * (kb + 4) + 4 * min(asked * d, d * sum(w)), "flops": 20 * asked * d}


# ---- the rules in numpy ------------------------------------------------------------------------

_U = np.uint64


def _fin(x):
    """SplitMix64's output finaliser."""
    x = (x ^ (x >> _U(30))) * _U(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> _U(27))) * _U(0x94D049BB133111EB)
    return x ^ (x >> _U(31))


def _words(keys):
    """Bytes 0-7 and 8-14 of each key, little-endian."""
    full = np.zeros((len(keys), 16), np.uint8)
    full[:, :keys.shape[1]] = keys
    return full.view("<u8")[:, 0].copy(), full.view("<u8")[:, 1].copy()


def _places(keys, d, w, z, seed):
    """(d, n) buckets and slots of the keys."""
    x0, x1 = _words(keys)
    h, f = [], []
    with np.errstate(over="ignore"):
        for i in range(d):
            hashed = _fin(x0 ^ _fin(np.array([seed], _U) + _U(i + 1) * _U(0x9E3779B97F4A7C15)))
            if keys.shape[1] > 8:
                hashed = _fin(hashed ^ x1)
            h.append((((hashed >> _U(32)) * _U(w)) >> _U(32)).astype(np.int64))
            f.append((((hashed & _U(0xFFFFFFFF)) * _U(z)) >> _U(32)).astype(np.int64))
    return np.array(h), np.array(f)


def _apply(A, B, keys, ops, seed, chunk):
    """One call's updates on the Slim A (d, w) and the Fat B (d, w, z), both int64: chunk by chunk the
    Fat takes every operation; a key inserted c times raises its Slim counters to min(chunk-start
    minimum + c, its chunk-end Fat minimum); a deletion first lowers them to the bucket's maximum."""
    d, w, z = B.shape
    h, f = _places(keys, d, w, z, seed)
    rows = np.arange(d)
    if chunk == 1:
        for t in range(len(keys)):
            ht, ft = h[:, t], f[:, t]
            B[rows, ht, ft] += ops[t]
            if ops[t] > 0:
                a = A[rows, ht]
                A[rows, ht] = np.maximum(a, min(a.min() + 1, B[rows, ht, ft].min()))
            else:
                A[rows, ht] = np.minimum(A[rows, ht], B[rows, ht].max(1))
        return
    x0, x1 = _words(keys)
    for t in range(0, len(keys), chunk):
        c = slice(t, min(t + chunk, len(keys)))
        hc, fc, up = h[:, c], f[:, c], ops[c] > 0
        for i in range(d):
            np.add.at(B[i], (hc[i], fc[i]), ops[c].astype(np.int64))
        ids = np.stack([x0[c][up], x1[c][up]], 1)
        _, first, count = np.unique(ids.view([("a", "<u8"), ("b", "<u8")]).ravel(), return_index=True, return_counts=True)
        hk, fk = hc[:, up][:, first], fc[:, up][:, first]
        if len(first):
            low = np.min([A[i, hk[i]] for i in range(d)], 0)
            end = np.min([B[i, hk[i], fk[i]] for i in range(d)], 0)
            target = np.minimum(low + count, end)
        for i in range(d):
            gone = np.unique(hc[i, ~up])
            A[i, gone] = np.minimum(A[i, gone], B[i, gone].max(1))
        for i in range(d):
            if len(first):
                np.maximum.at(A[i], hk[i], target)


def _read(A, keys, seed):
    h, _ = _places(keys, A.shape[0], A.shape[1], 1, seed)
    return np.min([A[i, h[i]] for i in range(A.shape[0])], 0)


def _filled(d, w, z, keys, seed, chunk):
    A, B = np.zeros((d, w), np.int64), np.zeros((d, w, z), np.int64)
    _apply(A, B, keys, np.ones(len(keys), np.int64), seed, chunk)
    return A


def exact(case, seed):
    """What run() returns on a fresh state; None where numpy would take too long."""
    kind, d, kb = case["kind"], case["d"], case["kb"]
    if kind == "query":
        if case["w"] > 1 << 19 or case["n"] > 1 << 22:
            return None
        fill, asked = _query_inputs(case, seed)
        A = _filled(d, case["w"], 4, fill.cpu().numpy(), 11, 16_384)
        return _read(A, asked.cpu().numpy(), 11)
    if kind == "update":
        if case["n"] > (200_000 if case["chunk"] == 1 else 2_000_000 if case["chunk"] >= 1024 else 50_000):
            return None
        keys, other = _stream(case["mode"], case["n"], case["ids"], case["zipf"], case["del"], kb, seed)
        A, B = np.zeros((d, case["w"]), np.int64), np.zeros((d, case["w"], case["z"]), np.int64)
        keys = keys.cpu().numpy()
        ops = other.cpu().numpy().astype(np.int64) if case["mode"] == "mixed" else np.ones(len(keys), np.int64)
        _apply(A, B, keys, ops, 5, case["chunk"])
        if case["mode"] == "insert_delete":
            gone = other.cpu().numpy()
            _apply(A, B, gone, -np.ones(len(gone), np.int64), 5, case["chunk"])
        out = {"fat": B, "slim": A}
        if case["export"]:
            out["exported"] = A.ravel().copy()
        return out
    w, n, s = _nodes(case, seed)
    if sum(n) > 2_000_000:
        return None
    if kind == "batch":
        out = []
        for k in range(case["sketches"]):
            keys, ops = _node_stream(case, k, n[k], w[k], s[k], seed)
            A, B = np.zeros((d, w[k]), np.int64), np.zeros((d, w[k], case["z"]), np.int64)
            ops = ops.cpu().numpy().astype(np.int64) if ops is not None else np.ones(len(keys), np.int64)
            _apply(A, B, keys.cpu().numpy(), ops, k, max(2, min(1 << 20, -(-n[k] // case["rounds"]))))
            out.append([B.ravel(), A.ravel()])
        return out
    slims = [_filled(d, w[k], 4, _node_stream(case, k, n[k], w[k], 1.0, seed)[0].cpu().numpy(), k, 2048)
             for k in range(case["sketches"])]
    return np.concatenate([_read(slims[k], a, k) for k, a in zip(_requests(case)[1], _request_keys(case, w, seed))])
