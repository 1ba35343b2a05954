"""The work a user of this library has it do, as measurable cases.

Every case goes through the Python entry points (vf_build, vf_build_batch,
vf_query, vf_query_batch) on inputs drawn from a seed. Two kinds of outputs
come back: what a function decodes for its members (the values it was built
from, whatever the cells hold) and what a filter says of members and of keys
outside the set (a filter accepts a few of the latter, and which ones depends
on the cells, which are not the same from build to build).

A build case builds a structure, asks it for every key and releases it; a
query case keeps the structure, as a serving program does.
"""
import math

import torch

import paper_2503_18397_gb300 as vf
from paper_2503_18397_gb300 import synth

DEV = "cuda"


def _case(name, op, n, m, kind, b, keys="u64", mode="auto", count=1):
    return {"name": name, "op": op, "n": n, "m": m, "kind": kind, "b": b, "keys": keys, "mode": mode, "count": count}


def listed():
    return [
        # one request of a serving program: a thousand lookups in a function that L2 holds
        _case("lookup-1k", "query", 1 << 20, 1000, "func", 8),
        # bulk membership test against the 10^8-key filter (110 MB: about L2's size), half members
        _case("probe-filter", "query", 100_000_000, 50_000_003, "filter", 8),
        # lookups in a function whose 0.9 GB of cells lie in HBM
        _case("probe-hbm", "query", 400_000_000, 30_000_001, "func", 16),
        # lookups of byte strings (8..64 bytes), small elimination shards
        _case("probe-strings", "query", 3_000_017, 3_000_017, "func", 16, keys="bytes", mode="lge"),
        # what the serving loop launches: many requests of uneven sizes against resident structures
        _case("serve-batch", "serve", 300_000, 1_500_000, "mixed", 0, count=96),
        # keys and answers in pinned host memory: chunks copied in, probed and copied out
        _case("probe-host", "host", 10_000_000, 33_554_467, "func", 8),
        # the smallest structures: one elimination shard
        _case("build-10k", "build", 10_007, 10_007, "func", 8),
        # one unsharded fuse graph
        _case("build-1m", "build", 1 << 20, 1 << 20, "func", 8),
        # byte strings in small elimination shards
        _case("build-strings", "build", 10_000_000, 10_000_000, "func", 16, keys="bytes", mode="lge"),
        # the headline: a sharded filter, retries included
        _case("build-1e8", "build", 100_000_000, 200_000_000, "filter", 8),
        # the largest: many shards, vertex words far beyond L2
        _case("build-1e9", "build", 1_000_000_000, 200_000_000, "filter", 8),
        # many uneven structures in one call
        _case("build-batch", "batch", 1000, 1_000_000, "mixed", 0, count=512),
    ]


def _log(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    # an unsharded fuse graph of 0.80 to 0.98 million keys rounds to a segment
    # count at which most seeds leave a 2-core: a build there may end in VF_EBUILD
    return n + 200_000 if 795_000 < n < 990_000 else n


def draw(rng):
    op = rng.choice(["query", "query", "build", "build", "build", "serve", "host", "batch"])
    if op == "serve":
        lo = _log(rng, 20_000, 300_000)
        return _drawn(op, lo, _log(rng, lo, 2_000_000), "mixed", 0, count=rng.randint(8, 200))
    if op == "batch":
        return _drawn(op, 1000, _log(rng, 50_000, 1_000_000), "mixed", 0, count=_log(rng, 16, 512))
    if op == "host":
        return _drawn(op, _log(rng, 100_000, 50_000_000), _log(rng, 10_000, 50_000_000), "func", rng.choice([8, 16, 32]))
    shape = rng.choice(["func", "func", "filter", "bytes", "mwhc", "fuse4"])
    if shape == "bytes":
        n = _log(rng, 2_000, 5_000_000)
        return _drawn(op, n, n, "func", rng.choice([1, 8, 16, 32]), keys="bytes", mode=rng.choice(["auto", "lge"]))
    if shape == "func":
        n = _log(rng, 1_000, 200_000_000)
        b = rng.choice([1, 8, 9, 13, 16, 17, 32, 40])
        return _drawn(op, n, n if op == "build" else min(n, _log(rng, 1_000, 50_000_000)), "func", b)
    lo = {"filter": 1_000_000, "mwhc": 1_000_000, "fuse4": 2_000_000}[shape]
    n = _log(rng, lo, 300_000_000 if op == "build" else 100_000_000)
    return _drawn(op, n, n if op == "build" else _log(rng, 500_000, 50_000_000), "filter", 8,
                  mode="auto" if shape == "filter" else shape)


def _drawn(op, n, m, kind, b, keys="u64", mode="auto", count=1):
    c = _case("", op, n, m, kind, b, keys, mode, count)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _params(c, kind, b, seed):
    p = vf.vf_params_default(kind=vf.FILTER if kind == "filter" else vf.FUNC, b=b, seed=seed,
                             key_kind=vf.KEYS_BYTES if c["keys"] == "bytes" else vf.KEYS_U64)
    if c["mode"] == "lge":
        p.mode = vf.MODE_LGE
    elif c["mode"] == "mwhc":  # the configuration of the MWHC workload
        p.mode, p.eps, p.eta = vf.MODE_MWHC, 0.01, 1e-3
    elif c["mode"] == "fuse4":
        p.mode, p.arity = vf.MODE_FUSE, 4
    return p


def _values(n, b, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if b <= 8:
        return torch.randint(0, 1 << b, (n,), dtype=torch.uint8, device=DEV, generator=g)
    if b <= 16:
        return torch.randint(0, 1 << b, (n,), dtype=torch.int32, device=DEV, generator=g).to(torch.uint16)
    if b <= 32:
        v = torch.randint(0, 1 << b, (n,), dtype=torch.int64, device=DEV, generator=g)
        return v.to(torch.uint32)
    return torch.randint(0, 1 << b, (n,), dtype=torch.int64, device=DEV, generator=g)


def _strings(n, seed):
    """Distinct byte strings of 8..64 bytes, packed, with their offsets."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    lens = torch.randint(8, 65, (n,), dtype=torch.int64, device=DEV, generator=g)
    offs = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=offs[1:])
    data = torch.randint(0, 256, (int(offs[-1]),), dtype=torch.uint8, device=DEV, generator=g)
    heads = synth.u64_keys_torch(0, n, seed).view(torch.uint8).view(n, 8)
    for j in range(8):  # the first eight bytes are the string's number, scrambled
        data[offs[:-1] + j] = heads[:, j]
    return data, offs


def _probes(keys, n, m, kind, seed):
    """What is asked: members in another order (a function), or as many keys
    outside the set as members, mixed (a filter)."""
    if kind == "func":
        if m == n:
            return keys, None
        g = torch.Generator(device=DEV)
        g.manual_seed(seed ^ 0x9E37)
        at = torch.randint(0, n, (m,), dtype=torch.int64, device=DEV, generator=g)
        return keys[at], at
    inside = m // 2
    outside = m - inside
    # odd places hold members
    q = torch.empty(m, dtype=torch.int64, device=DEV)
    q[0::2] = synth.u64_keys_torch(1 << 40, outside, seed)
    if inside <= n:
        q[1::2] = keys[:inside]
    else:
        at = torch.arange(inside, device=DEV) % n
        q[1::2] = keys[at]
    return q, None


def _sizes(c):
    """Uneven sizes, log-uniform between the case's two ends."""
    u = torch.rand(c["count"], generator=torch.Generator().manual_seed(c["n"]), dtype=torch.float64)
    lo, hi = math.log(c["n"]), math.log(c["m"])
    return [int(x) for x in torch.exp(lo + (hi - lo) * u)]


def prepare(case, seed):
    c = dict(case)
    op = c["op"]
    if op == "batch":
        items, outs, start = [], {8: 0, 16: 0, 32: 0}, 0
        for i, n in enumerate(_sizes(c)):
            b = [1, 8, 16, 32][i % 4]
            keys = synth.u64_keys_torch(start, n, seed)
            start += n
            items.append((keys, _values(n, b, seed + i), vf.FUNC, b, 1000 + seed + i))
            outs[max(b, 8)] += n
        types = {8: torch.uint8, 16: torch.uint16, 32: torch.uint32}
        # what vf_tune_batch settles on for such batches: elimination shards of 8192 keys for all
        opts = vf.vf_batch_opts_default(lge_threshold=(1 << 64) - 1, lge_target=8192)
        return {"op": op, "items": items, "opts": opts, "outs": {w: torch.empty(k, dtype=types[w], device=DEV) for w, k in outs.items()}}
    if op == "serve":
        # a dozen resident structures, half functions (b = 16), half filters (b = 8)
        sizes = _sizes(c)
        kept, reqs, total = [], [], {"func": 0, "filter": 0}
        for i in range(12):
            kind = "func" if i % 2 == 0 else "filter"
            n = 50_000 * (i + 1) + 3
            keys = synth.u64_keys_torch(i << 32, n, seed)
            b = 16 if kind == "func" else 8
            vals = _values(n, b, seed + i) if kind == "func" else None
            kept.append((vf.vf_build(keys, vals, params=_params(c, kind, b, seed + i)), keys, kind, n))
        for i, m in enumerate(sizes):
            s, keys, kind, n = kept[i % 12]
            q, _ = _probes(keys, n, m, kind, seed + i)
            reqs.append((s, q, kind, total[kind]))
            total[kind] += m
        outs = {"func": torch.empty(total["func"], dtype=torch.uint16, device=DEV),
                "filter": torch.empty(total["filter"], dtype=torch.uint8, device=DEV)}
        return {"op": op, "kept": kept, "outs": outs,
                "reqs": [(s, q, outs[kind][at:at + len(q)]) for s, q, kind, at in reqs]}
    n, b, kind = c["n"], c["b"], c["kind"]
    offs = None
    if c["keys"] == "bytes":
        keys, offs = _strings(n, seed)
        q = keys
    else:
        keys = synth.u64_keys_torch(0, n, seed)
        q, _ = _probes(keys, n, c["m"], kind, seed)
    vals = _values(n, b, seed) if kind == "func" else None
    p = _params(c, kind, b, seed)
    if op == "build":
        return {"op": op, "keys": keys, "offs": offs, "vals": vals, "params": p, "q": q}
    s = vf.vf_build(keys, vals, offsets=offs, params=p)
    if op == "host":
        q = q.cpu().pin_memory()
        out = torch.empty(c["m"], dtype=vals.dtype).pin_memory()
        return {"op": op, "s": s, "q": q, "out": out}
    return {"op": op, "s": s, "q": q, "offs": offs}


def _plain(x):
    """16- and 32-bit answers under the signed types, which torch indexes."""
    signed = {torch.uint16: torch.int16, torch.uint32: torch.int32}.get(x.dtype)
    return x if signed is None else x.view(signed)


def run(state):
    op = state["op"]
    if op == "query":
        return _plain(state["s"].query(state["q"], offsets=state["offs"]))
    if op == "host":
        return _plain(vf.vf_query(state["s"], state["q"], out=state["out"]))
    if op == "serve":
        vf.vf_query_batch(state["reqs"])
        return {k: _plain(x) for k, x in state["outs"].items()}
    if op == "batch":
        structs = vf.vf_build_batch(state["items"], opts=state["opts"])
        at, reqs = {8: 0, 16: 0, 32: 0}, []
        for s, (keys, _, _, b, _) in zip(structs, state["items"]):
            w = max(b, 8)
            reqs.append((s, keys, state["outs"][w][at[w]:at[w] + len(keys)]))
            at[w] += len(keys)
        vf.vf_query_batch(reqs)
        for s in structs:
            s.free()
        return {w: _plain(x) for w, x in state["outs"].items()}
    s = vf.vf_build(state["keys"], state["vals"], offsets=state["offs"], params=state["params"])
    out = s.query(state["q"], offsets=state["offs"])
    info = s.info
    s.free()
    return {"answers": _plain(out), "M": info.M, "cells": info.cells, "n_eff": info.n_eff, "seed": info.seed}


def work(case):
    """Keys (and values) read once, cells and answers written or read once."""
    c = dict(case)
    if c["op"] in ("batch", "serve"):
        k = sum(_sizes(c))
        if c["op"] == "serve":
            return {"bytes": k * (8 + 1.5) + 3_900_000 * 1.13 * 1.5, "flops": 0}
        return {"bytes": k * (2 * 8 + 3 * 2.0), "flops": 0}
    kb = 36 + 8 if c["keys"] == "bytes" else 8
    vb = 1 if c["kind"] == "filter" or c["b"] <= 8 else 2 if c["b"] <= 16 else 4 if c["b"] <= 32 else 8
    cells = c["n"] * 1.11 * c["b"] / 8
    asked = c["m"] * (kb + vb) + min(cells, 3.0 * c["m"] * max(1.0, c["b"] / 8))
    if c["op"] != "build":
        return {"bytes": asked, "flops": 0}
    return {"bytes": c["n"] * (kb + (0 if c["kind"] == "filter" else vb)) + cells + asked, "flops": 0}


def exact(case, seed):
    """What a function returns for its members is what it was given."""
    c = dict(case)
    if c["op"] in ("query", "host") and c["kind"] == "func":
        v = _plain(_values(c["n"], c["b"], seed))
        if c["keys"] == "bytes" or c["m"] == c["n"]:
            return v
        g = torch.Generator(device=DEV)
        g.manual_seed(seed ^ 0x9E37)
        return v[torch.randint(0, c["n"], (c["m"],), dtype=torch.int64, device=DEV, generator=g)]
    if c["op"] == "build" and c["kind"] == "func":
        return {"answers": _plain(_values(c["n"], c["b"], seed)), "M": None, "cells": None, "n_eff": None,
                "seed": None}
    if c["op"] == "batch":
        outs = {8: [], 16: [], 32: []}
        for i, n in enumerate(_sizes(c)):
            b = [1, 8, 16, 32][i % 4]
            outs[max(b, 8)].append(_plain(_values(n, b, seed + i)))
        return {w: torch.cat(x) for w, x in outs.items()}
    return None
