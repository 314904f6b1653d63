"""Performance cases of the library: what its users run, over the sizes they run it at.

A case is a dict of plain values.  ``prepare(case, seed)`` makes what a program
holds before the call (inputs drawn from the seed, and the workspace and output
buffers it keeps from call to call), ``run(state)`` is one pass through the
public entry points, and ``work(case)`` counts the bytes that pass cannot do
without: every input read once, every output written once.  All results are
whole numbers, fixed bit for bit by the inputs.

Kinds:
  mphf     a minimal perfect hash function built from keys, the call that
           decides on the host (``mphf_build``) or the device-driven one
           (``mphf_build_async``)
  peel     the peeling order of a hypergraph whose edges are in device memory
           (``peel``; ``general``: vertices anywhere)
  hashpeel the same from keys: ``hash_edges`` and then ``peel``
  batched  many bucket hypergraphs in one launch (``peel_batched``)
  lookup   queries of a built function (``mphf_lookup``)
  sf       a static function built from keys and values, then read back for
           all its keys (``sf_build``, ``sf_lookup``)
  large    the build with 64-bit ids (``mphf_build_large``)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1312_0526_gb300 as hp
from paper_1312_0526_gb300 import autotune, inputs


def listed():
    return [
        # the smallest request of the serving workload (key sets of 1e3 to
        # 1e7): launches and latency are all there is
        {"name": "mphf 1e3", "kind": "mphf", "n": 1009, "gamma": 1230, "form": "sync"},
        # the plain peel at the size a program starts with: keys hashed into
        # edges, peeled, order and claims returned
        {"name": "hash+peel 1e5", "kind": "hashpeel", "n": 100_000, "gamma": 1230, "r": 3},
        # the middle of the serving range, without a host round trip
        {"name": "mphf async 1e6", "kind": "mphf", "n": 1_000_003, "gamma": 1230,
         "form": "async"},
        # close above the threshold of 1.2218 a peel takes hundreds of rounds,
        # most of them small
        {"name": "peel near threshold 1e7", "kind": "peel", "n": 10_000_019, "gamma": 1222,
         "r": 3, "general": False},
        # a static function with values that straddle words (10 bits), built
        # and read back
        {"name": "sf 1e7 sigma 1000", "kind": "sf", "n": 10_000_019, "gamma": 1230,
         "sigma": 1000},
        # a general (not r-partite) hypergraph
        {"name": "general peel 2e7", "kind": "peel", "n": 20_000_003, "gamma": 1230, "r": 3,
         "general": True},
        # r = 4
        {"name": "peel r4 1e8", "kind": "peel", "n": 100_000_000, "gamma": 1300, "r": 4,
         "general": False},
        # the large MPHF build that fits 32-bit ids comfortably
        {"name": "mphf 1e8", "kind": "mphf", "n": 100_000_007, "gamma": 1230, "form": "sync"},
        # and its queries: every key of the set once
        {"name": "lookup 1e8", "kind": "lookup", "n": 100_000_007, "nq": 100_000_007,
         "gamma": 1230},
        # 65,536 buckets of lognormal sizes (64 to 65,536 keys), with g values
        {"name": "batched 65536", "kind": "batched", "B": 65_536, "median": 2000,
         "gamma": 1230, "with_g": True},
        # the headline: one huge plain peel, all arrays far larger than L2
        {"name": "peel 8e8", "kind": "peel", "n": 800_000_011, "gamma": 1230, "r": 3,
         "general": False},
        # 64-bit ids, for key sets past 2^32; at a size that runs within a second
        {"name": "large mphf 1e9", "kind": "large", "n": 1_000_000_007, "gamma": 1230},
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi], odd as often as even."""
    return int(round(10.0 ** rng.uniform(math.log10(lo), math.log10(hi))))


def draw(rng):
    kind = rng.choice(["mphf", "mphf", "peel", "peel", "hashpeel", "batched", "lookup", "sf",
                       "large"])
    if kind == "mphf":
        return {"kind": kind, "n": _size(rng, 1e3, 1e8),
                "gamma": rng.choice([1230, 1230, 1250, 1300]),
                "form": rng.choice(["sync", "async"])}
    if kind in ("peel", "hashpeel"):
        r = rng.choice([3, 3, 3, 4])
        gamma = rng.choice([1230, 1230, 1222, 1200]) if r == 3 else 1300
        if kind == "hashpeel":
            return {"kind": kind, "n": _size(rng, 1e3, 1e8), "gamma": gamma, "r": r}
        general = rng.random() < 0.3
        return {"kind": kind, "n": _size(rng, 1e4, 1e8 if general or r == 4 else 8e8),
                "gamma": gamma, "r": r, "general": general}
    if kind == "batched":
        return {"kind": kind, "B": _size(rng, 256, 65_536), "median": _size(rng, 200, 2000),
                "gamma": 1230, "with_g": rng.random() < 0.5}
    if kind == "lookup":
        return {"kind": kind, "n": _size(rng, 1e3, 1e8), "nq": _size(rng, 1e3, 1e8),
                "gamma": 1230}
    if kind == "sf":
        return {"kind": kind, "n": _size(rng, 1e3, 1e8), "gamma": 1230,
                "sigma": rng.choice([2, 3, 256, 1000, 65_536, 1 << 32])}
    return {"kind": kind, "n": _size(rng, 1e6, 1e9), "gamma": 1230}


def _bytes(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device="cuda")


def _words(n):
    return torch.empty(max(int(n), 1), dtype=torch.int64, device="cuda")


def _ids(n):
    return torch.empty(int(n), dtype=torch.int32, device="cuda")


def _sizes(case):
    """Bucket sizes of a batched case (of the shape alone, the keys vary)."""
    return inputs.lognormal_bucket_sizes(case["B"], median=case["median"], seed=3)


MAX_LAYERS = 4096


def prepare(case, seed):
    kind, gamma = case["kind"], case["gamma"]
    # streams of different seeds share no part: SplitMix64 states far apart
    stream = (seed + 1) * 0x5851F42D4C957F2D % (1 << 63)
    s = {"case": case}
    if kind == "batched":
        off = np.zeros(case["B"] + 1, dtype=np.int64)
        off[1:] = np.cumsum(_sizes(case))
        s["off"] = torch.from_numpy(off).cuda()
        s["keys"] = inputs.keys_torch(int(off[-1]), stream)
        # the launch shape a program picks once for its workload (cached on disk)
        s["tuning"] = autotune.tune(s["keys"], s["off"], gamma, with_g=case["with_g"])
        s["ws"] = _bytes(hp.batched_workspace_size(case["B"], gamma, s["tuning"]))
        s["out"] = hp.BatchedResult(_ids(off[-1]), _ids(case["B"]), _ids(case["B"]), None, None)
        if case["with_g"]:
            s["out"].G_off = hp.batched_g_offsets(s["off"], gamma, s["ws"])
            s["out"].G = _words(int(s["out"].G_off[-1].item()))
        return s
    n = case["n"]
    r = case.get("r", 3)
    m = s["m"] = hp.num_vertices(n, gamma, r)
    keys = inputs.keys_torch(n, stream)
    if kind in ("peel", "hashpeel"):
        general = case.get("general", False)
        s["edges"] = torch.empty((n, r), dtype=torch.int32, device="cuda")
        if kind == "peel":
            hp.hash_edges(keys, m, r, seed=1, out=s["edges"], general=general)
        else:
            s["keys"] = keys
        s["ws"] = _bytes(hp.peel_workspace_size(n, m, r, general))
        s["out"] = (_ids(n), _ids(n), _words(MAX_LAYERS + 1).zero_())
        return s
    s["keys"] = keys
    if kind == "sf":
        g = torch.Generator(device="cuda").manual_seed(seed)
        v = torch.randint(0, case["sigma"], (n,), generator=g, device="cuda", dtype=torch.int64)
        s["values"] = v.to(torch.int32)  # the uint32 value, bit for bit
        s["ws"] = _bytes(hp.sf_workspace_size(n, gamma))
        s["U"] = _words((m * hp.sf_bits(case["sigma"]) + 63) // 64)
        s["got"] = _ids(n)
        return s
    s["G"] = _words((m + 31) // 32)
    s["D"] = _words((m + 511) // 512 + 1)
    if kind == "large":
        s["ws"] = _bytes(hp.mphf_large_workspace_size(n, gamma))
        return s
    s["ws"] = _bytes(hp.mphf_workspace_size(n, gamma))
    if kind == "lookup":
        built = hp.mphf_build(keys, 1, gamma, workspace=s.pop("ws"), G=s["G"], rank_dir=s["D"])
        s["seed"] = built.stats["seed_used"]
        # the queries: keys of the set in another order, as often as it takes
        g = torch.Generator(device="cuda").manual_seed(seed)
        nq = case["nq"]
        s["keys"] = keys[torch.randint(0, n, (nq,), generator=g, device="cuda")]
        s["got"] = _ids(nq)
        return s
    s["stats"] = torch.zeros(128, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "mphf":
        if case["form"] == "async":
            G, D, _ = hp.mphf_build_async(s["keys"], 1, case["gamma"], workspace=s["ws"], G=s["G"],
                                          rank_dir=s["D"], stats=s["stats"])
            return {"G": G, "rank_dir": D}
        b = hp.mphf_build(s["keys"], 1, case["gamma"], workspace=s["ws"], G=s["G"],
                          rank_dir=s["D"])
        return {"G": b.G, "rank_dir": b.rank_dir, "seed": b.stats["seed_used"],
                "rounds": b.stats["rounds"]}
    if kind in ("peel", "hashpeel"):
        if kind == "hashpeel":
            hp.hash_edges(s["keys"], s["m"], case["r"], seed=1, out=s["edges"])
        p = hp.peel(s["edges"], s["m"], workspace=s["ws"], max_layers=MAX_LAYERS,
                    general=case.get("general", False), out=s["out"])
        # the whole layer table: p.layer_off is its first rounds + 1 entries
        return {"order": p.order, "claim": p.claim, "layer_off": s["out"][2],
                "rounds": p.rounds, "n_peeled": p.n_peeled}
    if kind == "batched":
        b = hp.peel_batched(s["keys"], s["off"], case["gamma"], with_g=case["with_g"],
                            tuning=s["tuning"], workspace=s["ws"], out=s["out"])
        got = {"order": b.order, "rounds": b.rounds, "status": b.status}
        if case["with_g"]:
            got["G"] = b.G
        return got
    if kind == "lookup":
        return hp.mphf_lookup(s["keys"], s["seed"], s["m"], s["G"], s["D"], out=s["got"])
    if kind == "sf":
        b = hp.sf_build(s["keys"], s["values"], case["sigma"], 1, case["gamma"],
                        workspace=s["ws"], U=s["U"])
        got = hp.sf_lookup(s["keys"], b.stats["seed_used"], s["m"], case["sigma"], b.U,
                           out=s["got"])
        return {"U": b.U, "values": got}
    b = hp.mphf_build_large(s["keys"], 1, case["gamma"], workspace=s["ws"], G=s["G"],
                            rank_dir=s["D"])
    return {"G": b.G, "rank_dir": b.rank_dir, "seed": b.stats["seed_used"],
            "rounds": b.stats["rounds"]}


def work(case):
    kind = case["kind"]
    if kind == "batched":
        sizes = _sizes(case)
        n, m = int(sizes.sum()), 1.23 * int(sizes.sum())
        b = 8 * n + 8 * case["B"] + 4 * n + 8 * case["B"] + (m / 4 if case["with_g"] else 0)
        return {"bytes": b, "flops": 0}
    n = case["n"]
    r = case.get("r", 3)
    m = hp.num_vertices(n, case["gamma"], r)
    function = m / 4 + m / 64  # g values and rank directory
    if kind == "peel":  # edges in, order and claim words out
        b = 4 * r * n + 8 * n
    elif kind == "hashpeel":  # keys in, edges, order and claim words out
        b = 8 * n + 4 * r * n + 8 * n
    elif kind == "lookup":
        b = 12 * case["nq"] + min(function, case["nq"] * 128.0)
    elif kind == "sf":  # keys and values in, the function out; keys in, values out
        b = 12 * n + m * hp.sf_bits(case["sigma"]) / 8 + 12 * n
    else:  # mphf, large
        b = 8 * n + function
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """All outputs are whole numbers, compared bit for bit."""
    return None
