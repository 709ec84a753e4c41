"""Performance cases: what programs that use this library have it do.

Every case goes through the public Python binding (``burr.build``, ``Handle.query``,
``Handle.export``, ``burr.build_batch``, ``burr.Server``), the call path of a user's program.
Sizes, value widths and options are those of the repository's benchmark and tests
(2^20, 10^7, 10^8 and 10^9 keys, batches and request streams of log-uniform sizes, r from 1 to 32,
2-bit and 1+-bit thresholds, cut search), with odd sizes among them.

Outputs are bit patterns (exports) or table values, so two implementations agree exactly or not at
all.  Stored values of member keys are known independently of the library; ``exact`` gives those.

  build   keys and values on the device (or in page-locked host memory) -> structure -> its export
          in a page-locked host buffer that the program keeps
  query   a resident structure, a batch of keys on the device (half of them members) -> values
  batch   many independent structures built in one call, each then queried once
  serve   a burst of build requests and one query batch for each, from host memory, through the
          build/query server
"""
import math

import numpy as np
import torch

from paper_2411_12365_gb300 import burr
from paper_2411_12365_gb300 import inputs as I

BUILD = dict(kind="build", thresholds="2bit", cut_search="none", host=False)
QUERY = dict(kind="query", thresholds="2bit")


def listed():
    return [
        # one small filter, e.g. a shard's delta or a per-tenant set: launches and latency
        dict(BUILD, name="build_1k", n=1_003, r=8),
        # a small retrieval table with an odd value width
        dict(BUILD, name="build_50k_r3", n=50_021, r=3),
        # the repository's smallest benchmark configuration
        dict(BUILD, name="build_1m", n=1 << 20, r=8),
        # 16-bit fingerprints with the space-saving options (1+-bit thresholds, searched cuts)
        dict(BUILD, name="build_10m_r16_1plus", n=10_000_019, r=16, thresholds="1plus", cut_search="diff"),
        # end to end from page-locked host memory
        dict(BUILD, name="build_30m_host", n=30_000_001, r=8, host=True),
        # the 10^8-key configuration
        dict(BUILD, name="build_100m", n=100_000_000, r=8),
        # the largest single structure, the benchmark's default step
        dict(BUILD, name="build_1b", n=1_000_000_000, r=8),
        # many independent structures, sizes log-uniform, mixed value widths
        dict(kind="batch", name="batch_300", count=300, lo=100, hi=1_000_000, thresholds="2bit"),
        # requests of a lookup service: a small key batch on a resident structure
        dict(QUERY, name="query_10k_r3", n=1_000_003, nq=10_007, r=3),
        # 16-bit values, 1+-bit thresholds, a mid-sized batch
        dict(QUERY, name="query_5m_r16_1plus", n=10_000_019, nq=5_000_011, r=16, thresholds="1plus"),
        # bulk probing: 10^8 positive and negative keys against 10^8 stored ones
        dict(QUERY, name="query_100m", n=100_000_000, nq=100_000_000, r=8),
        # a burst of requests to the build/query server
        dict(kind="serve", name="serve_48", count=48, lo=1_000, hi=1_000_000, r=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "query", "query", "batch", "serve"])
    r = rng.choice([1, 2, 3, 4, 5, 7, 8, 8, 8, 12, 16, 16, 24, 32])
    thresholds = rng.choice(["2bit", "2bit", "2bit", "1plus"])
    if kind == "build":
        cut = rng.choice(["none", "none", "none", "minbump", "maxprev", "diff"])
        host = rng.random() < 0.25
        return dict(kind=kind, n=_log(rng, 500, 50_000_000 if host else 300_000_000), r=r, thresholds=thresholds,
                    cut_search=cut, host=host)
    if kind == "query":
        return dict(kind=kind, n=_log(rng, 1_000, 100_000_000), nq=_log(rng, 1_000, 100_000_000), r=r,
                    thresholds=thresholds)
    if kind == "batch":
        count = _log(rng, 20, 1_000)
        return dict(kind=kind, count=count, lo=_log(rng, 100, 1_000), hi=_log(rng, 10_000, 1_000_000),
                    thresholds=thresholds)
    return dict(kind=kind, count=rng.randint(8, 60), lo=1_000, hi=_log(rng, 10_000, 1_000_000), r=rng.choice([4, 8, 16]))


_CUT = dict(none=burr.CUT_NONE, minbump=burr.CUT_MINBUMP, maxprev=burr.CUT_MAXPREV, diff=burr.CUT_DIFF)
_MODE = {"2bit": burr.THRESH_2BIT, "1plus": burr.THRESH_1PLUS}


def _seed(seed, salt=0):
    """Counter base of a run's keys: runs of different seeds use disjoint counters."""
    return (I.KEY_SEED + ((int(seed) * 64 + salt) << 34)) & ((1 << 64) - 1)


def _sizes(case, seed):
    """Sizes log-uniform in [lo, hi].  They are the case's, not the seed's: the same amount of work
    for every seed."""
    g = np.random.default_rng(2024 + case["count"])
    return np.exp(g.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"])).astype(np.int64)


def _params(case):
    return burr.default_params(threshold_mode=_MODE[case.get("thresholds", "2bit")],
                               cut_search=_CUT[case.get("cut_search", "none")])


def _export_bound(n, r):
    """Bytes that hold any export of n keys (tables, thresholds, headers)."""
    return int(1.08 * n * r / 8) + n // 8 + 4096 * (r + 1)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "build":
        n, r = case["n"], case["r"]
        keys = I.keys_torch(n, "cuda", seed=_seed(seed))
        vals = I.values_torch(keys, r)
        if case["host"]:
            st["keys"] = torch.empty(n, dtype=keys.dtype, pin_memory=True).copy_(keys)
            st["vals"] = torch.empty(n, dtype=vals.dtype, pin_memory=True).copy_(vals)
        else:
            st["keys"], st["vals"] = keys, vals
        st.update(r=r, params=_params(case), out=torch.zeros(_export_bound(n, r), dtype=torch.uint8, pin_memory=True))
    elif kind == "query":
        n, nq, r = case["n"], case["nq"], case["r"]
        keys = I.keys_torch(n, "cuda", seed=_seed(seed))
        st["h"] = burr.build(keys, I.values_torch(keys, r), r, params=_params(case))
        half = nq // 2
        pick = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(int(seed)))[:half] \
            if half < n else torch.arange(half, device="cuda") % n
        others = I.keys_torch(nq - half, "cuda", seed=_seed(seed), offset=1 << 32)
        st.update(half=half, keys=torch.cat([keys[pick], others]),
                  out=torch.empty(nq, dtype=burr.value_torch_dtype(r), device="cuda"))
    elif kind == "batch":
        n = _sizes(case, seed)
        offs = np.concatenate([[0], np.cumsum(n)])
        rs = np.random.default_rng(7 + case["count"]).choice([1, 2, 3, 4, 8], case["count"]).tolist()
        keys = I.keys_torch(int(offs[-1]), "cuda", seed=_seed(seed))
        vals = I.values_torch(keys, 8)
        for s, r in enumerate(rs):
            vals[offs[s]:offs[s + 1]] &= (1 << r) - 1
        # each structure's query batch: its first half of members, then as many other keys
        others = I.keys_torch(int(offs[-1]), "cuda", seed=_seed(seed), offset=1 << 32)
        q, cut = [], []
        for a, b in zip(offs[:-1], offs[1:]):
            h = int(b - a + 1) // 2
            q += [keys[a:a + h], others[a:a + int(b - a) - h]]
            cut.append(h)
        st.update(keys=keys, vals=vals, offs=offs, rs=rs, params=_params(case), queries=torch.cat(q),
                  out=torch.empty(int(offs[-1]), dtype=torch.uint8, device="cuda"), cut=cut)
    else:
        n, r = _sizes(case, seed), case["r"]
        g = np.random.default_rng(99 + case["count"])
        nq = np.exp(g.uniform(math.log(1_000), math.log(100_000), case["count"])).astype(np.int64)
        reqs = []
        for s in range(case["count"]):
            k = I.keys_np(int(n[s]), seed=_seed(seed, s))
            half = int(min(nq[s] // 2, n[s]))
            others = I.keys_np(int(nq[s]) - half, seed=_seed(seed, s), offset=1 << 32)
            reqs.append((k, I.values_np(k, r), np.concatenate([k[:half], others])))
        st.update(r=r, reqs=reqs, server=burr.Server(40 << 30, host_staging_bytes=256 << 20))
    return st


def run(st):
    kind = st["kind"]
    if kind == "build":
        h = burr.build(st["keys"], st["vals"], st["r"], params=st["params"])
        return {"bytes": h.export(out=st["out"]), "export": st["out"]}   # zeros past the export's end
    if kind == "query":
        out = st["h"].query(st["keys"], out=st["out"])
        return {"members": out[:st["half"]], "others": out[st["half"]:]}
    if kind == "batch":
        hs = burr.build_batch(st["keys"], st["vals"], st["offs"], st["rs"], params=st["params"])
        q, out, offs = st["queries"], st["out"], st["offs"]
        for s, h in enumerate(hs):
            h.query(q[offs[s]:offs[s + 1]], out=out[offs[s]:offs[s + 1]])
        burr.free_all(hs)
        return out
    srv, r = st["server"], st["r"]
    builds = [srv.submit_build(k, v, r) for k, v, _ in st["reqs"]]
    queries = [srv.submit_query(t, q) for t, (_, _, q) in zip(builds, st["reqs"])]
    for t in builds:
        srv.wait(t)
    outs = [srv.wait(t)[0] for t in queries]
    for t in builds:
        srv.release(t)
    return outs


def _table_bytes(n, r):
    """Table and thresholds of a structure of n keys (space overhead about 1%)."""
    return 1.01 * n * r / 8


def work(case):
    """Each key and value read once, each table, export or value written once; queries read a
    threshold sector and the table window of each key, at most the whole table."""
    kind = case["kind"]
    vb = lambda r: 1 if r <= 8 else (2 if r <= 16 else 4)   # noqa: E731
    if kind == "build":
        n, r = case["n"], case["r"]
        b = n * (8 + vb(r)) + _table_bytes(n, r)
    elif kind == "query":
        r = case["r"]
        b = case["nq"] * (8 + vb(r)) + min(_table_bytes(case["n"], r), case["nq"] * (32 + 16 * r))
    elif kind == "batch":
        n = float(_sizes(case, 0).sum())
        b = n * (8 + 1) * 2 + 2 * _table_bytes(n, 3.6)
    else:
        n = float(_sizes(case, 0).sum())
        b = n * (8 + vb(case["r"])) + _table_bytes(n, case["r"]) + case["count"] * 20_000 * 9
    return {"bytes": b, "flops": 0}


def _fmix64(x):
    """MurmurHash3's 64-bit finalizer, the generator of the stored values, in numpy."""
    with np.errstate(over="ignore"):
        for c in (0xFF51AFD7ED558CCD, 0xC4CEB9FE1A85EC53):
            x = (x ^ (x >> np.uint64(33))) * np.uint64(c)
        return x ^ (x >> np.uint64(33))


def exact(case, seed):
    """The stored values of the queried members; what other keys return is the method's choice."""
    if case["kind"] != "query" or case["nq"] > 20_000_000:
        return None
    n, half, r = case["n"], case["nq"] // 2, case["r"]
    pick = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(int(seed)))[:half] \
        if half < n else torch.arange(half, device="cuda") % n
    with np.errstate(over="ignore"):
        keys = _fmix64(pick.cpu().numpy().astype(np.uint64) + np.uint64(_seed(seed)))
    v = _fmix64(keys ^ np.uint64(I.VALUE_SEED)) & np.uint64((1 << r) - 1)
    kind = (np.uint8, np.int16, np.int32)[0 if r <= 8 else (1 if r <= 16 else 2)]
    return {"members": v.astype(np.uint32).astype(kind) if r > 8 else v.astype(np.uint8), "others": None}
