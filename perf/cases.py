"""The joins whose speed is looked after, from the smallest call to the largest, through the binding's public calls.

A case is a dict of plain values:
  call      "join" (hj_join), "probe" (hj_build once, then hj_probe of each S), "batch" (hj_join_batch) or
            "host" (hj_join_host: relations and pairs in page-locked host memory)
  nr, ns    tuples of R and of S (of a batch: the smallest and largest |R| of its joins, with |S| = 4 |R|)
  width     bytes of a key and of a rid: 4 or 8
  mode      "pairs" (every pair written), "count" or "checksum" (the count with two order-free checksums)
  keys      "dense": R's keys are a permutation of 1 .. |R|; "spread": the same scattered over the whole key domain;
            "heavy": a quarter or so of R's rows share one key; "zipf": R and S draw from the same Zipf ranks
  match     the share of S's rows that meet R (dense and spread keys)
  skew      the heavy key's share of R's rows, or the exponent of S's ranks (R's are drawn with 0.75)
  joins     the number of joins of a batch

A join's pairs come in no specified order (the library promises a multiset), and two runs of the same program give
two orders.  `run` therefore returns the library's buffer as it is, in a dict that puts the pairs in order only when
they are read out of it: no user's program sorts them, and the sort is no part of a pass.
Row numbers are the rids, as in the paper's data sets, and stay below 2^31.
"""
import math

import numpy as np
import torch

from paper_1307_1955_gb300 import hj

MODES = {"pairs": hj.HJ_MATERIALIZE, "count": hj.HJ_COUNT, "checksum": hj.HJ_COUNT_CHECKSUM}
DEV = "cuda"


def _case(name, call, nr, ns, width=4, mode="pairs", keys="dense", match=1.0, skew=0.0, joins=1):
    return {"name": name, "call": call, "nr": nr, "ns": ns, "width": width, "mode": mode, "keys": keys,
            "match": match, "skew": skew, "joins": joins}


def listed():
    return [
        # the smallest request that a server sees: latency, launches and host work
        _case("join_4k_10k", "join", 4097, 10007, match=0.5),
        # a small dimension table met by a large fact table: the table stays in L2
        _case("join_256k_16m", "join", 1 << 18, 1 << 24),
        # equal small sides: the build costs as much as the probe
        _case("join_1m_1m", "join", 1 << 20, 1 << 20),
        # the paper's default size, and its most skewed data set at that size
        _case("join_16m_16m", "join", 1 << 24, 1 << 24),
        _case("join_16m_heavy25", "join", 1 << 24, 1 << 24, keys="heavy", skew=0.25),
        # a large fact table, half of it matching: the headline workload, the largest case
        _case("join_16m_256m", "join", 1 << 24, 1 << 28, match=0.5),
        # 64-bit keys scattered over their domain, ragged sizes
        _case("join_3m_20m_u64", "join", 3000017, 20000003, width=8, keys="spread", match=0.5),
        # how many rows a join would give, before it is run: ragged sizes
        _case("count_6m_50m", "join", 6000011, 50000001, mode="count", match=0.75),
        # skewed 64-bit keys on both sides; 3e11 pairs are counted and checked, never written
        _case("checksum_zipf_4m_64m_u64", "join", 1 << 22, 1 << 26, width=8, mode="checksum", keys="zipf", skew=1.0),
        # a lookup table that a program keeps, met by one block of rows after another
        _case("probe_1m_6m_u64", "probe", 1000003, 6000001, width=8, keys="spread", match=0.75),
        # many independent joins of all sizes in one call, as a server's waves are
        _case("batch_200", "batch", 1 << 10, 1 << 20, match=0.75, joins=200),
        # relations in host memory: the host link and the device at once
        _case("host_5m_40m", "host", 5000011, 40000003, match=0.5),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["join", "u64", "count", "checksum", "heavy", "zipf", "probe", "batch", "host"],
                       [6, 2, 1, 1, 1, 1, 2, 1, 1])[0]
    match = rng.choice([0.125, 0.5, 0.75, 1.0])
    keys = rng.choice(["dense", "spread"])
    name = ""
    if kind == "batch":
        lo = _log_uniform(rng, 1 << 10, 1 << 13)
        hi = _log_uniform(rng, 1 << 16, 1 << 20)
        c = _case(name, "batch", lo, hi, match=match, keys=keys, joins=rng.randint(16, 256))
    elif kind == "heavy":
        n = _log_uniform(rng, 1 << 20, 1 << 24)
        c = _case(name, "join", n, _log_uniform(rng, n, min(4 * n, 1 << 25)), keys="heavy",
                  skew=rng.choice([0.1, 0.25]))
    elif kind == "zipf":
        n = _log_uniform(rng, 1 << 18, 1 << 22)
        c = _case(name, "join", n, _log_uniform(rng, n, 16 * n), width=8, mode="checksum", keys="zipf",
                  skew=round(rng.uniform(0.5, 1.0), 3))
    elif kind == "host":
        n = _log_uniform(rng, 1 << 16, 1 << 22)
        c = _case(name, "host", n, _log_uniform(rng, n, 1 << 25), match=match, keys=keys)
    elif kind == "probe":
        n = _log_uniform(rng, 1 << 12, 1 << 21)
        c = _case(name, "probe", n, _log_uniform(rng, n, 1 << 23), width=rng.choice([4, 8]), match=match, keys=keys)
    else:
        nr = _log_uniform(rng, 1 << 10, 1 << 24)
        width = 8 if kind == "u64" else rng.choice([4, 4, 8]) if kind in ("count", "checksum") else 4
        ns = _log_uniform(rng, nr, min(256 * nr, (1 << 27) if width == 4 else 1 << 26))
        c = _case(name, "join", nr, ns, width=width, mode="pairs" if kind in ("join", "u64") else kind, match=match,
                  keys=keys)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------------- inputs

_SPREAD = {4: 0x9E3779B1, 8: 0x9E3779B97F4A7C15}  # odd: a multiple of it is another key for each row number


def _signed(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _relation(keys, width, spread):
    if spread:
        keys = keys * _signed(_SPREAD[width])
    if width == 4:
        keys = keys.to(torch.int32)  # (the low 32 bits)
    rids = torch.arange(len(keys), dtype=keys.dtype, device=keys.device)
    return torch.stack([keys, rids], dim=1)


def _zipf(n, ranks, theta, g):
    cdf = torch.arange(1, ranks + 1, dtype=torch.float64, device=DEV).pow(-theta).cumsum(0)
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g) * cdf[-1]
    return torch.searchsorted(cdf, u).clamp_(max=ranks - 1) + 1


def _one(case, nr, ns, g):
    """R and S on the device, as (n, 2) tensors of key and rid."""
    width, keys = case["width"], case["keys"]
    if keys == "zipf":
        ranks = max(1, nr // 4)
        rk, sk = _zipf(nr, ranks, 0.75, g), _zipf(ns, ranks, case["skew"], g)
        return _relation(rk, width, True), _relation(sk, width, True)
    perm = torch.randperm(nr, device=DEV, generator=g)
    if keys == "heavy":
        # key 1 for nh rows of R, keys 2 .. nr - nh + 1 for the others; S meets every key of R equally often, and
        # the heavy one exactly so (its pairs are most of the output)
        nh = int(round(case["skew"] * nr))
        nd = nr - nh
        rk = torch.where(perm < nh, 1, perm - nh + 2)
        hs = max(1, round(ns / (nd + 1)))
        sk = torch.randint(2, nd + 2, (ns,), device=DEV, generator=g)
        sk[:hs] = 1
        sk = sk[torch.randperm(ns, device=DEV, generator=g)]
        return _relation(rk, width, False), _relation(sk, width, False)
    rk = perm + 1
    sk = torch.randint(1, nr + 1, (ns,), device=DEV, generator=g)
    if case["mode"] == "pairs":  # the share exactly: outputs of one shape whatever the seed
        hit = _hits(case, ns)
        if hit < ns:
            sk[hit:] += nr
            sk = sk[torch.randperm(ns, device=DEV, generator=g)]
    else:
        sk += nr * (torch.rand(ns, device=DEV, generator=g) >= case["match"])
    return _relation(rk, width, keys == "spread"), _relation(sk, width, keys == "spread")


def _hits(case, ns):
    return int(round(case["match"] * ns))


def _sizes(case):
    """(|R|, |S|) of every join of the case: of a batch, |R| evenly over the logarithm of its range, in a mixed order."""
    if case["call"] != "batch":
        return [(case["nr"], case["ns"])]
    n, lo, hi = case["joins"], math.log(case["nr"]), math.log(case["ns"])
    nr = [int(math.exp(lo + (hi - lo) * ((i * 0.6180339887498949) % 1.0))) for i in range(n)]
    return [(x, 4 * x) for x in nr]


def _inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return [_one(case, nr, ns, g) for nr, ns in _sizes(case)]


# --------------------------------------------------------------------------------------------------------- calls

_context = None


def _ctx():
    """The context that a program makes once, on torch's current stream."""
    global _context
    if _context is None:
        _context = hj.hj_create()
    return _context


class State:
    def __init__(self, case, seed):
        self.call, self.mode, self.width, self.ctx = case["call"], MODES[case["mode"]], case["width"], _ctx()
        pairs = _inputs(case, seed)
        self.R, self.S = pairs[0]
        self.table = None
        if self.call == "probe":
            self.table = hj.hj_build(self.ctx, self.R, mode=self.mode)
        elif self.call == "batch":
            self.keep = pairs
            self.Rs = hj.rel_array([r for r, _ in pairs])
            self.Ss = hj.rel_array([s for _, s in pairs])
        elif self.call == "host":
            self.R, self.S = self.R.cpu().pin_memory(), self.S.cpu().pin_memory()
            self.out = torch.empty((_hits(case, case["ns"]), 2), dtype=self.R.dtype, pin_memory=True)

    def __del__(self):
        if self.table is not None:
            self.table.free()


def prepare(case, seed):
    return State(case, seed)


class _Buffer:
    """n values of the library's device memory, for torch to look at."""

    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i8", "data": (ptr, False), "version": 2}


def _in_order(words, width):
    """Pairs (one 8-byte word each, or two) sorted by S's row and R's row."""
    if width == 4:
        return torch.sort(words).values.view(torch.int32).view(-1, 2)
    key = torch.sort((words[1::2] << 32) | words[0::2]).values
    return torch.stack([key & 0xFFFFFFFF, key >> 32], dim=1)


class Output(dict):
    """The library's results: counts at once, pairs in order when they are read (see the top)."""

    def __init__(self, fields, read, free):
        super().__init__(fields)
        self["pairs"] = None
        self._read, self._free = read, free

    def __getitem__(self, key):
        return self._read() if key == "pairs" else super().__getitem__(key)

    def __iter__(self):
        return iter(self.keys())

    def items(self):
        return [(k, self[k]) for k in self.keys()]

    def values(self):
        return [self[k] for k in self.keys()]

    def __del__(self):
        self._free()


def _device_pairs(ptr, count, width):
    if not count:
        return torch.zeros((0, 2), dtype=torch.int32 if width == 4 else torch.int64, device=DEV)
    return _in_order(torch.as_tensor(_Buffer(ptr, count * width // 4), device=DEV), width)


def run(state):
    s = state
    if s.call == "batch":
        outs = hj.hj_join_batch(s.ctx, s.Rs, s.Ss, mode=s.mode, graph=True, raw=True)
        return Output({"count": np.array([o.count for o in outs], np.int64)},
                      lambda: torch.cat([_device_pairs(o.pairs, o.count, s.width) for o in outs]),
                      lambda: hj.hj_results_free(s.ctx, outs))
    if s.call == "host":
        r = hj.hj_join_host(s.ctx, s.R, s.S, pairs_out=s.out)
        return Output({"count": r.count}, lambda: _in_order(s.out[:r.count].to(DEV).view(torch.int64).view(-1), s.width),
                      lambda: None)
    if s.call == "probe":
        r = hj.hj_probe(s.ctx, s.table, s.S, mode=s.mode)
    else:
        r = hj.hj_join(s.ctx, s.R, s.S, mode=s.mode)
    if s.mode == hj.HJ_MATERIALIZE:
        return Output({"count": r.count}, lambda: _device_pairs(r.pairs_ptr, r.count, s.width), r.free)
    out = {"count": r.count}
    if s.mode == hj.HJ_COUNT_CHECKSUM:
        out["c0"], out["c1"] = (_signed(c) for c in r.checksum)
    r.free()
    return out


# ---------------------------------------------------------------------------------------------------- accounting


def _pairs_of(case, nr, ns):
    if case["mode"] != "pairs":
        return 0
    if case["keys"] == "heavy":
        nh = int(round(case["skew"] * nr))
        hs = max(1, round(ns / (nr - nh + 1)))
        return ns - hs + hs * nh
    return _hits(case, ns)


def work(case):
    """Every tuple of both sides read once (of a kept table: once, as the build's tuples), every pair written once."""
    b = sum((nr + ns + _pairs_of(case, nr, ns)) * 2 * case["width"] for nr, ns in _sizes(case))
    return {"bytes": b, "flops": 0}


def tolerance(case):
    # whole numbers: every pair, count and checksum is the same
    return "exact"


def _mixed(x):
    """The finaliser of the checksums (the SplitMix64 one) on 64-bit patterns."""
    def srl(v, s):
        return (v >> s) & ((1 << (64 - s)) - 1)
    x = (x ^ srl(x, 30)) * _signed(0xBF58476D1CE4E5B9)
    x = (x ^ srl(x, 27)) * _signed(0x94D049BB133111EB)
    return x ^ srl(x, 31)


def exact(case, seed):
    """The join by its definition: R sorted by key, each key of S looked up in it."""
    counts, pairs = [], []
    for R, S in _inputs(case, seed):
        rk, order = torch.sort(R[:, 0])
        lo = torch.searchsorted(rk, S[:, 0].contiguous())
        n = torch.searchsorted(rk, S[:, 0].contiguous(), right=True) - lo
        counts.append(int(n.sum()))
        if case["mode"] == "pairs":
            at = torch.arange(counts[-1], device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n)
            r = R[order[torch.repeat_interleave(lo, n) + at], 1].long()
            s = torch.repeat_interleave(S[:, 1].long(), n)
            key = torch.sort((s << 32) | r).values
            pairs.append(torch.stack([key & 0xFFFFFFFF, key >> 32], dim=1).to(R.dtype))
        elif case["mode"] == "checksum":
            unsigned = 0xFFFFFFFF if case["width"] == 4 else -1
            a = _mixed(R[order, 1].long() & unsigned).cumsum(0)
            a = torch.cat([a.new_zeros(1), a])
            a = a[lo + n] - a[lo]  # of R's rows with the S row's key (modulo 2^64, as everything here)
            b = _mixed((S[:, 1].long() & unsigned) ^ _signed(0x9E3779B97F4A7C15))
            return {"count": counts[0], "c0": int((a * b).sum()), "c1": int((a + n * b).sum())}
    if case["mode"] == "count":
        return {"count": counts[0]}
    if case["call"] == "batch":
        return {"count": np.array(counts, np.int64), "pairs": torch.cat(pairs)}
    return {"count": counts[0], "pairs": pairs[0]}
