"""hj_join of a build side that fits shared memory whole (SHJ, pairs): every CTA builds
its own table and probes a share of S.  Against the CPU oracle, at the edges of the
build sizes, odd probe sizes and shares of one group; keys of all ones (the marker of
empty slots, kept in a list of 64), repeated keys up to the key-list fallback, and a pair
buffer that is too small.  Integer results: every comparison is exact."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def hjm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_1955_gb300 import hj

    return hj


@pytest.fixture(scope="module")
def ctx(hjm):
    c = hjm.Context(0)
    yield c
    c.close()


def _rel(keys, width):
    dt = np.uint32 if width == 4 else np.uint64
    return np.stack([keys.astype(dt), np.arange(len(keys), dtype=dt)], 1)


def _check(hjm, ctx, r, s, **kw):
    def gpu(a):
        return torch.from_numpy(np.ascontiguousarray(a).view(np.int32 if a.dtype == np.uint32 else np.int64)).to(DEV)

    want = oracle.sorted_pairs(*oracle.hash_join(r, s))
    res = hjm.hj_join(ctx, gpu(r), gpu(s), algo=hjm.HJ_ALGO_SHJ, **kw)
    got = res.pairs_numpy().astype(np.uint64)
    assert res.count == len(want) and res.algo == hjm.HJ_ALGO_SHJ
    res.free()
    assert np.array_equal(oracle.sorted_pairs(got[:, 0], got[:, 1]), want)


LIMIT = {4: 8192, 8: 4096}


@pytest.mark.parametrize("ns", [1, 127, 1281, 50_001, 700_001])
@pytest.mark.parametrize("nr", ["1", "3", "half", "limit-1", "limit", "limit+1"])
@pytest.mark.parametrize("width", [4, 8])
def test_sizes(hjm, ctx, width, nr, ns):
    n = {"1": 1, "3": 3, "half": LIMIT[width] // 2 + 1, "limit-1": LIMIT[width] - 1, "limit": LIMIT[width],
         "limit+1": LIMIT[width] + 1}[nr]
    rng = np.random.default_rng(ns + n)
    _check(hjm, ctx, _rel(rng.permutation(np.arange(1, n + 1)), width), _rel(rng.integers(1, 2 * n + 1, ns), width))


@pytest.mark.parametrize("n_ones", [0, 1, 64, 65])
@pytest.mark.parametrize("width", [4, 8])
def test_keys_of_all_ones(hjm, ctx, width, n_ones):
    # in R (64 fit the list, 65 take the fallback) and in S, where they meet no empty slot;
    # one of R's has a rid of all ones too
    dt = np.uint32 if width == 4 else np.uint64
    ones = np.iinfo(dt).max
    rng = np.random.default_rng(n_ones)
    r = _rel(np.arange(1, 1500), width)
    r[rng.choice(len(r), n_ones, replace=False), 0] = ones
    if n_ones:
        r[np.nonzero(r[:, 0] == ones)[0][0], 1] = ones
    s = _rel(rng.integers(1, 2500, 9999), width)
    s[::111, 0] = ones
    _check(hjm, ctx, r, s)


@pytest.mark.parametrize("copies", [2, 5, 200, 3000])
@pytest.mark.parametrize("width", [4, 8])
def test_repeated_keys(hjm, ctx, width, copies):
    # one key `copies` times (thousands pass the walk limit), every other key twice
    rng = np.random.default_rng(copies)
    rk = np.concatenate([np.full(copies, 7), np.repeat(np.arange(10, 400), 2)])
    s = _rel(rng.integers(1, 600, 6001), width)
    _check(hjm, ctx, _rel(rk[rng.permutation(len(rk))], width), s)
    _check(hjm, ctx, _rel(rk[rng.permutation(len(rk))], width), s, out_capacity=17)
