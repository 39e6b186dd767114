"""The shared-memory join of partition pairs, against the CPU oracle: the probe loop
for tables whose keys are all different and the general one, chosen per partition by
comparing the table's keys (also those that moved past a full bucket); runs of repeated
keys; slice sizes around whole groups; the largest build partitions that the table takes;
more tasks than two per CTA, so that some are taken ahead; a pair buffer that ends inside
a warp's chunk.  Integer results: every comparison is exact."""
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


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32 if a.dtype == np.uint32 else np.int64)).to(DEV)


def _check(hjm, ctx, r, s, **kw):
    want = oracle.sorted_pairs(*oracle.hash_join(r, s))
    res = hjm.hj_join(ctx, _gpu(r), _gpu(s), algo=hjm.HJ_ALGO_PHJ, passes=1, **kw)
    got = res.pairs_numpy().astype(np.uint64)
    res.free()
    assert np.array_equal(oracle.sorted_pairs(got[:, 0], got[:, 1]), want)
    cnt, c0, c1 = oracle.join_aggregate(r, s)
    agg = hjm.hj_join(ctx, _gpu(r), _gpu(s), mode=hjm.HJ_COUNT_CHECKSUM, algo=hjm.HJ_ALGO_PHJ, passes=1,
                      radix_bits=kw["radix_bits"])
    assert (agg.count, *agg.checksum) == (cnt, c0, c1)


# R rows of a partition: small, an ordinary one, and one that fills the larger table
@pytest.mark.parametrize("per", [40, 1500, 7000])
@pytest.mark.parametrize("dups", ["none", "one", "pairs"])
@pytest.mark.parametrize("width", [4, 8])
def test_unique_and_repeated_keys(hjm, ctx, width, dups, per):
    # two partitions; "one": a single key twice in all of R (one partition takes the
    # general loop, the other the one for different keys); "pairs": every key twice
    if width == 8:
        per = per // 2
    rng = np.random.default_rng(per + width)
    n = 2 * per
    keys = rng.permutation(np.arange(1, n + 1))
    if dups == "one":
        keys[-1] = keys[0]
    elif dups == "pairs":
        keys = (keys + 1) // 2
    sk = rng.integers(1, 2 * n + 1, 4 * n + 77)
    _check(hjm, ctx, _rel(keys, width), _rel(sk, width), radix_bits=1)


@pytest.mark.parametrize("copies", [3, 4, 5, 9, 33, 100, 300])
@pytest.mark.parametrize("width", [4, 8])
def test_runs_of_repeated_keys(hjm, ctx, width, copies):
    # every key of R `copies` times, beside keys of one, two and twice as many rows: matches
    # that fill the home bucket, runs over many buckets, all walked together or one after the
    # other (the longest pass the insert's limit and take the key-list table)
    rng = np.random.default_rng(copies + width)
    k = 1200 // copies + 1
    keys = np.concatenate([np.repeat(np.arange(1, k + 1), copies), np.repeat(np.arange(k + 1, k + 4), 2 * copies),
                           np.arange(2000, 2400), np.repeat(np.arange(3000, 3100), 2)])
    sk = rng.integers(1, 3200, 9001)
    sk[:4000] = rng.integers(1, k + 4, 4000)
    _check(hjm, ctx, _rel(rng.permutation(keys), width), _rel(sk, width), radix_bits=1)


@pytest.mark.parametrize("cap", [0, 700])
@pytest.mark.parametrize("copies", [1, 2, 7, 40])
@pytest.mark.parametrize("width", [4, 8])
def test_pairs_with_checksums(hjm, ctx, width, copies, cap):
    # the sums are taken where the pairs are appended, of pairs that pass the buffer too
    rng = np.random.default_rng(copies)
    n = 3000
    r = _rel(rng.permutation(n) // copies + 1, width)
    s = _rel(rng.integers(1, 2 * n // copies, 4 * n + 1), width)
    res = hjm.hj_join(ctx, _gpu(r), _gpu(s), algo=hjm.HJ_ALGO_PHJ, radix_bits=2, passes=1, checksum=True,
                      out_capacity=cap)
    got = res.pairs_numpy().astype(np.uint64)
    assert (res.count, *res.checksum) == oracle.join_aggregate(r, s)
    res.free()
    assert np.array_equal(oracle.sorted_pairs(got[:, 0], got[:, 1]), oracle.sorted_pairs(*oracle.hash_join(r, s)))


@pytest.mark.parametrize("ns", [1280, 1281, 1279, 2559, 2600, 5120 + 3])
@pytest.mark.parametrize("width", [4, 8])
def test_slices_around_whole_groups(hjm, ctx, width, ns):
    # a group is 64 vectors (of two 4-byte tuples or one 8-byte), a CTA takes 20 at once
    rng = np.random.default_rng(ns)
    r = _rel(rng.permutation(np.arange(1, 201)), width)
    s = _rel(rng.integers(1, 301, ns), width)
    _check(hjm, ctx, r, s, radix_bits=1)


@pytest.mark.parametrize("cap", [0, 1, 1500, 40_000])
def test_many_tasks_and_a_buffer_that_ends_inside_a_chunk(hjm, ctx, cap):
    # 2^11 tasks of a few tuples each, more than two per CTA
    rng = np.random.default_rng(cap)
    r = _rel(rng.permutation(np.arange(1, 30_001)), 4)
    s = _rel(rng.integers(1, 45_001, 90_003), 4)
    _check(hjm, ctx, r, s, radix_bits=11, out_capacity=cap)


@pytest.mark.parametrize("nr,ns", [(50_001, 3), (3, 50_001), (70_001, 70_000), (100, 0), (0, 100), (1, 1)])
@pytest.mark.parametrize("width,bits", [(4, 3), (4, 11), (8, 10)])
def test_both_relations_in_one_pass(hjm, ctx, width, bits, nr, ns):
    # one histogram and one scatter launch take the chunks of both, the larger first
    rng = np.random.default_rng(nr + ns)
    r = _rel(rng.permutation(np.arange(1, nr + 1)), width)
    s = _rel(rng.integers(1, 2 * nr + 2, ns), width)
    _check(hjm, ctx, r, s, radix_bits=bits)


@pytest.mark.parametrize("width,per", [(4, 18_000), (4, 19_400), (8, 8_900), (8, 9_400)])
def test_largest_partitions_stay_in_shared_memory(hjm, ctx, width, per):
    # 25088 4-byte or 12160 8-byte slots at a load of at most 4/5 take partitions of up to 20070
    # or 9728 rows (the largest of these 8 hold 19593 and 9577, and less than 60 of padding)
    rng = np.random.default_rng(per)
    r = _rel(rng.permutation(np.arange(1, 8 * per + 1)), width)
    s = _rel(rng.integers(1, 16 * per, 100_003), width)
    hjm.prof_reset(ctx)
    hjm.prof_enable(ctx, True)
    try:
        res = hjm.hj_join(ctx, _gpu(r), _gpu(s), algo=hjm.HJ_ALGO_PHJ, radix_bits=3, passes=1)
        launched = set(hjm.prof_read(ctx))
    finally:
        hjm.prof_enable(ctx, False)
    got = res.pairs_numpy().astype(np.uint64)
    res.free()
    assert np.array_equal(oracle.sorted_pairs(got[:, 0], got[:, 1]), oracle.sorted_pairs(*oracle.hash_join(r, s)))
    assert "partition_join" in launched and "fallback_tasks" not in launched
