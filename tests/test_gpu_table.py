"""The simple hash join's table of 32-byte buckets: build and probe against the CPU
oracle at the edges of a warp's probe group and of a bucket, with repeated keys, the
key that empty slots hold, and runs that fill many buckets and wrap at the table's
end.  All results are whole numbers: exact."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hjm():
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
    keys = np.asarray(keys, dtype=dt)
    return np.stack([keys, np.arange(len(keys), dtype=dt) * dt(3) + dt(1)], axis=1)


def _gpu(a):
    return torch.from_numpy(a.view(np.int32 if a.dtype == np.uint32 else np.int64).copy()).to("cuda:0")


def _check(hjm, ctx, R, S, budget=0):
    want = oracle.sorted_pairs(*oracle.hash_join(R, S))
    agg = oracle.join_aggregate(R, S)
    Rg, Sg = _gpu(R), _gpu(S)
    c = hjm.Context(0, budget=budget) if budget else ctx
    for run in ("join", "probe"):
        table = hjm.hj_build(c, Rg) if run == "probe" else None
        for checksum in (False, True):
            res = hjm.hj_probe(c, table, Sg, checksum=checksum) if table else \
                hjm.hj_join(c, Rg, Sg, algo=hjm.HJ_ALGO_SHJ, checksum=checksum)
            p = res.pairs_numpy().astype(np.uint64)
            assert res.count == len(want) == agg[0]
            np.testing.assert_array_equal(oracle.sorted_pairs(p[:, 0], p[:, 1]), want)
            if checksum:
                assert res.checksum == (agg[1], agg[2])
            res.free()
        if table:
            table.free()
    res = hjm.hj_join(c, Rg, Sg, algo=hjm.HJ_ALGO_SHJ, mode=hjm.HJ_COUNT_CHECKSUM)
    assert (res.count,) + tuple(res.checksum) == agg
    res.free()
    if budget:
        c.close()


@pytest.mark.parametrize("width", [4, 8])
@pytest.mark.parametrize("nr,ns", [(0, 5), (1, 1), (2, 63), (15, 64), (16, 65), (17, 127), (64, 128), (300, 129),
                                   (4097, 10007), (70001, 8191)])
def test_sizes_at_the_edges_of_groups_and_tables(hjm, ctx, width, nr, ns):
    rng = np.random.default_rng(nr * 131 + ns)
    rk = rng.permutation(max(nr, 1))[:nr] + 1
    sk = rng.integers(1, 2 * nr + 2, ns)
    _check(hjm, ctx, _rel(rk, width), _rel(sk, width))
    if nr == 4097:  # under a memory budget the table keeps its smaller size
        _check(hjm, ctx, _rel(rk, width), _rel(sk, width), budget=64 << 20)


@pytest.mark.parametrize("width", [4, 8])
@pytest.mark.parametrize("copies", [1, 2, 3, 40])
def test_repeated_and_extreme_keys(hjm, ctx, width, copies):
    ones = 2 ** (8 * width) - 1
    keys = np.concatenate([np.arange(500, dtype=np.uint64)] + [np.array([0, 7, ones], np.uint64)] * copies)
    R = _rel(np.random.default_rng(copies).permutation(keys), width)
    if copies != 2:  # the tuple that equals an empty slot
        R[-1] = ones
        if copies == 40:
            R[:3] = ones
    S = _rel(np.concatenate([np.arange(600, dtype=np.uint64), np.full(70, ones, np.uint64)]), width)
    _check(hjm, ctx, R, S)


@pytest.mark.parametrize("width", [4, 8])
@pytest.mark.parametrize("repeat", [1, 2])
def test_long_runs_that_wrap(hjm, ctx, width, repeat):
    # 120 distinct keys of one home bucket, the table's last: four slots per tuple
    # make as many buckets as tuples (4-byte) or twice as many (8-byte)
    n = 600
    nb = n if width == 4 else 2 * n
    crowd = []
    k = 1
    while len(crowd) < 120 // repeat:
        h = oracle.key_hash(k, width) >> (0 if width == 4 else 32)
        if h * nb >> 32 == nb - 1:
            crowd.append(k)
        k += 1
    others = np.arange(10 ** 6, 10 ** 6 + n - repeat * len(crowd))
    R = _rel(np.concatenate([crowd] * repeat + [others]), width)
    S = _rel(np.concatenate([crowd, crowd, others, np.arange(3 * 10 ** 6, 3 * 10 ** 6 + 4000)]), width)
    _check(hjm, ctx, R, S)
