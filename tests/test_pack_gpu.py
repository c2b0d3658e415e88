"""Many small groups of one contraction (four to a warp, output positions in chunks), against the
oracle: one product per group up to the class's limit and past it, runs that repeat keys, more
products than keys, groups of more than 32 entries, and free key spaces at the limit of the packed
key (2^30)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def check(X, Y, **kw):
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    p = W.Problem(X, Y, (1,), (0,), **kw)
    res = gpu_contract(p, strategy=2, accumulator=1)
    ref = oracle.contract(p.X, p.Y, p.cx, p.cy, p.out_order)
    assert_matches_oracle(*result_host(res), ref)
    assert res.stats.products == ref.products
    return res


@pytest.mark.parametrize("groups", [16_383, 16_384, 16_385, 30_002])
@pytest.mark.parametrize("entries,fy,ny", [(1, 50_000, 400), (3, 50_000, 2_000), (2, 9, 3_000), (5, 7_000, 4_000)])
def test_packed_groups(groups, entries, fy, ny):
    rng = W.rng_for(8600 + groups + entries + fy)
    xc = np.stack([np.repeat(np.arange(groups), entries), rng.integers(0, 100, groups * entries)], 1)
    X = W.COO((groups, 100), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    check(X, W.uniform_coo(rng, (100, fy), ny))


def test_uneven_groups():
    """From empty groups to groups of 80 entries and of the next class, in one list."""
    rng = W.rng_for(8650)
    n = rng.integers(0, 4, 24_000)
    n[::97] = 80
    n[5::301] = 12
    xc = np.stack([np.repeat(np.arange(24_000), n), rng.integers(0, 60, n.sum())], 1)
    X = W.COO((24_000, 60), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    check(X, W.uniform_coo(rng, (60, 3_000), 700))


@pytest.mark.parametrize("fy", [(1 << 30) - 1, 1 << 30])
def test_widest_packed_key(fy):
    rng = W.rng_for(8660 + (fy & 3))
    X = W.uniform_coo(rng, (20_000, 50), 60_000)
    yc = np.stack([rng.integers(0, 50, 600), rng.integers(0, fy, 600)], 1)
    yc[::7, 1] = fy - 1
    Y = W.COO((50, fy), yc.astype(np.int32), W.nonzero_values(rng, 600))
    res = check(X, Y, out_order=(1, 0))
    if fy == 1 << 30:  # not packed: no room for chunks either (no group has as many products as free keys)
        assert res.stats.out_capacity == res.stats.products
