"""Many small groups of one contraction (four to a warp), against the
oracle: one product per group up to the class's limit and past it, runs that repeat keys, more
products than keys, groups of more than 32 entries, and free key spaces at the limit of the packed
key (2^30)."""
import gc

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


@pytest.mark.parametrize("fy", [1, 100, 700, 1 << 33])
@pytest.mark.parametrize("entries", [15, 16, 17, 400])
def test_many_products_on_few_keys(entries, fy):
    """Groups of 1,920 to 51,200 products among packed ones, on either side of the 2,048 that a warp takes,
    over fewer keys than its table has slots; and with 64-bit keys."""
    rng = W.rng_for(8655 + entries + fy % 999)
    groups = 16_500
    n = np.ones(groups, np.int64)
    n[::1000] = entries
    xc = np.stack([np.repeat(np.arange(groups), n), rng.integers(0, 50, n.sum())], 1)
    X = W.COO((groups, 50), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    yc = np.stack([np.repeat(np.arange(50), 128), rng.integers(0, min(fy, 700), 50 * 128)], 1)
    if fy > 1 << 31:  # two free modes of Y
        yc = np.insert(yc, 2, rng.integers(0, 9, len(yc)), 1)
        check(X, W.COO((50, 1 << 17, 1 << 16), yc.astype(np.int32), W.nonzero_values(rng, len(yc))))
    else:
        check(X, W.COO((50, fy), yc.astype(np.int32), W.nonzero_values(rng, len(yc))))


@pytest.mark.parametrize("fy", [(1 << 30) - 1, 1 << 30])
def test_widest_packed_key(fy):
    rng = W.rng_for(8660 + (fy & 3))
    X = W.uniform_coo(rng, (20_000, 50), 60_000)
    yc = np.stack([rng.integers(0, 50, 600), rng.integers(0, fy, 600)], 1)
    yc[::7, 1] = fy - 1
    Y = W.COO((50, fy), yc.astype(np.int32), W.nonzero_values(rng, 600))
    res = check(X, Y, out_order=(1, 0))
    assert res.stats.out_capacity == res.stats.products  # no group has as many products as free keys


def smallest_budget(call):
    """The smallest budget of a context in which call(ctx) finds its memory."""
    import paper_2410_10094_gb300 as stc

    def fits(budget):
        ctx = stc.Context(mem_budget_bytes=budget)
        try:
            call(ctx)
            return True
        except stc.StcError as e:
            assert e.status == 4
            return False
        finally:
            gc.collect()
            ctx.close()

    lo, hi = 1, 1 << 33
    assert fits(hi)
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    return hi


def test_budget_of_the_scanned_tables():
    """Small groups enough to be packed, beside groups whose tables lie in global memory, in the smallest
    budget of the call that scans its tables: the call with direct output needs no more, and its result
    holds no more."""
    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, result_host, to_dev

    rng = W.rng_for(8670)
    small, large, fy = 20_000, 10, 60_000
    length = np.array([45] * 40 + [5_000] * 5)
    yk = np.repeat(np.arange(45), length)
    Y = W.COO((45, fy), np.stack([yk, rng.integers(0, fy, len(yk))], 1).astype(np.int32), W.nonzero_values(rng, len(yk)))
    xc = np.stack([np.concatenate([np.arange(small), small + np.repeat(np.arange(large), 5)]),
                   np.concatenate([rng.integers(0, 40, small), np.tile(np.arange(40, 45), large)])], 1)
    X = W.COO((small + large, 45), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    dev = to_dev(X), to_dev(Y), (1,), (0,)
    how = dict(strategy=2, operands=stc.OPERANDS_AS_GIVEN)
    need = smallest_budget(lambda ctx: stc.contract(*dev, accumulator=3, ctx=ctx, **how))
    ctx = stc.Context(mem_budget_bytes=need)
    res = stc.contract(*dev, accumulator=1, ctx=ctx, **how)
    assert res.stats.table_slots > 0  # some groups' tables did lie in global memory
    assert res.stats.out_capacity == res.stats.products  # every group has fewer products than free keys
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (1,), (0,), None))
    del res
    gc.collect()
    ctx.close()
