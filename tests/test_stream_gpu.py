"""The streaming kernel (csrc/stream.cu) at the sizes where it can go wrong, against the oracle:
groups of one product up to its capacity of 8,192 products, runs around the quarter-slot's 8
entries, repeats around the 512 that its list holds, free key spaces around a bitmap word and a
segment, and every form of output row. Tolerance: REL_TOL * sum|x*y| (see helpers)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def check(p, **kw):
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    res = gpu_contract(p, strategy=2, **kw)
    ref = oracle.contract(p.X, p.Y, p.cx, p.cy, p.out_order)
    assert_matches_oracle(*result_host(res), ref)
    assert res.stats.products == ref.products
    return res


def runs(rng, keys, length, fy, distinct=False):
    """Y with `length` entries on each of `keys` contract keys."""
    c = np.empty((keys * length, 2), np.int32)
    c[:, 0] = np.repeat(np.arange(keys), length)
    if distinct:
        c[:, 1] = np.concatenate([rng.permutation(fy)[:length] for _ in range(keys)])
    else:
        c[:, 1] = rng.integers(0, fy, keys * length)
    return W.COO((keys, fy), c, W.nonzero_values(rng, len(c)))


def rows(rng, groups, entries, keys):
    """X with `entries` entries on different contract keys in each of `groups` rows."""
    c = np.empty((groups * entries, 2), np.int32)
    c[:, 0] = np.repeat(np.arange(groups), entries)
    c[:, 1] = np.concatenate([rng.permutation(keys)[:entries] for _ in range(groups)])
    return W.COO((groups, keys), c, W.nonzero_values(rng, len(c)))


@pytest.mark.parametrize("entries,length", [(1, 1), (1, 7), (1, 8), (1, 9), (1, 8192), (16, 512), (257, 31), (300, 27),
                                            (1000, 8), (4, 2049), (5, 1638)])
def test_group_sizes(entries, length):
    rng = W.rng_for(8000 + 31 * entries + length)
    check(W.Problem(rows(rng, 5, entries, max(entries, 3)), runs(rng, max(entries, 3), length, 40_000), (1,), (0,)),
          accumulator=2)


@pytest.mark.parametrize("fy", [33, 64, 1000, 65_535, 65_536, 65_537, 200_000])
@pytest.mark.parametrize("per_key", [1, 2])
def test_repeats_and_free_key_spaces(fy, per_key):
    """From hardly any repeats to every key met several times; the last free key is present."""
    rng = W.rng_for(8100 + fy + per_key)
    length = min(fy, 900)
    Y = runs(rng, 4, length, fy, distinct=True)
    Y.coords[::length, 1] = fy - 1
    X = rows(rng, 700, 3, 4)
    X = W.COO(X.shape, np.concatenate([X.coords] * per_key), W.nonzero_values(rng, X.nnz * per_key))
    check(W.Problem(X, Y, (1,), (0,)), accumulator=2)


@pytest.mark.parametrize("reps", [0, 1, 511, 512, 513, 2000])
def test_list_of_repeats(reps):
    """Two runs of 3,000 keys that share `reps` of them, in groups large enough to be streamed."""
    rng = W.rng_for(8200 + reps)
    keys = rng.permutation(30_000)
    c = np.concatenate([np.stack([np.zeros(3000), keys[:3000]], 1), np.stack([np.ones(3000), keys[3000 - reps:6000 - reps]], 1)])
    Y = W.COO((2, 30_000), c.astype(np.int32), W.nonzero_values(rng, 6000))
    res = check(W.Problem(rows(rng, 900, 2, 2), Y, (1,), (0,)))
    assert res.nnz == 900 * (6000 - reps)


@pytest.mark.parametrize("length", [800, 1_301])
@pytest.mark.parametrize("repeats", [False, True])
def test_groups_handing_on_positions(length, repeats):
    """Many groups per CTA whose leftover positions the next group fills: groups without a repeat
    between groups that leave hundreds, so that every thread of a CTA has to carry the same leftovers
    on (a group without repeats has no barrier between its counts and the end of the group)."""
    rng = W.rng_for(8250 + length + repeats)
    fy = 30_000
    Y = runs(rng, 12, length, fy, distinct=True)
    groups = 5_000
    c = np.stack([np.arange(groups), rng.integers(0, 12, groups)], 1)
    if repeats:  # every third group meets its run twice: as many repeats as outputs
        c = np.concatenate([c, c[::3]])
    X = W.COO((groups, 12), c.astype(np.int32), W.nonzero_values(rng, len(c)))
    for _ in range(2):
        res = check(W.Problem(X, Y, (1,), (0,)), accumulator=2)
        assert res.nnz == groups * length


def mostly_repeats(rng):
    """4,000 groups of 6,000 products on 500 to 520 keys each: more than ten million positions left over,
    where the first filling of holes expects five."""
    pool = rng.permutation(8192)[:520]
    c = np.stack([np.repeat(np.arange(12), 500), np.concatenate([rng.permutation(pool)[:500] for _ in range(12)])], 1)
    Y = W.COO((12, 8192), c.astype(np.int32), W.nonzero_values(rng, len(c)))
    return W.Problem(rows(rng, 4_000, 12, 12), Y, (1,), (0,))


def test_more_holes_than_expected():
    """Filled in further rounds."""
    check(mostly_repeats(W.rng_for(8260)), accumulator=2)


def test_holes_without_memory_for_them():
    """A context whose budget is the bound of stc_count: the holes are filled in rounds through an array
    that the call has already."""
    import gc

    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, result_host, to_dev

    p = mostly_repeats(W.rng_for(8270))
    dev = to_dev(p.X), to_dev(p.Y), p.cx, p.cy
    wide = stc.Context(mem_budget_bytes=8 << 30)
    _, need = stc.count(*dev, ctx=wide)
    wide.close()
    tight = stc.Context(mem_budget_bytes=need)
    res = stc.contract(*dev, ctx=tight, strategy=2, accumulator=2, operands=stc.OPERANDS_AS_GIVEN)
    assert res.stats.out_capacity == res.stats.products == 24_000_000
    assert_matches_oracle(*result_host(res), oracle.contract(p.X, p.Y, p.cx, p.cy, None))
    del res
    gc.collect()
    tight.close()


@pytest.mark.parametrize("xs,ys,out", [((30, 5), (40, 25), None), ((32, 4), (64, 16), None), ((32, 4), (64, 16), (3, 1, 0, 2)),
                                       ((7, 5), (9, 120), (1, 0, 3, 2)), ((100,), (50, 20), None), ((100,), (1000,), None),
                                       ((10, 10), (10, 10, 10), None), ((5, 4, 3), (12, 9, 10), None),
                                       ((2, 3, 4, 5), (10, 10, 10), None), ((128,), (16, 8, 8), None),
                                       ((16, 8, 4), (1024,), None)])
def test_output_rows(xs, ys, out):
    rng = W.rng_for(8300 + sum(xs) * 7 + sum(ys))
    X = W.uniform_coo(rng, xs + (50,), 4_000)
    Y = W.uniform_coo(rng, (50,) + ys, 3_000)
    check(W.Problem(X, Y, (len(xs),), (0,), out_order=out), accumulator=2)


def test_output_keys():
    import paper_2410_10094_gb300 as stc
    from gpu_util import to_dev

    rng = W.rng_for(8400)
    X, Y = W.uniform_coo(rng, (300, 40), 6_000), W.uniform_coo(rng, (40, 60, 50), 9_000)
    a = stc.contract(to_dev(X), to_dev(Y), (1,), (0,), strategy=2, accumulator=2, output_keys=True)
    b = stc.contract(to_dev(X), to_dev(Y), (1,), (0,), strategy=2, accumulator=1)
    bc = b.coords.cpu().numpy().astype(np.int64)
    want = np.sort((bc[:, 0] * 60 + bc[:, 1]) * 50 + bc[:, 2])
    np.testing.assert_array_equal(np.sort(a.keys.cpu().numpy()), want)
