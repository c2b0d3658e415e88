"""The larger groups of a batch by the two-pass kernel, against the oracle, called (also under a
budget, which keeps the hash tables) and replayed: group sizes, free key spaces and entry counts at the
limits of its three forms and one past them, as many repeats as a small and a larger group list and one
more, keys that repeat many times, runs scaled by one entry, rows of 2 to 9 coordinates, and more
problems than the binning holds offsets for."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def problem(seed, groups, yfree, products, entries, keys=None, xfree=None, out_order=None):
    """`groups` groups of `entries` X entries with `products` products each over Y's free modes; the
    free keys are drawn from the first `keys` of them (default all), without repeats within a run."""
    rng = W.rng_for(8700 + seed)
    fy = int(np.prod(yfree))
    share = np.full(entries, products // entries)
    share[: products % entries] += 1
    fk = np.concatenate([rng.choice(keys or fy, n, replace=n > (keys or fy)) for n in share])
    yc = np.column_stack([np.repeat(np.arange(entries), share), *np.unravel_index(fk, yfree)])
    Y = W.COO((entries, *yfree), yc.astype(np.int32), W.nonzero_values(rng, products))
    xfree = xfree or (groups,)
    fx = rng.choice(int(np.prod(xfree)), groups, replace=False)
    xc = np.column_stack([*(np.repeat(c, entries) for c in np.unravel_index(fx, xfree)),
                          np.tile(np.arange(entries), groups)])
    X = W.COO((*xfree, entries), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    return W.Problem(X, Y, (len(xfree),), (0,), out_order=out_order)


def check(probs):
    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, result_host, to_dev

    dev = [(to_dev(p.X), to_dev(p.Y), p.cx, p.cy, p.out_order) for p in probs]
    small = stc.Context(mem_budget_bytes=8 << 30)
    refs = [oracle.contract(p.X, p.Y, p.cx, p.cy, p.out_order) for p in probs]
    runs = [stc.contract_batch(dev), stc.contract_batch(dev, ctx=small)]
    plan = stc.BatchPlan(dev, group_load_factor=0.5)
    runs += [plan.run() for _ in range(3)]
    plan.close()
    for res in runs:
        for ref, r in zip(refs, res):
            assert_matches_oracle(*result_host(r), ref)
            assert r.stats.products == ref.products
    del runs, res, r
    small.close()


@pytest.mark.parametrize("yfree", [(256, 256), (255, 257), (65537,), (512, 512), (511, 513), (262145,)])
@pytest.mark.parametrize("products", [(770, 1025), (2048, 2049), (8192, 8193), (16384, 16385), (49152, 49153)])
def test_limits(yfree, products):
    check([problem(i, 4, yfree, p, 4) for i, p in enumerate(products)])


@pytest.mark.parametrize("entries", [1, 2, 255, 256, 257, 512, 513, 1024, 1025])
def test_entries(entries):
    check([problem(10 + i, 7, (9973,), 2311, entries, keys) for i, keys in enumerate([None, 2311])])


@pytest.mark.parametrize("products", [6400, 6404])
def test_most_products_per_key(products):
    check([problem(15, 5, (40, 40), products, 50)])


@pytest.mark.parametrize("keys", [2, 40, 700])
def test_keys_that_repeat(keys):
    """More repeats than are listed, most of few keys."""
    check([problem(20 + i, 4, fy, n, 3 * n // 6000, keys)
           for i, (fy, n) in enumerate([((251, 241), 6000), ((401, 503), 6000), ((401, 503), 20000)])])


@pytest.mark.parametrize("runs,repeats", [((1500, 1300), 255), ((1500, 1300), 256), ((1500, 1300), 257), ((1500, 1300), 513),
                                          ((1100, 948), 511), ((1100, 948), 512), ((1100, 948), 513), ((1100, 949), 512)])
def test_listed_repeats(runs, repeats):
    m, n = runs
    p = problem(30, 6, (9001,), m + n, 2, 2)
    first, second = np.arange(m), np.concatenate([np.arange(repeats), m + np.arange(n - repeats)])
    p.Y.coords[:, 0] = np.repeat([0, 1], runs)
    p.Y.coords[:, 1] = np.concatenate([first * 5, second * 5 % 9001])
    check([p])


@pytest.mark.parametrize("xfree,yfree", [((8,), (4001,)), ((3, 4), (61, 67)), ((2, 2, 3), (7, 5, 3, 11, 13)),
                                         ((2, 2, 3, 2), (7, 5, 3, 11, 13)), ((8, 2), (64, 64))])
def test_rows(xfree, yfree):
    q = [problem(40, 6, yfree, 1100, 3, xfree=xfree)]
    n = len(xfree) + len(yfree)
    q.append(problem(41, 6, yfree, 1100, 3, xfree=xfree, out_order=tuple(range(n))[::-1]))
    check(q)


def test_many_problems():
    check([problem(50 + i, 1 + i % 3, (3001,) if i % 9 == 0 else (40,), 900 if i % 9 == 0 else 30, 2)
           for i in range(1100)])
