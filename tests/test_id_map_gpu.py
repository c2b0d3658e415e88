"""Contract keys numbered through a bitmap of the key space (AUTO, key spaces above 2^22 that dwarf
the entries), against the oracle and against the other two ways (direct counting, the table of
contract_ids DENSE): mode orders, operand orders 1 to 5, both strategies, keys at the ends of the
space and of a bitmap word, empty intersections, and coordinates out of range."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def pools(rng, X, Y, cx, cy, n=40):
    """Puts the paired coordinates of both tensors on n common cells, the first and last among them."""
    cells = np.stack([rng.integers(0, X.shape[a], n) for a in cx], 1)
    cells[0] = 0
    cells[1] = [X.shape[a] - 1 for a in cx]
    cells[2, -1] = 31 % X.shape[cx[-1]]
    cells[3, -1] = 32 % X.shape[cx[-1]]
    X.coords[:, list(cx)] = cells[rng.integers(0, n, X.nnz)]
    Y.coords[:, list(cy)] = cells[rng.integers(0, n, Y.nnz)]


def check(p, ids, **kw):
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    ref = oracle.contract(p.X, p.Y, p.cx, p.cy, p.out_order)
    for way in (0, 1, 2):
        res = gpu_contract(p, contract_ids=way, **kw)
        assert_matches_oracle(*result_host(res), ref)
        assert res.stats.products == ref.products
        assert res.stats.contract_ids == (ids if way != 1 else 0)


def distinct(p):
    return len(np.unique(p.Y.coords[:, list(p.cy)], axis=0))


@pytest.mark.parametrize("strategy", [1, 2])
@pytest.mark.parametrize("xs,ys,cx,cy", [((2101, 2003, 9), (2101, 2003, 11), (0, 1), (0, 1)),
                                         ((7, 2003, 2101), (2101, 5, 2003), (2, 1), (0, 2)),
                                         ((5_000_003, 6), (5_000_003,), (0,), (0,)), ((9, 4_194_305), (4_194_305, 3), (1,), (0,)),
                                         ((3, 200, 4, 150, 160), (160, 200, 150, 8, 2), (1, 3, 4), (1, 2, 0)),
                                         ((40, 4_194_310), (4_194_310, 200_000), (1,), (0,))])
def test_forms(xs, ys, cx, cy, strategy):
    rng = W.rng_for(8700 + sum(xs) % 1000 + strategy)
    X, Y = W.uniform_coo(rng, xs, 4_000), W.uniform_coo(rng, ys, 3_000)
    pools(rng, X, Y, cx, cy)
    p = W.Problem(X, Y, cx, cy)
    check(p, distinct(p), strategy=strategy)


@pytest.mark.parametrize("k", [(1 << 28) - 1, 1 << 28, (1 << 28) + 1])
def test_widest_map(k):
    """The last key spaces with a map and the first with the table again; the number is the same."""
    rng = W.rng_for(8760 + k % 7)
    X, Y = W.uniform_coo(rng, (40, k), 600_000), W.uniform_coo(rng, (k, 30), 500_000)
    pools(rng, X, Y, (1,), (0,), n=100_000)
    p = W.Problem(X, Y, (1,), (0,))
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    res = gpu_contract(p)
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (1,), (0,)))
    assert res.stats.contract_ids == distinct(p)


@pytest.mark.parametrize("k,n,expect", [(1 << 22, 3_000, 0), ((1 << 22) + 1, 3_000, -1), ((1 << 22) + 1, 600_000, 0)])
def test_line(k, n, expect):
    """On either side of the rule: 2^22 keys are counted, more are numbered, unless they are few
    beside the entries (then the number is not reported either)."""
    rng = W.rng_for(8750 + k % 7 + n)
    X, Y = W.uniform_coo(rng, (40, k), n), W.uniform_coo(rng, (k, 30), n)
    pools(rng, X, Y, (1,), (0,), n=n // 4)
    p = W.Problem(X, Y, (1,), (0,))
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    res = gpu_contract(p)
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (1,), (0,)))
    assert res.stats.contract_ids == (distinct(p) if expect < 0 else 0)


def test_nothing_in_common_and_count():
    import paper_2410_10094_gb300 as stc
    from gpu_util import to_dev

    rng = W.rng_for(8770)
    X, Y = W.uniform_coo(rng, (50, 5_000_000), 900), W.uniform_coo(rng, (5_000_000, 60), 800)
    X.coords[:, 1] |= 1
    Y.coords[:, 0] &= ~1
    res = stc.contract(to_dev(X), to_dev(Y), (1,), (0,))
    assert res.nnz == 0 and res.stats.products == 0 and res.stats.contract_ids == len(np.unique(Y.coords[:, 0]))
    X.coords[::9, 1] = Y.coords[5, 0]
    same = int((Y.coords[:, 0] == Y.coords[5, 0]).sum())
    assert stc.count(to_dev(X), to_dev(Y), (1,), (0,))[0] == 100 * same


@pytest.mark.parametrize("which", ["X", "Y"])
@pytest.mark.parametrize("value", [-1, 5_000_000])
def test_out_of_range(which, value):
    import paper_2410_10094_gb300 as stc
    from gpu_util import to_dev

    rng = W.rng_for(8780)
    X, Y = W.uniform_coo(rng, (50, 5_000_000), 900), W.uniform_coo(rng, (5_000_000, 60), 800)
    (X if which == "X" else Y).coords[17, 1 if which == "X" else 0] = value
    with pytest.raises(stc.StcError) as e:
        stc.contract(to_dev(X), to_dev(Y), (1,), (0,))
    assert e.value.status == 8


def test_budget_keeps_the_table():
    """Under a budget the keys that were renumbered through the table still are."""
    import gc

    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, result_host, to_dev

    rng = W.rng_for(8960)
    X, Y = W.uniform_coo(rng, (1 << 23, 50), 60_000), W.uniform_coo(rng, (1 << 23, 30), 50_000)
    X.coords[:, 0] = Y.coords[rng.integers(0, 50_000, 60_000), 0]
    wide = stc.Context(mem_budget_bytes=8 << 30)
    _, need = stc.count(to_dev(X), to_dev(Y), (0,), (0,), ctx=wide)
    tight = stc.Context(mem_budget_bytes=need)
    res = stc.contract(to_dev(X), to_dev(Y), (0,), (0,), ctx=tight)
    assert res.stats.contract_ids == len(np.unique(Y.coords[:, 0]))
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (0,), (0,), None))
    del res
    gc.collect()
    wide.close()
    tight.close()
