"""Small output key spaces (F up to 2^18) accumulated in an array of the whole space, against the
oracle: survivors around a block of 1,024 and none at all, products around a tile of 1,024, runs
long and short, spaces that are no multiple of a word, keys that only receive zeros."""
import numpy as np
import pytest

import workloads as W
from helpers import REL_TOL

pytestmark = pytest.mark.gpu


def check(X, Y, **kw):
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    res = gpu_contract(W.Problem(X, Y, (1,), (0,)), strategy=1, **kw)
    ref = oracle.contract(X, Y, (1,), (0,))
    # Two orders of summing n products differ by at most 2 (n - 1) u of sum|x*y|.
    most = int(ref.cnt.max()) if len(ref.cnt) else 0
    assert_matches_oracle(*result_host(res), ref, max(REL_TOL, 2.0 ** -52 * most))
    assert res.stats.products == ref.products and res.stats.survivors == np.isin(X.coords[:, 1], Y.coords[:, 0]).sum()
    return res


@pytest.mark.parametrize("probe", [0, 1])
@pytest.mark.parametrize("survivors", [0, 1, 31, 1023, 1024, 1025, 5000])
@pytest.mark.parametrize("run", [1, 3, 700])
def test_survivors(survivors, run, probe):
    rng = W.rng_for(8900 + survivors + run)
    nx = survivors + 4000
    X = W.uniform_coo(rng, (61, 3000), nx)
    X.coords[:, 1] = 1000 + X.coords[:, 1] % 2000
    X.coords[rng.permutation(nx)[:survivors], 1] = rng.integers(0, 40, survivors)
    Y = W.uniform_coo(rng, (3000, 97), 40 * run)
    Y.coords[:, 0] = np.repeat(np.arange(40), run)
    check(X, Y, probe=probe)


@pytest.mark.parametrize("f", [(1, 1), (1, 7), (33, 31), (512, 512), (262_144, 1), (3, 87_381)])
def test_spaces(f):
    rng = W.rng_for(8950 + f[0])
    check(W.uniform_coo(rng, (f[0], 90), 9_000), W.uniform_coo(rng, (90, f[1]), 5_000))


def test_cancelled_outputs_stay():
    X = W.COO((4, 2), np.array([[1, 0], [1, 1], [3, 0]], np.int32), np.array([2.0, -2.0, 1.0]))
    Y = W.COO((2, 5), np.array([[0, 4], [1, 4]], np.int32), np.array([3.0, 3.0]))
    check(X, Y)


@pytest.mark.parametrize("x,y", [(-0.0, 3.0), (0.0, -3.0), (-0.0, -3.0), (1e-200, -1e-200)])
def test_products_of_zero(x, y):
    """Zeros of either sign, given or underflown, are products like any other: their outputs exist, and
    are +0.0 where nothing else is added."""
    X = W.COO((4, 2), np.array([[1, 0], [2, 0], [3, 1]], np.int32), np.array([x, x, 2.0]))
    Y = W.COO((2, 5), np.array([[0, 4], [0, 4], [0, 0], [1, 0]], np.int32), np.array([y, y, y, 1.0]))
    import oracle
    from gpu_util import gpu_contract, result_host

    c, v = result_host(gpu_contract(W.Problem(X, Y, (1,), (0,)), strategy=1))
    ref = oracle.contract(X, Y, (1,), (0,))
    at = np.lexsort(c.T[::-1])
    np.testing.assert_array_equal(c[at], ref.coords)
    np.testing.assert_array_equal(v[at], ref.vals)
    assert not np.signbit(v[v == 0]).any()


@pytest.mark.parametrize("shape,row", [((2000, 130), 1), ((4096, 64), 3), ((37, 4095), 1), ((1, 300), 1)])
def test_most_products_on_few_rows(shape, row):
    rng = W.rng_for(8970 + shape[0])
    X, Y = W.uniform_coo(rng, (shape[0], 200), 8_000), W.uniform_coo(rng, (200, shape[1]), 6_000)
    X.coords[500:, 0] = rng.integers(0, row, 7_500)
    check(X, Y)


@pytest.mark.parametrize("probe", [0, 1])
@pytest.mark.parametrize("nx,run", [(12_000, 2_000), (2_050, 11_000), (9, 2_800_000)])
def test_many_products_per_survivor(nx, run, probe):
    """Tiles of more than 1,024 products: from several survivors to a part of one."""
    rng = W.rng_for(8980 + nx)
    X = W.uniform_coo(rng, (50, 4), nx)
    Y = W.uniform_coo(rng, (4, 60), 4 * run)
    Y.coords[:, 0] = np.repeat(np.arange(4), run)
    res = check(X, Y, probe=probe)
    assert res.stats.products == nx * run


def test_one_long_run_among_short_ones():
    rng = W.rng_for(8960)
    Y = W.uniform_coo(rng, (500, 64), 20_000)
    Y.coords[:15_000, 0] = 77
    X = W.uniform_coo(rng, (900, 500), 30_000)
    check(X, Y)
