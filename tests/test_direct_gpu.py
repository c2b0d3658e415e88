"""One global table whose outputs are written as their keys are claimed (csrc/global.cu), against the
oracle: products around a tile of 1,024, one X entry over many tiles, many X entries without a
product between those with, every product on few keys, the line to the table of values (twice the
products), output orders and key form."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def check(X, Y, out=None):
    import oracle
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    res = gpu_contract(W.Problem(X, Y, (1,), (0,), out), strategy=1)
    ref = oracle.contract(X, Y, (1,), (0,), out)
    assert_matches_oracle(*result_host(res), ref)
    assert res.stats.products == ref.products
    return res


@pytest.mark.parametrize("products", [1, 255, 1023, 1024, 1025, 4096, 70_001])
def test_one_entry_over_tiles(products):
    rng = W.rng_for(8800 + products)
    X = W.COO((3_000_000, 2), np.array([[7, 1]], np.int32), np.array([0.5]))
    Y = W.uniform_coo(rng, (2, 100_000), products)
    Y.coords[:, 0] = 1
    check(X, Y)


@pytest.mark.parametrize("nx,ny,fx,fy", [(5_000, 4_000, 900_000, 7_001), (30_000, 300, 2_000_000, 900), (700, 60_000, 60_000, 60_000)])
def test_uneven_runs(nx, ny, fx, fy):
    rng = W.rng_for(8810 + nx)
    X, Y = W.uniform_coo(rng, (fx, 500), nx), W.uniform_coo(rng, (500, fy), ny)
    Y.coords[: ny // 2, 0] = 3
    Y.coords[ny // 2:, 0] %= 90
    check(X, Y, (1, 0))


@pytest.mark.parametrize("nx,ny,fx,fy", [(6_000, 900, 3, 2), (6_000, 900, 1, 1), (12_000, 10_000, 32, 32), (12_000, 10_000, 25, 41)])
def test_all_products_on_few_keys(nx, ny, fx, fy):
    """Almost every product finds its key claimed: on either side of the 1,024 keys whose repeats each
    CTA sums first. Up to 2.7e5 terms of random signs in a sum: rounding errors of two orders of
    summation differ by about sqrt(n) u = 6e-14 of sum|x*y|, well inside REL_TOL."""
    rng = W.rng_for(8820 + fx + fy)
    X, Y = W.uniform_coo(rng, (3_000_000, 20), nx), W.uniform_coo(rng, (20, 4_100), ny)
    X.coords[:, 0] = rng.integers(0, fx, nx) * 30_001
    Y.coords[:, 1] = rng.integers(0, fy, ny) * 99
    res = check(X, Y)
    assert res.nnz == fx * fy


@pytest.mark.parametrize("fy", [2 * 1_300 - 1, 2 * 1_300, 2 * 1_300 + 1])
def test_line(fy):
    """F around twice the products."""
    rng = W.rng_for(8830 + fy)
    X = W.COO((200, 1), np.stack([np.arange(200), np.zeros(200)], 1).astype(np.int32), W.nonzero_values(rng, 200))
    Y = W.COO((1, fy), np.stack([np.zeros(1300), rng.integers(0, fy, 1300)], 1).astype(np.int32), W.nonzero_values(rng, 1300))
    check(X, Y)


def test_output_keys_beyond_32_bits():
    import paper_2410_10094_gb300 as stc
    from gpu_util import to_dev

    rng = W.rng_for(8840)
    X, Y = W.uniform_coo(rng, (2_000_000, 40), 3_000), W.uniform_coo(rng, (40, 90_000), 900)
    a = stc.contract(to_dev(X), to_dev(Y), (1,), (0,), strategy=1, output_keys=True, operands=stc.OPERANDS_AS_GIVEN)
    import oracle

    ref = oracle.contract(X, Y, (1,), (0,), None)
    want = ref.coords[:, 0].astype(np.int64) * 90_000 + ref.coords[:, 1]
    got = a.keys.cpu().numpy()
    order = np.argsort(got)
    np.testing.assert_array_equal(got[order], want)
    assert np.all(np.abs(a.vals.cpu().numpy()[order] - ref.vals) <= 1e-12 * ref.abs)


def test_within_the_counted_bytes():
    """A context whose budget is the bound of stc_count keeps the table of values."""
    import gc

    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, result_host, to_dev

    rng = W.rng_for(8850)
    X, Y = W.uniform_coo(rng, (2_000_000, 40), 30_000), W.uniform_coo(rng, (40, 90_000), 4_000)
    wide = stc.Context(mem_budget_bytes=8 << 30)
    _, need = stc.count(to_dev(X), to_dev(Y), (1,), (0,), ctx=wide)
    tight = stc.Context(mem_budget_bytes=need)
    res = stc.contract(to_dev(X), to_dev(Y), (1,), (0,), ctx=tight)
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (1,), (0,), None))
    del res
    gc.collect()
    wide.close()
    tight.close()
