"""The lane-private rows (accumulator ROWS) by a CTA per group and by a warp per group, against
the oracle: pieces of 16 X entries or fewer and their remainders, one column up to 64, empty groups,
runs long and short. The numbers of groups, products and entries decide the kernel: up to two groups per
SM take a CTA each, up to four and eight per SM from 6,144 and 16,384 products and 8 entries on average,
more from 49,152 products and 13 entries."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [3, 700])
@pytest.mark.parametrize("entries", [1, 12, 13, 14, 27, 207, 208, 209, 250])
@pytest.mark.parametrize("fy,run", [(1, 3), (33, 40), (64, 1), (64, 130)])
def test_rows_kernels(groups, entries, fy, run):
    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    rng = W.rng_for(8500 + groups + 7 * entries + fy + run)
    if groups * entries * run > 3_000_000:
        entries = 40
    xc = np.stack([np.repeat(np.arange(groups), entries), rng.integers(0, 20, groups * entries)], 1)
    xc = xc[xc[:, 0] % 5 != 1]  # some groups have no entries
    X = W.COO((groups, 20), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    yc = np.stack([np.repeat(np.arange(20), run), rng.integers(0, fy, 20 * run)], 1)
    Y = W.COO((20, fy), yc.astype(np.int32), W.nonzero_values(rng, len(yc)))
    p = W.Problem(X, Y, (1,), (0,))
    res = gpu_contract(p, strategy=2, accumulator=stc.ACC_ROWS)
    ref = oracle.contract(X, Y, (1,), (0,))
    assert_matches_oracle(*result_host(res), ref)
    assert res.stats.accumulator == stc.ACC_ROWS


@pytest.mark.parametrize("groups,entries,run", [(305, 8, 768), (305, 8, 767), (305, 7, 900), (609, 8, 2048), (609, 8, 2047), (1300, 16, 3072)])
def test_line(groups, entries, run):
    """On either side of the rules for more than two groups per SM."""
    import oracle
    import paper_2410_10094_gb300 as stc
    from gpu_util import assert_matches_oracle, gpu_contract, result_host

    rng = W.rng_for(8590 + groups + entries + run)
    xc = np.stack([np.repeat(np.arange(groups), entries), np.tile(np.arange(entries), groups)], 1)
    X = W.COO((groups, entries), xc.astype(np.int32), W.nonzero_values(rng, len(xc)))
    yc = np.stack([np.repeat(np.arange(entries), run), rng.integers(0, 64, entries * run)], 1)
    Y = W.COO((entries, 64), yc.astype(np.int32), W.nonzero_values(rng, len(yc)))
    res = gpu_contract(W.Problem(X, Y, (1,), (0,)), strategy=2, accumulator=stc.ACC_ROWS)
    assert_matches_oracle(*result_host(res), oracle.contract(X, Y, (1,), (0,)))
