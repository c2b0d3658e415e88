"""The lane-private rows (accumulator ROWS) by a CTA per group and by a warp per group, against
the oracle: pieces of 16 X entries and their remainders, one column up to 64, empty groups, runs
long and short. The number of groups decides the kernel (four per SM)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [3, 700])
@pytest.mark.parametrize("entries", [1, 15, 16, 17, 33, 250])
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
