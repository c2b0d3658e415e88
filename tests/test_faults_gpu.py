"""Failure paths, each made on the host (nothing faults, traps or hangs the GPU):

* an accumulation table sized too small on purpose (stc_opts.table_shrink): the kernel's
  bounded probe flags the overflow, the call retries at full capacity and the result still
  matches the oracle;
* a context budget smaller than one call's bound: STC_ERR_OUT_OF_MEMORY, nothing left held,
  and the context still serves smaller calls; a budget of the counted bound is enough;
* a request cancelled while it waits in the server's queue: its wait reports
  STC_ERR_CANCELLED, every other request finishes with its correct product count, and the
  server keeps serving.
"""
import pytest

import oracle
import workloads as W
from gpu_util import assert_matches_oracle, gpu_contract, result_host, to_dev

pytestmark = pytest.mark.gpu

STATUS_OUT_OF_MEMORY = 4
STATUS_CANCELLED = 10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_10094_gb300 import build

    build.build()
    import paper_2410_10094_gb300 as stc

    stc.load()


@pytest.mark.parametrize("probe", [1, 4, 8])
@pytest.mark.parametrize("shrink", [0, 8])
def test_undersized_global_table_is_retried(shrink, probe):
    rng = W.rng_for(9500)
    X = W.uniform_coo(rng, (30, 20, 40), 60_000)
    Y = W.uniform_coo(rng, (40, 25), 3_000)
    p = W.Problem(X, Y, (2,), (0,))
    ref = oracle.contract(p.X, p.Y, p.cx, p.cy)
    res = gpu_contract(p, strategy=1, table_shrink=shrink, probe=probe)
    c, v = result_host(res)
    assert_matches_oracle(c, v, ref)
    # A table with fewer slots than distinct output keys must overflow and be retried once (a
    # small one: every product whose key is missing probes the whole table before it gives up).
    first = max(64, res.stats.table_slots >> shrink)
    assert res.stats.retries == (1 if first < ref.nnz else 0)
    assert res.stats.retries == (1 if shrink else 0)


def test_budget_smaller_than_one_call():
    import paper_2410_10094_gb300 as stc

    rng = W.rng_for(9510)
    p = W.Problem(W.uniform_coo(rng, (64, 64, 64), 200_000), W.uniform_coo(rng, (64, 64, 64), 200_000), (2,), (0,))
    _, need = stc.count(to_dev(p.X), to_dev(p.Y), p.cx, p.cy)
    ctx = stc.Context(0, mem_budget_bytes=need // 4)
    try:
        with pytest.raises(stc.StcError) as e:
            stc.contract(to_dev(p.X), to_dev(p.Y), p.cx, p.cy, ctx=ctx)
        assert e.value.status == STATUS_OUT_OF_MEMORY
        assert ctx.stats() == (0, 0)  # the failed call released what it had taken
        small = W.Problem(W.uniform_coo(rng, (16, 8), 300), W.uniform_coo(rng, (8, 16), 300), (1,), (0,))
        r = stc.contract(to_dev(small.X), to_dev(small.Y), small.cx, small.cy, ctx=ctx)
        c, v = result_host(r)
        assert_matches_oracle(c, v, oracle.contract(small.X, small.Y, small.cx, small.cy))
        del r
    finally:
        import gc

        gc.collect()
        ctx.close()


def bounded():
    """One contraction for each way that the counted bound is put together."""
    rng = W.rng_for(9515)
    yield "one table of values", W.Problem(W.uniform_coo(rng, (2_000_000, 40), 30_000), W.uniform_coo(rng, (40, 90_000), 4_000), (1,), (0,))
    yield "a small output space", W.Problem(W.uniform_coo(rng, (300, 40), 30_000), W.uniform_coo(rng, (40, 200), 4_000), (1,), (0,))
    yield "a tiny output space", W.Problem(W.uniform_coo(rng, (3, 4), 9), W.uniform_coo(rng, (4, 2), 6), (1,), (0,))
    yield "streamed groups", W.Problem(W.uniform_coo(rng, (64, 64, 64), 20_000), W.uniform_coo(rng, (64, 80, 90), 20_000), (2,), (0,))
    yield "several segments", W.Problem(W.uniform_coo(rng, (500, 50), 3_000), W.uniform_coo(rng, (50, 300_000), 90_000), (1,), (0,))
    yield "small groups", W.Problem(W.uniform_coo(rng, (30_000, 90), 60_000), W.uniform_coo(rng, (90, 50_000), 3_000), (1,), (0,))
    yield "numbered keys", W.Problem(W.uniform_coo(rng, (2_000, 1 << 24), 60_000), W.uniform_coo(rng, (1 << 24, 3_000), 50_000), (1,), (0,))
    yield "few survivors", W.Problem(W.uniform_coo(rng, (5_000, 300_000), 100_000), W.uniform_coo(rng, (300_000, 2_000), 30_000), (1,), (0,))
    yield "rows", W.Problem(W.uniform_coo(rng, (500, 20), 9_000), W.uniform_coo(rng, (20, 30), 30_000), (1,), (0,))
    yield "nothing in common", W.Problem(W.uniform_coo(rng, (5_000_000, 40), 3_000), W.uniform_coo(rng, (40, 5_000_000), 0), (1,), (0,))


@pytest.mark.parametrize("p", [pytest.param(p, id=n.replace(" ", "_")) for n, p in bounded()])
def test_counted_bytes_are_enough(p):
    """A context whose budget is the bound of stc_count runs the call, again and again."""
    import gc

    import paper_2410_10094_gb300 as stc

    dev = to_dev(p.X), to_dev(p.Y), p.cx, p.cy
    wide = stc.Context(0, mem_budget_bytes=8 << 30)
    P, need = stc.count(*dev, ctx=wide)
    wide.close()
    ctx = stc.Context(0, mem_budget_bytes=need)
    for _ in range(2):
        r = stc.contract(*dev, ctx=ctx)
        assert r.stats.products == P
        c, v = result_host(r)
        assert_matches_oracle(c, v, oracle.contract(p.X, p.Y, p.cx, p.cy))
        del r
        gc.collect()
    ctx.close()


def test_server_cancel_queued_request():
    import paper_2410_10094_gb300 as stc

    rng = W.rng_for(9520)
    probs = [W.served_large(rng, nnz=300_000, n=128) for _ in range(12)]
    dev = [(to_dev(p.X), to_dev(p.Y), p.cx, p.cy) for p in probs]
    # A budget of one byte admits one request at a time, so the later ones wait in the queue.
    srv = stc.Server(mem_budget_bytes=1)
    try:
        tickets = [srv.submit(*d) for d in dev]
        cancelled = {t for t in reversed(tickets[-4:]) if srv.cancel(t)}
        assert cancelled, "no queued request to cancel"
        for t, p in zip(tickets, probs):
            if t in cancelled:
                with pytest.raises(stc.StcError) as e:
                    srv.wait(t)
                assert e.value.status == STATUS_CANCELLED
            else:
                r, _ = srv.wait(t, timeout_ms=600_000)
                assert r.stats.products == oracle.group_bounds(p.X, p.Y, p.cx, p.cy).total
                del r
        t = srv.submit(*dev[1])  # the server keeps serving after the cancellations
        r, _ = srv.wait(t, timeout_ms=600_000)
        assert r.stats.products == oracle.group_bounds(probs[1].X, probs[1].Y, probs[1].cx, probs[1].cy).total
    finally:
        srv.close()
