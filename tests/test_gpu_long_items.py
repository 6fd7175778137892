"""Batches with more long extensions than a level's latency form takes (8 per SM,
the longest): the others run several to a warp, whole length buckets of them.
Results are integers and equal the oracle's on both sides of the limit; a
batch of only long extensions is not held back by the few warps that the
latency form has beside the other forms."""
import numpy as np
import pytest

from paper_2002_05200_gb300 import logan, synth
from tests.gpu_common import assert_same, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


def limit():
    import torch
    return 8 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("X", [10, 30, 90, 250, 600])
@pytest.mark.parametrize("more", [0, 2])
def test_one_length_at_the_limit(ctx, X, more):
    # every extension in one bucket: all fit, or none stays
    b = synth.uniform_pairs(n_pairs=(limit() + more) // 2, length=300, X=X, seed=X)
    ref = run_oracle(b)
    ctx.set_option(logan.OPT_LONG_ITEM, 200)
    assert_same(run_gpu(ctx, b), ref, f"X {X}, {b.n_pairs} pairs")


@pytest.mark.parametrize("concurrent", [0, 1])
@pytest.mark.parametrize("long_item", [1, 300, 900])
def test_the_longest_stay(ctx, long_item, concurrent):
    # X of levels 0 to 4, lengths over several buckets, items on both sides of the
    # limit at each level
    n = 3 * limit()
    b = synth.lognormal_batch(n_pairs=n, median=700, lo=50, hi=4000, related_frac=0.9, seed=2, X=100)
    b.Xs = np.array([10, 30, 90, 250, 600], np.int32)[np.arange(n) % 5]
    ref = run_oracle(b)
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    ctx.set_option(logan.OPT_CONCURRENT, concurrent)
    assert_same(run_gpu(ctx, b, packed2bit=True), ref, f"long {long_item}, concurrent {concurrent}")


def test_many_long_extensions(ctx):
    import torch
    b = synth.uniform_pairs(n_pairs=32, length=140_000, X=50, seed=5)
    A, B, S, _ = logan.batch_to_device(b, packed2bit=True)
    S = S.repeat(94, 1)

    def ms(long_item):
        ctx.set_option(logan.OPT_LONG_ITEM, long_item)
        best = 1e9
        for _ in range(4):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            ctx.extend(A, B, S, 1, -1, -1, 50)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best
    assert ms(-2) < 2 * ms(-1)


def test_requests_share_the_latency_forms(ctx):
    # more long extensions in one request than its latency forms take, then in
    # six requests together
    b = synth.uniform_pairs(n_pairs=64, length=9000, X=50, seed=8)
    ref = run_oracle(b)
    take = np.arange(700) % 64
    b.seeds = b.seeds[take]
    srv = logan.Server(ctx, 8 << 30, 8)
    try:
        for n in (1, 6):
            reqs = [logan.HostRequest(b) for _ in range(n)]
            for t in [srv.submit(r) for r in reqs]:
                assert srv.wait(t)[0] == logan.OK
            for r in reqs:
                got = r.results.numpy().view(logan.RESULT_DTYPE).reshape(-1)
                assert_same(got, ref[take], f"{n} requests")
    finally:
        srv.close()
