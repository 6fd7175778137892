"""Alignment paths when the packed recording sweeps' storage cannot be had: whatever
limit lets the general sweep run every extension lets the call run, whether
the packed storage is refused or, granted, leaves no room for the general sweep
of the rest.  The codes are those of a call without a limit."""
import numpy as np
import pytest

from paper_2002_05200_gb300 import logan, synth

pytestmark = pytest.mark.gpu

SLACK = 48  # MiB: the pool's granularity and a few words per extension


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    c.set_option(logan.OPT_MIGRATION_MB, 0)
    c.set_option(logan.OPT_TIMING, 1)
    yield c
    c.close()


def run(ctx, dev, b, limit):
    """The codes and the code words, None when the limit is too small."""
    ctx.set_option(logan.OPT_SCRATCH_MB, limit)
    A, B, S, Xs = dev
    try:
        codes, start, count = ctx.traceback(A, B, S, b.match, b.mismatch, b.gap, b.X, Xs)
    except logan.LoganError as e:
        assert e.code == logan.ENOMEM
        return None
    keep = np.repeat(start.cpu().numpy(), count.cpu().numpy())
    at = keep + np.concatenate([np.arange(n) for n in count.cpu().numpy()])
    return (codes.cpu().numpy()[at], count.cpu().numpy()), ctx.traceback_stats()["code_words"]


@pytest.mark.parametrize("kind,ring_cap", [("refused", 12), ("no room for the rest", 16)])
def test_general_sweep_takes_all(ctx, kind, ring_cap):
    n = 1000 if kind == "refused" else 600
    b = synth.lognormal_batch(n_pairs=n, median=10000, lo=8000, hi=12000, related_frac=1.0, seed=3, X=15)
    if kind != "refused":  # two pairs past the packed sweeps' X
        b.Xs = np.full(n, 15, np.int32)
        b.Xs[:2] = 1500
    dev = logan.batch_to_device(b, packed2bit=True)
    ctx.set_option(logan.OPT_RING_CAP, ring_cap)
    want, packed_words = run(ctx, dev, b, 0)
    # the smallest limit at which the general sweep alone runs
    ctx.set_option(logan.OPT_PACKED16, 0)
    _, general_words = run(ctx, dev, b, 0)
    assert general_words < packed_words
    lo, hi = 0, 8192
    while hi - lo > 16:
        mid = (lo + hi) // 2
        if run(ctx, dev, b, mid) is None:
            lo = mid
        else:
            hi = mid
    assert lo > 0
    ctx.set_option(logan.OPT_PACKED16, 1)
    words = []
    for limit in range(hi + SLACK, hi + SLACK + 800, 40):  # to where the packed sweeps have room
        got = run(ctx, dev, b, limit)
        assert got is not None, f"out of memory at {limit} MiB"
        assert all(np.array_equal(g, w) for g, w in zip(got[0], want)), limit
        words.append(got[1])
    assert words[0] == general_words and words[-1] == packed_words
    assert run(ctx, dev, b, lo // 2) is None
