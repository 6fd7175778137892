"""Band-state records of the narrow levels: a 64 MiB pool holds the record of every
band that outgrows level 0 or 1 in a batch of 80,000 extensions, so that each
resumes (its cells at the narrow level count) and none restarts."""
import pytest

from paper_2002_05200_gb300 import logan, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [0, 1])
def test_records_for_a_large_batch(level):
    import torch
    times = 50
    b = synth.uniform_pairs(n_pairs=1000, length=900, X=100, seed=4)
    A, B, S, _ = logan.batch_to_device(b, packed2bit=True)
    ctx = logan.Context(0)
    try:
        ctx.set_option(logan.OPT_FORCE_LEVEL, level)
        ctx.set_option(logan.OPT_LONG_ITEM, -1)  # the several-to-a-warp forms in both batches
        ctx.set_option(logan.OPT_TIMING, 1)
        one = ctx.extend(A, B, S, b.match, b.mismatch, b.gap, b.X)
        st1 = ctx.last_stats()
        many = ctx.extend(A, B, S.repeat(times, 1), b.match, b.mismatch, b.gap, b.X)
        st = ctx.last_stats()
    finally:
        ctx.close()
    assert st["packed_levels"] & 7 == 7
    assert torch.equal(many, one.repeat(times, 1))
    moved = st["items"][level + 1]
    assert moved == times * st1["items"][level + 1] and moved > 75000
    assert st["cells"][level] == times * st1["cells"][level]
