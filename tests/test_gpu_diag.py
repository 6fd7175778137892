"""The packed linear kernel in diagonal coordinates: its latency forms at the
batch sizes where the extensions per warp change, the split of a level's
queue into long and other items, the widest X and steepest scores that still
run packed, and gap schemes on both sides of its one-multiply substitution.
Results are integers: every field equals the oracle's."""
import pytest

from paper_2002_05200_gb300 import logan, synth
from tests.gpu_common import assert_same, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_pairs", [1, 304, 305, 608, 609, 2432, 2433])
def test_latency_units_by_batch_size(ctx, n_pairs):
    # 2 n items: one extension per warp up to 4 per SM (608 on 152 SMs), two up
    # to 8, four up to 32, then the several-to-a-warp forms
    b = synth.uniform_pairs(n_pairs=n_pairs, length=150, X=30, seed=n_pairs)
    assert_same(run_gpu(ctx, b), run_oracle(b), f"{n_pairs} pairs")


@pytest.mark.parametrize("long_item", [0, 1500, 6000, -1])
@pytest.mark.parametrize("X", [10, 30, 90, 250, 600])
def test_long_items_beside_the_rest(ctx, X, long_item):
    # levels 0-4 by X; items on both sides of the length that sends them to
    # the latency form, bands that escalate with and without records
    b = synth.lognormal_batch(n_pairs=90, median=3000, lo=300, hi=9000, seed=X, X=X)
    ref = run_oracle(b)
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    for mig in (64, 0):
        ctx.set_option(logan.OPT_MIGRATION_MB, mig)
        assert_same(run_gpu(ctx, b, packed2bit=True), ref, f"X {X}, long {long_item}, records {mig}")


@pytest.mark.parametrize("scheme", [
    (1, -1, -1, 900), (1, -1, -1, 1000),   # packed with X near its bound, and past it
    (2, -2, -2, 150), (1, -5, -4, 60),     # bonus = 2 base, but a match of 2; base 3
    (5, -4, -3, 120), (1, 0, -2, 40), (1, 1, -1, 20), (0, -1, -1, 25), (-1, -1, 0, 9),
    (40, -40, -40, 200), (90, -90, -90, 300)])
@pytest.mark.parametrize("long_item", [0, -1])
def test_scoring_schemes(ctx, scheme, long_item):
    match, mismatch, gap, X = scheme
    b = synth.lognormal_batch(n_pairs=60, median=1200, lo=100, hi=3000, related_frac=0.9, seed=7, X=X)
    b.match, b.mismatch, b.gap = match, mismatch, gap
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    assert_same(run_gpu(ctx, b, packed2bit=True), run_oracle(b), f"{scheme}")
