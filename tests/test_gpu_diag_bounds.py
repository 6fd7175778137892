"""Scoring schemes at the packed linear kernels' bounds: a mismatch far below two
gaps on both sides of the bound, X at the largest value that runs packed, and
X per pair of classes that start at the highest level allowed.
Results are integers: every field, and every path, equals the oracle's."""
import numpy as np
import pytest

from paper_2002_05200_gb300 import logan, synth
from tests.gpu_common import assert_same, run_gpu, run_oracle
from tests.test_gpu_traceback import check, gpu_paths

pytestmark = pytest.mark.gpu

# (match, mismatch, gap, X): the first ones need 32 bits, the others run packed
SCHEMES = [(25, -1000, -10, 100), (100, -1000, -50, 100), (30, -1000, -20, 300),
           (60, -1000, -30, 300), (50, -1000, -10, 300), (100, -1000, -50, 300), (1000, -1000, -1, 50),
           (10, -1000, -5, 100),
           (9, -1000, -5, 100), (9, -1000, -5, 600), (1, -1000, -1, 100), (1, -1000, 0, 40),
           (2, -800, -10, 300), (1, -1, -1, 1013)]


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


def batch(scheme, n_pairs=60):
    match, mismatch, gap, X = scheme
    b = synth.lognormal_batch(n_pairs=n_pairs, median=1200, lo=100, hi=3000, related_frac=0.9,
                              seed=11, X=X)
    b.match, b.mismatch, b.gap = match, mismatch, gap
    return b


@pytest.mark.parametrize("scheme", SCHEMES)
@pytest.mark.parametrize("long_item", [0, -1])
def test_extend(ctx, scheme, long_item):
    b = batch(scheme)
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    assert_same(run_gpu(ctx, b, packed2bit=True), run_oracle(b), f"{scheme}")


@pytest.mark.parametrize("scheme", SCHEMES)
def test_paths(ctx, scheme):
    b = batch(scheme, n_pairs=40)
    check(b, *gpu_paths(ctx, b, packed2bit=True))


@pytest.mark.parametrize("max_level", [0, 1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("long_item", [0, -1])
def test_x_classes_above_the_highest_level(ctx, max_level, long_item):
    # per-pair X: the classes that would start above the highest level start at
    # it, so its bound has to hold for their X too
    b = batch((1, -1, -1, 100), n_pairs=72)
    b.Xs = np.array([10, 60, 140, 400, 1200, 2000], np.int32)[np.arange(72) % 6]
    ctx.set_option(logan.OPT_MAX_LEVEL, max_level)
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    assert_same(run_gpu(ctx, b, packed2bit=True), run_oracle(b), f"level {max_level}, long {long_item}")
