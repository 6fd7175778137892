"""Alignment paths through the packed recording sweeps: every window class (128
to 2048 rows) and the round that takes bands which left their window to a
wider one, gap schemes on both sides of the one-multiply substitution, X per
pair past the packed sweeps' bound beside pairs inside it.  The run-length
codes equal the oracle's."""
import numpy as np
import pytest

from paper_2002_05200_gb300 import logan, synth
from tests.test_gpu_traceback import check, gpu_paths

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("X", [15, 60, 100, 180, 400])
def test_window_classes(ctx, X):
    # unrelated pairs under +1/-1/-1 drift to bands of about 12 X rows
    b = synth.lognormal_batch(n_pairs=30, median=2500, lo=300, hi=5000, related_frac=0.4, seed=X, X=X)
    check(b, *gpu_paths(ctx, b, packed2bit=True))


@pytest.mark.parametrize("scheme", [(2, -3, -5, 80), (1, -2, -2, 40), (3, -1, -4, 60), (1, -1, 0, 30),
                                    (60, -60, -60, 300)])
def test_schemes(ctx, scheme):
    b = synth.lognormal_batch(n_pairs=40, median=900, lo=100, hi=2000, related_frac=0.9, seed=5, X=scheme[3])
    b.match, b.mismatch, b.gap = scheme[:3]
    check(b, *gpu_paths(ctx, b, packed2bit=True))


def test_per_pair_x_past_the_bound(ctx):
    b = synth.lognormal_batch(n_pairs=40, median=700, lo=100, hi=1500, related_frac=0.8, seed=6, X=100)
    b.Xs = np.array([20, 100, 600, 900, 1500], np.int32)[np.arange(40) % 5]
    check(b, *gpu_paths(ctx, b, packed2bit=True))
