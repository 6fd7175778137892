"""The packed affine and matrix windows in diagonal coordinates: every window
and both lane lengths (batches on either side of the one that fills the GPU),
gap schemes with large and zero openings, scores at the bounds, tables of 2
to 32 letters with negative and positive ranges.  Results are integers:
every field equals the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2002_05200_gb300 import logan, synth
from tests.gpu_common import assert_same
from tests.test_gpu_affine import run_affine
from tests.test_gpu_matrix import run_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_pairs", [60, 2433])  # small-batch lanes, full lanes
@pytest.mark.parametrize("scheme", [(1, -1, -2, -1, 30), (1, -1, -8, -1, 90), (2, -3, 0, -2, 150),
                                    (1, -1, -1, 0, 40), (5, -4, -20, -1, 200), (30, -30, -30, -10, 120)])
def test_affine_schemes(ctx, scheme, n_pairs):
    match, mismatch, go, ge, X = scheme
    b = synth.lognormal_batch(n_pairs=n_pairs, median=500, lo=100, hi=1200, seed=X, X=X)
    b.match, b.mismatch = match, mismatch
    assert_same(run_affine(ctx, b, go, ge, packed2bit=True), oracle.run_batch_affine(b, go, ge)[0], f"{scheme}")


@pytest.mark.parametrize("n_pairs", [50, 2433])
@pytest.mark.parametrize("K,lo,hi,go,ge,X", [(20, -4, 9, -11, -1, 60), (2, -1, 1, 0, -1, 20), (32, -9, -1, -3, 0, 15),
                                             (32, 0, 12, -20, -3, 200), (7, -90, 40, -40, -5, 100)])
def test_matrix_tables(ctx, K, lo, hi, go, ge, X, n_pairs):
    rng = np.random.default_rng(K + X)
    b = synth.protein_pairs(n_pairs=n_pairs, lo=30, hi=300, X=X, seed=K)
    b.poolA, b.poolB = b.poolA % K, b.poolB % K
    M = rng.integers(lo, hi + 1, size=(K, K)).astype(np.int32)
    M[np.arange(K), np.arange(K)] = hi
    assert_same(run_matrix(ctx, b, M, go, ge), oracle.run_batch_matrix(b, M, go, ge)[0], f"K {K}")
