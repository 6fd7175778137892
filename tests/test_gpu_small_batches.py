"""Small batches, whose extensions all take latency forms: on both sides of every
batch size where the extensions per warp change, at levels 0 to 3, for the
one-multiply substitution and the general one (whose narrow levels hold half
the window: bands that outgrow it with and without records).  Results are
integers: every field equals the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2002_05200_gb300 import logan, synth
from tests.gpu_common import assert_same, run_gpu, run_oracle
from tests.test_gpu_matrix import run_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("per_sm", [4, 8, 12, 16, 24])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("scheme", [(1, -1, -1), (2, -3, -5), (2, -2, -2)])
def test_extensions_per_warp(ctx, scheme, per_sm, more):
    n = per_sm * sms() // 2 + more
    b = synth.lognormal_batch(n_pairs=n, median=200, lo=20, hi=700, related_frac=0.8, seed=n, X=50)
    b.match, b.mismatch, b.gap = scheme
    b.Xs = np.array([8, 15, 30, 90, 250], np.int32)[np.arange(n) % 5]
    ref = run_oracle(b)
    for mig in (64, 0):
        ctx.set_option(logan.OPT_MIGRATION_MB, mig)
        assert_same(run_gpu(ctx, b, packed2bit=True), ref, f"{scheme}, {n} pairs, records {mig}")


@pytest.mark.parametrize("n", [1, 8, 9])
@pytest.mark.parametrize("scheme", [(1, -1, -1), (2, -3, -5)])
def test_tiny_batches_of_wide_bands(ctx, scheme, n):
    # level 6 in a block or in one warp, its records to and from the others
    b = synth.lognormal_batch(n_pairs=n, median=6000, lo=2000, hi=12_000, related_frac=0.5, seed=n, X=50)
    b.match, b.mismatch, b.gap = scheme
    for X, level in ((800, -1), (200, 5)):
        b.X = X
        ctx.set_option(logan.OPT_FORCE_LEVEL, level)
        assert_same(run_gpu(ctx, b, packed2bit=True), run_oracle(b), f"{scheme}, {n} pairs, X {X}")


@pytest.mark.parametrize("X,ge", [(219, -1), (220, -1), (439, -2), (440, -2)])
@pytest.mark.parametrize("more", [0, 1])
def test_few_proteins_with_wide_bands(ctx, X, ge, more):
    # the matrix call's windows in 32 bits: few extensions whose bands are wide
    n = 8 * sms() + more
    b = synth.protein_pairs(n, lo=20, hi=400, seed=X)
    b.X = X
    got = run_matrix(ctx, b, synth.BLOSUM62, -11, ge)
    few = more == 0 and X >= 220 * -ge
    assert (ctx.get_option(logan.OPT_MATRIX_PACKED) == 0) == few
    assert_same(got, oracle.run_batch_matrix(b, synth.BLOSUM62, -11, ge)[0], f"{n} pairs, X {X}")
