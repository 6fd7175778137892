"""Overlap seeding at the edges of its key forms: one class of 32-bit codes (k
<= 16), classes by the upper bits (17, 18), 64-bit codes (19 and more); reads
shorter than k between others; repeats, where a k-mer of one read meets
several of another and the middle hit is a tie in pos_a; more candidates
than the binding's first buffer holds.  Candidates equal the oracle's."""
import numpy as np
import pytest

from oracle import overlap_oracle as ov
from paper_2002_05200_gb300 import logan, synth

pytestmark = pytest.mark.gpu


def device_pool(reads):
    lens = np.array([len(r) for r in reads], np.uint32)
    off = np.concatenate([[0], np.cumsum(lens[:-1], dtype=np.uint64)]).astype(np.uint64)
    asc = np.frombuffer(b"".join(reads), np.uint8)
    return logan.pool_to_device(synth.pack2bit(asc), off, lens, True, asc.size)


def check(reads, k, fmin, fmax, shared):
    ctx = logan.Context(0)
    try:
        got = ctx.overlap_candidates(device_pool(reads), k, fmin, fmax, shared).cpu().numpy().view(np.uint32)
    finally:
        ctx.close()
    want = ov.candidates(reads, k, fmin, fmax, shared)
    assert got.shape[0] == want.size
    for j, f in enumerate(ov.CAND_DTYPE.names):
        assert np.array_equal(got[:, j], want[f]), f
    return want.size


def genome_reads(rng, n, glen, unit=None):
    g = rng.integers(0, 4, glen if unit is None else unit)
    g = np.resize(g, glen)  # unit: a tandem repeat
    reads = []
    for _ in range(n):
        m = int(rng.integers(0, 400))
        p = int(rng.integers(0, glen - m + 1))
        r = g[p:p + m].copy()
        e = rng.random(m) < 0.02
        r[e] = rng.integers(0, 4, int(e.sum()))
        if rng.random() < 0.5:
            r = 3 - r[::-1]
        reads.append(bytes(np.frombuffer(b"ACGT", np.uint8)[r]))
    return reads


@pytest.mark.parametrize("k", [5, 15, 16, 17, 18, 19, 31])
def test_key_forms(k):
    rng = np.random.default_rng(k)
    reads = genome_reads(rng, 120, 6000) + [b"", b"ACG", b"ACGTACGT"]
    assert check(reads, k, 2, 8, 2) > 0 or k == 5


@pytest.mark.parametrize("k,unit", [(11, 37), (17, 61), (21, 50)])
def test_ties_in_repeats(k, unit):
    rng = np.random.default_rng(unit)
    assert check(genome_reads(rng, 24, 900, unit), k, 2, 1024, 1) > 0


def test_more_candidates_than_the_first_buffer():
    # 66 copies of one read, some reverse complements: 2,145 pairs, past 32 a read
    rng = np.random.default_rng(3)
    r = bytes(np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 90)])
    rc = r[::-1].translate(bytes.maketrans(b"ACGT", b"TGCA"))
    assert check([r if i % 3 else rc for i in range(66)], 17, 2, 70, 1) > 2112
