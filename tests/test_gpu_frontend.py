"""The input checks and the work-queue scan: a bad byte at every place of a
sequence that starts at every address modulo 16, and lengths that put items
in the first and last buckets of a queue on both sides of the long-item
length."""
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


@pytest.mark.parametrize("bad", [0, ord("N"), ord("a"), ord("U"), ord("A") | 0x80, ord("A") ^ 0x01, 255])
def test_a_bad_byte_at_every_place(ctx, bad):
    # 53 bases: 0-15 up to the boundary, two or three vectors, the rest; the
    # start moves by 5 modulo 16 from pair to pair, so 16 pairs share a place;
    # pair p has its bad byte at place p // 16 (place 53: none) of sequence A
    L, n = 53, 54 * 16
    b = synth.uniform_pairs(n_pairs=n, length=L, X=20, seed=3)
    lenA = np.full(n, L, np.uint32)
    offA = (np.arange(n, dtype=np.uint64) * L)
    pool = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(5).integers(0, 4, n * L)].copy()
    place = np.arange(n) // 16
    hit = place < L
    pool[(offA[hit] + place[hit].astype(np.uint64)).astype(np.int64)] = bad
    b.poolA, b.offA, b.lenA = pool, offA, lenA
    seeds = b.seeds.copy()
    seeds["posA"], seeds["posB"], seeds["len"] = 4, 4, 5
    seeds["idxA"] = np.arange(n)
    b.seeds = seeds
    g = run_gpu(ctx, b)
    assert np.array_equal(g["status"] != logan.OK, hit)
    assert_same(g, run_oracle(b), f"byte {bad}")


@pytest.mark.parametrize("long_item", [0, 1, 2, 40, 700, 1 << 20, -1])
def test_long_items_of_a_queue_with_every_length(ctx, long_item):
    b = synth.tiny_pairs(300, 60, seed=21)
    ctx.set_option(logan.OPT_LONG_ITEM, long_item)
    assert_same(run_gpu(ctx, b), run_oracle(b), f"tiny, long {long_item}")
    b = synth.lognormal_batch(n_pairs=60, median=500, lo=20, hi=3000, seed=22, X=60)
    assert_same(run_gpu(ctx, b, packed2bit=True), run_oracle(b), f"lengths, long {long_item}")
