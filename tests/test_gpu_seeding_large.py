"""Overlap seeding of more than 2^28 occurrences in short reads: the table that
finds an occurrence's read has an entry per occurrence there, more than one
grid's threads.  Random reads of 34 bases with 4 k-mers each (2e15 pairs against
4^34 reads: none alike by chance), a thousand of them twice, the first ones
again as the last ones: those are the candidates."""
import pytest

from paper_2002_05200_gb300 import logan

pytestmark = pytest.mark.gpu


def test_more_cells_than_a_grid_has_threads():
    import torch
    n, length, k, twice = (1 << 26) + (1 << 18) + 7, 34, 31, 1000
    assert n * (length - k + 1) > 1 << 28
    g = torch.Generator(device="cuda").manual_seed(1)
    words = torch.randint(-2**31, 2**31, ((n * length + 15) // 16 + 1,), dtype=torch.int64,
                          device="cuda", generator=g).to(torch.int32)
    off = torch.arange(n, dtype=torch.int64, device="cuda") * length
    off[n - twice:] = off[:twice].flip(0)
    pool = logan.DevicePool(words, off, torch.full((n,), length, dtype=torch.int32, device="cuda"),
                            True, n * length)
    ctx = logan.Context(0)
    try:
        got = ctx.overlap_candidates(pool, k, 2, 8, 4).cpu()
    finally:
        ctx.close()
    a = torch.arange(twice, dtype=torch.int32)
    want = torch.stack([a, n - 1 - a, *(torch.full_like(a, v) for v in (0, 2, 2, 4))], dim=1)
    assert torch.equal(got, want)
