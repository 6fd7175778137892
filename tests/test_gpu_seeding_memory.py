"""What overlap_candidates holds on to: the result's own size (twice it or 4 MiB
more at most), and a first buffer that does not grow with the read set without end."""
import numpy as np
import pytest

from paper_2002_05200_gb300 import logan
from tests.test_gpu_seeding import device_pool, genome_reads

pytestmark = pytest.mark.gpu

ROW = 24  # bytes of a candidate


@pytest.fixture()
def ctx():
    c = logan.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_reads,glen", [(3, 300000), (120, 3000), (20000, 1000000), (20000, 10000000)])
def test_result_storage(ctx, n_reads, glen):
    reads = genome_reads(np.random.default_rng(n_reads), n_reads, glen)
    got = ctx.overlap_candidates(device_pool(reads), 15, 2, 8, 1)
    assert got.is_contiguous() and got.shape[1] == 6
    held, n = got.untyped_storage().nbytes(), got.shape[0]
    assert held <= max(2 * ROW * n, ROW * n + (4 << 20))


def test_first_buffer_of_a_large_read_set(ctx):
    import torch
    n = 50_000_000  # reads without k-mers
    pool = logan.DevicePool(torch.zeros(16, dtype=torch.int32, device="cuda"),
                            torch.zeros(n, dtype=torch.int64, device="cuda"),
                            torch.zeros(n, dtype=torch.int32, device="cuda"), True, 0)
    before = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    got = ctx.overlap_candidates(pool, 17, 2, 8, 1)
    assert got.shape == (0, 6)
    assert torch.cuda.max_memory_allocated() - before <= 2 << 30
