"""The CSR transpose at the edges of its tiles and digits: bit-exact against the oracle's counting sort."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [1, 31, 4095, 4096, 4097, 12_289, 70_001])
@pytest.mark.parametrize("k", [1, 2, 128, 129, 256, 257, 16_384, 16_385, 70_000, 1 << 21])
def test_tile_and_digit_edges(gpu_lib, nnz, k):
    """Rows of every kind in one matrix: leading, inner and trailing runs of empty rows, short rows, and one that
    holds half of the nonzeros; columns repeat."""
    import torch

    rng = np.random.default_rng(nnz + k)
    cuts = np.sort(rng.integers(0, nnz // 2 + 1, 500))
    cuts[100:200] = cuts[100]
    rp = np.concatenate([[0, 0, 0], cuts, [nnz, nnz, nnz]]).astype(np.int32)
    ci = rng.integers(0, k, nnz).astype(np.int32)
    if nnz > 4000:
        ci[1000:3500] = k - 1  # a column that fills most of a tile
    rpt, cit, perm = gpu_lib.csr_transpose(*(torch.from_numpy(x).cuda() for x in (rp, ci)), k)
    ref = oracle.csr_transpose(rp, ci, k)
    for got, want in zip((rpt, cit, perm), ref):
        assert np.array_equal(got.cpu().numpy(), want)


def sparse_rows(gap, m=300_000):
    """Nonzeros in the first and the last few rows and `gap` empty rows between two of one tile."""
    lens = np.concatenate([np.full(900, 3), np.zeros(gap), [1, 0, 4], np.zeros(m - 1003), np.full(100, 20)])
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


@pytest.mark.parametrize("gap", [4000, 8100, 8192, 8193, 3_000_000])
def test_long_runs_of_empty_rows(gpu_lib, gap):
    import torch

    rp = sparse_rows(gap)
    ci = np.random.default_rng(gap).integers(0, 5000, rp[-1]).astype(np.int32)
    got = gpu_lib.csr_transpose(*(torch.from_numpy(x).cuda() for x in (rp, ci)), 5000)
    for x, want in zip(got, oracle.csr_transpose(rp, ci, 5000)):
        assert np.array_equal(x.cpu().numpy(), want)


def test_work_does_not_grow_with_the_empty_rows(gpu_lib):
    """20M empty rows between two nonzeros: the few kernels of a transpose take well below a millisecond, one CTA's
    walk over the rows tens of them."""
    import torch

    rp = torch.from_numpy(sparse_rows(20_000_000)).cuda()
    ci = torch.randint(5000, (int(rp[-1]),), device="cuda").int()
    times = []
    for _ in range(5):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        gpu_lib.csr_transpose(rp, ci, 5000)
        t1.record()
        t1.synchronize()
        times.append(t0.elapsed_time(t1))
    assert min(times) < 5.0, times
