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
