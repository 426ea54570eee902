"""GPU parity of the row split where rows of B are not 16-byte aligned: every chunk layout and its ragged
edges.  Small integers make every sum exact in float32."""
import numpy as np
import pytest

import oracle
from spmm_cases import csr_arrays
from test_gpu_merge import edge_lengths

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 33, 34, 47, 63, 65, 66, 100, 127, 129, 130, 257])
@pytest.mark.parametrize("pad", [0, 1, 2])
def test_layouts_are_bitwise(gpu_lib, n, pad):
    import torch

    rng = np.random.default_rng(10 * n + pad)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 6, int_vals=True)
    B = rng.integers(-4, 5, size=(7000, n + pad)).astype(np.float32)
    ref = oracle.spmm(rp, ci, v, np.ascontiguousarray(B[:, :n])).astype(np.float32)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    for tuning in (None, dict(column_slabs=2), dict(lanes_per_row=32)):
        out = torch.full((len(rp) - 1, n + pad), 7.0, device="cuda")
        gpu_lib.spmm(d_rp, d_ci, d_v, d_B[:, :n], alg="row_split", out=out[:, :n], nnz=int(rp[-1]), tuning=tuning)
        got = out.cpu().numpy()
        assert np.array_equal(got[:, :n], ref), tuning
        assert np.all(got[:, n:] == 7.0)


@pytest.mark.parametrize("semiring", ["min_plus", "max_times"])
def test_semirings(gpu_lib, semiring):
    import torch

    rng = np.random.default_rng(3)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 7)
    B = rng.standard_normal((7000, 47)).astype(np.float32)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    C = gpu_lib.semiring_spmm(d_rp, d_ci, d_v, d_B, semiring, alg="row_split", nnz=int(rp[-1]))
    assert np.array_equal(C.cpu().numpy(), oracle.spmm_semiring(rp, ci, v, B, semiring).astype(np.float32))
