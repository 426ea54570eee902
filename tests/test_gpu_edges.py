"""Layouts and values at the edges of the merge, row-split and SDDMM kernels: 16-bit storage and results at every
unaligned width, the semirings in several chunks, and a first row of B that holds infinities and NaN, which the kernels
gather for slots past a tile's or run's last nonzero and for lanes past the last column, and must drop.

Small integers make every sum exact in float32, and exact in 16-bit results too where it stays below 256; larger sums
are compared after one rounding to the result type."""
import numpy as np
import pytest

import oracle
from spmm_cases import csr_arrays
from test_gpu_merge import edge_lengths

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 34, 66, 100, 127, 130, 257])
@pytest.mark.parametrize("pad", [0, 1, 3])
@pytest.mark.parametrize("storage,result", [("bfloat16", "bfloat16"), ("bfloat16", "float32"), ("float16", "float16")])
@pytest.mark.parametrize("alg", ["row_split", "merge"])
def test_16bit_unaligned_layouts(gpu_lib, n, pad, storage, result, alg):
    import torch

    dt, ct = getattr(torch, storage), getattr(torch, result)
    rng = np.random.default_rng(n + pad)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 11, int_vals=True)
    B = rng.integers(-4, 5, size=(7000, n + pad)).astype(np.float32)
    ref = torch.from_numpy(oracle.spmm(rp, ci, v, np.ascontiguousarray(B[:, :n])).astype(np.float32)).to(ct)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    for hint in (0, 6000):  # the longest row unknown, and known to be what the call waits for
        out = torch.full((len(rp) - 1, n + pad), 7.0, device="cuda", dtype=ct)
        gpu_lib.spmm(d_rp, d_ci, d_v.to(dt), d_B.to(dt)[:, :n], alg=alg, out=out[:, :n], nnz=int(rp[-1]),
                     tuning=dict(max_row_len=hint))
        assert torch.equal(out[:, :n].cpu(), ref)
        assert torch.all(out[:, n:] == 7.0)


@pytest.mark.parametrize("semiring", ["min_plus", "max_plus", "max_times"])
@pytest.mark.parametrize("n", [34, 47, 66, 100, 127, 130, 257])
def test_semirings_in_chunks(gpu_lib, semiring, n):
    """Chunks of one and of two elements, one to four of them."""
    import torch

    rng = np.random.default_rng(n)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 12)
    B = rng.standard_normal((7000, n)).astype(np.float32)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    C = gpu_lib.semiring_spmm(d_rp, d_ci, d_v, d_B, semiring, alg="merge", nnz=int(rp[-1]))
    assert np.array_equal(C.cpu().numpy(), oracle.spmm_semiring(rp, ci, v, B, semiring).astype(np.float32))


@pytest.mark.parametrize("n", [3, 5, 8, 13, 16, 20, 31, 32, 47, 64, 72, 100, 128, 130, 196, 256, 260])
@pytest.mark.parametrize("storage", ["float32", "bfloat16"])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_an_unused_first_row_stays_out(gpu_lib, n, storage, value):
    """No nonzero is in column 0, whose row of B is not finite."""
    import torch

    dt = getattr(torch, storage)
    rng = np.random.default_rng(n)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 13, int_vals=True)
    ci = np.maximum(ci, 1)
    B = rng.integers(-4, 5, size=(7000, n)).astype(np.float32)
    dC = rng.integers(-3, 4, size=(len(rp) - 1, n)).astype(np.float32)
    d_rp, d_ci, d_v, d_B, d_dC = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B, dC))
    d_v, d_B, d_dC = d_v.to(dt), d_B.to(dt), d_dC.to(dt)
    d_B[0] = value
    ref = oracle.spmm(rp, ci, v, B).astype(np.float32)
    for alg in ("merge", "row_split", "hybrid"):
        C = gpu_lib.spmm(d_rp, d_ci, d_v, d_B, alg=alg, out_dtype=torch.float32, nnz=int(rp[-1]))
        assert np.array_equal(C.cpu().numpy(), ref), alg
    out = gpu_lib.sddmm(d_rp, d_ci, d_dC, d_B, out_dtype=torch.float32)
    assert np.array_equal(out.cpu().numpy(), oracle.sddmm(rp, ci, dC, B).astype(np.float32))
