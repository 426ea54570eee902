"""GPU parity of the merge-path compute kernel over its lane layouts: every access width and
alignment, tile and batch edges, empty rows and rows that cross warps and CTAs.

Small integers make every product and partial sum exact in float32, so the result must equal the
oracle's whatever the summation order."""
import numpy as np
import pytest

import oracle
from spmm_cases import csr_arrays

pytestmark = pytest.mark.gpu


def edge_lengths(rng):
    """Row lengths at the edges of a batch of 32 nonzeros, runs of empty rows, short rows, and rows that span
    several warps' tiles and several CTAs."""
    parts = [np.arange(0, 70), np.zeros(200), np.ones(90), [31, 32, 33, 0, 0, 32, 64, 63, 65, 0], rng.integers(0, 4, 700),
             [6000], np.zeros(40), rng.integers(0, 40, 300), [0, 1500, 0, 0, 511, 512, 513], np.zeros(3)]
    return np.concatenate(parts).astype(np.int64)


@pytest.mark.parametrize("n", [2, 3, 5, 8, 13, 16, 20, 31, 32, 33, 34, 47, 64, 66, 96, 100, 127, 128, 130, 257])
@pytest.mark.parametrize("pad", [0, 1, 2, 4])
def test_layouts_are_bitwise(gpu_lib, n, pad):
    """pad: ldb - n and ldc - n, which with n decides the aligned access width."""
    import torch

    rng = np.random.default_rng(100 * n + pad)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 3, int_vals=True)
    B = rng.integers(-4, 5, size=(7000, n + pad)).astype(np.float32)
    ref = oracle.spmm(rp, ci, v, np.ascontiguousarray(B[:, :n])).astype(np.float32)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    for tuning in (None, dict(items_per_subwarp=4), dict(items_per_subwarp=13, column_slabs=2)):
        out = torch.full((len(rp) - 1, n + pad), 7.0, device="cuda")
        gpu_lib.spmm(d_rp, d_ci, d_v, d_B[:, :n], alg="merge", out=out[:, :n], nnz=int(rp[-1]), tuning=tuning)
        got = out.cpu().numpy()
        assert np.array_equal(got[:, :n], ref), tuning
        assert np.all(got[:, n:] == 7.0)  # padding untouched


@pytest.mark.parametrize("storage", ["bfloat16", "float16"])
@pytest.mark.parametrize("n", [4, 7, 8, 24, 33, 40, 64, 100, 128, 136, 256])
def test_16bit_layouts_are_bitwise(gpu_lib, storage, n):
    import torch

    rng = np.random.default_rng(n)
    rp, ci, v = csr_arrays(edge_lengths(rng), 7000, 5, int_vals=True)
    B = rng.integers(-4, 5, size=(7000, n)).astype(np.float32)
    dt = getattr(torch, storage)
    d_rp, d_ci = (torch.from_numpy(x).cuda() for x in (rp, ci))
    C = gpu_lib.spmm(d_rp, d_ci, torch.from_numpy(v).cuda().to(dt), torch.from_numpy(B).cuda().to(dt), alg="merge",
                     out_dtype=torch.float32, nnz=int(rp[-1]))
    assert np.array_equal(C.cpu().numpy(), oracle.spmm(rp, ci, v, B).astype(np.float32))


@pytest.mark.parametrize("n", [1, 8, 32, 100])
def test_auto_gb300_runs_merge_on_small_type1_matrices(gpu_lib, n):
    """Where the GB300 rule names the hybrid for a skewed matrix of few nonzeros, the call runs merge: the same
    bits as a forced merge."""
    import torch

    rng = np.random.default_rng(n)
    rp, ci, v = csr_arrays(np.concatenate([rng.integers(0, 9, 4000), [3000]]), 5000, 4)
    d_rp, d_ci, d_v = (torch.from_numpy(x).cuda() for x in (rp, ci, v))
    B = torch.randn(5000, n, device="cuda")
    nnz = int(rp[-1])
    auto = gpu_lib.spmm(d_rp, d_ci, d_v, B, alg="auto_gb300", nnz=nnz)
    assert torch.equal(auto, gpu_lib.spmm(d_rp, d_ci, d_v, B, alg="merge", nnz=nnz))


def test_noalloc_keeps_accepting_wide_products(gpu_lib):
    """With full tiles the partial sums of this product fit the fixed scratch of 16 MiB twice over; tiles made
    smaller to fill the GPU must not take more."""
    import torch

    rng = np.random.default_rng(1)
    m, k, n = 20_000, 500, 2048
    rp, ci, v = csr_arrays(np.full(m, 50), k, 8, int_vals=True)
    d_rp, d_ci, d_v = (torch.from_numpy(x).cuda() for x in (rp, ci, v))
    B = torch.from_numpy(rng.integers(-4, 5, size=(k, n)).astype(np.float32)).cuda()
    C = torch.empty(m, n, device="cuda")
    st = gpu_lib.spmm_csr_noalloc(m, k, n, int(rp[-1]), d_rp.data_ptr(), d_ci.data_ptr(), d_v.data_ptr(), gpu_lib.F32,
                                  B.data_ptr(), gpu_lib.F32, n, C.data_ptr(), gpu_lib.F32, n, gpu_lib.ALG_MERGE, None,
                                  None, torch.cuda.current_stream().cuda_stream)
    assert st == gpu_lib.OK, gpu_lib.spmm_status_string(st)
    assert torch.equal(C, gpu_lib.spmm(d_rp, d_ci, d_v, B, alg="row_split", nnz=int(rp[-1])))


@pytest.mark.parametrize("n", [5, 6, 7])
@pytest.mark.parametrize("mean", [1, 3, 4])
def test_unaligned_short_rows_are_bitwise(gpu_lib, n, mean):
    """Both sides of the mean row length at which rows of up to 8 unaligned columns change their kernel."""
    import torch

    rng = np.random.default_rng(10 * n + mean)
    rp, ci, v = csr_arrays(np.concatenate([rng.poisson(mean, 20_000), np.zeros(70), [900], np.zeros(3)]).astype(np.int64),
                           5000, 6, int_vals=True)
    B = rng.integers(-4, 5, size=(5000, n)).astype(np.float32)
    ref = oracle.spmm(rp, ci, v, B).astype(np.float32)
    d_rp, d_ci, d_v, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, v, B))
    for tuning in (None, dict(column_slabs=2), dict(items_per_subwarp=5)):
        C = gpu_lib.spmm(d_rp, d_ci, d_v, d_B, alg="merge", nnz=int(rp[-1]), tuning=tuning)
        assert np.array_equal(C.cpu().numpy(), ref), tuning


@pytest.mark.parametrize("n,storage,mean,m", [(12, "float32", 1, 5000), (36, "float32", 1, 5000), (48, "float32", 1, 5000),
                                              (64, "float32", 1, 9000), (64, "float32", 2, 600_000), (64, "bfloat16", 7, 5000),
                                              (40, "float16", 9, 5000), (64, "bfloat16", 12, 250_000), (72, "bfloat16", 1, 5000),
                                              (128, "bfloat16", 1, 5000), (128, "bfloat16", 2, 5000), (2, "float32", 15, 60_000),
                                              (4, "float32", 60, 14_000)])
def test_the_lines_of_the_narrow_kernel(gpu_lib, n, storage, mean, m):
    """Mean row lengths at which rows of 2 to 16 lanes change their kernel, with one long row and empty ones."""
    import torch

    dt = getattr(torch, storage)
    g = torch.Generator(device="cuda").manual_seed(n + m)
    lens = torch.full((m,), mean, dtype=torch.int64, device="cuda")
    if mean > 1:
        lens[::50], lens[7], lens[100:180], lens[-3:] = 2 * mean, 700, 0, 0
    rp = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    nnz = int(rp[-1])
    ci = torch.randint(3000, (nnz,), device="cuda", generator=g).int()
    v = torch.randint(-2, 3, (nnz,), device="cuda", generator=g).to(dt)
    B = torch.randint(-3, 4, (3000, n), device="cuda", generator=g).to(dt)
    C = gpu_lib.spmm(rp, ci, v, B, alg="merge", out_dtype=torch.float32, nnz=nnz)
    assert torch.equal(C, gpu_lib.spmm(rp, ci, v, B, alg="row_split", out_dtype=torch.float32, nnz=nnz))
