"""The workspace of a product: one buffer sized for the largest pattern serves every smaller one, and the fixed
scratch takes every product whose full merge tiles fit."""
import random

import pytest

import paper_1803_08601_gb300 as pkg


@pytest.mark.parametrize("alg", [pkg.ALG_MERGE, pkg.ALG_ROW_SPLIT_HYBRID])
@pytest.mark.parametrize("tuning", [None, dict(items_per_subwarp=5), dict(items_per_subwarp=700), dict(lanes_per_row=8),
                                    dict(column_slabs=3)])
@pytest.mark.parametrize("dtype", [pkg.F32, pkg.BF16])
def test_size_does_not_fall_as_the_pattern_grows(alg, tuning, dtype):
    pkg.build()
    rng = random.Random(5)

    def size(m, n, nnz):
        return pkg.spmm_csr_workspace_size(m, m, n, nnz, alg, dtype, tuning)

    assert size(4478, 64, 17_135) <= size(4478, 64, 18_218)  # either side of 4 nonzeros per row
    assert size(1_829_694, 64, 7_180_000) <= size(1_829_694, 64, 7_510_000)
    for _ in range(3000):
        n = rng.choice([1, 2, 3, 5, 8, 13, 16, 31, 32, 47, 64, 100, 128, 256, 300, 2048])
        m, nnz = int(10 ** rng.uniform(0, 7)), int(10 ** rng.uniform(0, 8.5))
        m2 = rng.choice([m, rng.randint(1, m), m - m // 50])
        nnz2 = rng.choice([nnz, rng.randint(0, nnz), nnz - nnz // 50])
        assert size(m2, n, nnz2) <= size(m, n, nnz), (m, n, nnz, m2, nnz2)


def problem(torch, m, k, n, nnz):
    """m rows of nnz nonzeros in all; small integers: every sum is exact in float32."""
    g = torch.Generator(device="cuda").manual_seed(m)
    rp = (torch.arange(m + 1, device="cuda", dtype=torch.int64) * nnz // m).int()
    ci = torch.randint(k, (nnz,), device="cuda", generator=g).int()
    v = torch.randint(-2, 3, (nnz,), device="cuda", generator=g).float()
    return rp, ci, v, torch.randint(-4, 5, (k, n), device="cuda", generator=g).float()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [5, 16, 32, 47, 64, 128])
def test_one_buffer_serves_smaller_patterns(gpu_lib, n):
    """Down to a few nonzeros, across the sizes at which the merge changes its kernel and tiles; also a buffer
    that holds no more than full tiles with one entry each (of 2048 items, or 1024 for up to 8 lanes a row)."""
    import torch

    m, k, largest = 4478, 1000, 40_000
    ws = torch.empty(gpu_lib.workspace_size(m, k, n, largest, "merge"), dtype=torch.uint8, device="cuda")
    lanes = n if n % 4 else n // 4
    tile = 2048 if lanes > 8 else 1024
    entries = (m + largest + tile - 1) // tile
    full = sum((x + 255) // 256 * 256 for x in (8 * (entries + 1), 4 * entries, 4 * entries, 4 * n * entries, 4 * n * entries))
    for nnz in (largest, 18_218, 17_135, 9000, 300, 1):
        rp, ci, v, B = problem(torch, m, k, n, nnz)
        ref = gpu_lib.spmm(rp, ci, v, B, alg="row_split", nnz=nnz)
        assert torch.equal(gpu_lib.spmm(rp, ci, v, B, alg="merge", nnz=nnz, workspace=ws), ref), nnz
        assert torch.equal(gpu_lib.spmm(rp, ci, v, B, alg="merge", nnz=nnz, workspace=ws[:full]), ref), nnz


@pytest.mark.gpu
def test_noalloc_takes_what_full_tiles_fit(gpu_lib):
    """30,734 full tiles with one entry each take 16,320,512 of the 16,777,216 bytes."""
    import torch

    m, k, n, nnz = 358_265, 2000, 64, 62_944_710
    rp, ci, v, B = problem(torch, m, k, n, nnz)
    C = torch.empty(m, n, device="cuda")
    st = gpu_lib.spmm_csr_noalloc(m, k, n, nnz, rp.data_ptr(), ci.data_ptr(), v.data_ptr(), gpu_lib.F32, B.data_ptr(),
                                  gpu_lib.F32, n, C.data_ptr(), gpu_lib.F32, n, gpu_lib.ALG_MERGE, None, None,
                                  torch.cuda.current_stream().cuda_stream)
    assert st == gpu_lib.OK, gpu_lib.spmm_status_string(st)
    assert torch.equal(C, gpu_lib.spmm(rp, ci, v, B, alg="row_split", nnz=nnz))


@pytest.mark.gpu
def test_a_buffer_below_full_tiles_is_refused(gpu_lib):
    import torch

    rp, ci, v, B = problem(torch, 5000, 1000, 64, 60_000)
    ws = torch.empty(8192, dtype=torch.uint8, device="cuda")  # full tiles take 18 KB
    with pytest.raises(gpu_lib.SpMMError) as e:
        gpu_lib.spmm(rp, ci, v, B, alg="merge", nnz=60_000, workspace=ws)
    assert e.value.status == gpu_lib.ERR_WORKSPACE
