"""The row split's default column slabs, once B outgrows L2.  Slabs do not
change the order of any sum, so the result equals the one-slab result bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,k,n,slabs", [
    ("float32", 200_000, 128, 2),   # 256 bytes per row fit half of L2
    ("float32", 400_000, 128, 4), ("float32", 140_000, 192, 3), ("float32", 300_000, 192, 6), ("float32", 300_000, 96, 3),
    ("float32", 300_000, 127, 4),
    ("float32", 300_000, 100, 1),   # four slabs would cover 128 columns
    ("float32", 700_000, 100, 2),   # B above twice the L2: two slabs as for ragged rows
    ("float32", 100_000, 128, 1),   # 512 bytes per row fit half of L2
    ("float32", 100_000, 256, 1),   # a pass covers 512 bytes of the 1024
    ("float32", 900_000, 32, 1),    # rows of 128 bytes
    ("bfloat16", 600_000, 128, 2), ("bfloat16", 400_000, 256, 4), ("float16", 400_000, 192, 3), ("float16", 400_000, 136, 1)])
def test_default_slabs_do_not_change_a_bit(gpu_lib, storage, k, n, slabs):
    import torch

    dt = getattr(torch, storage)
    code = gpu_lib.dtype_code(dt)
    if torch.cuda.get_device_properties(0).L2_cache_size == 0:
        pytest.skip("unknown L2 size")
    assert gpu_lib.default_column_slabs(gpu_lib.ALG_ROW_SPLIT, k, n, code) == slabs
    g = torch.Generator(device="cuda").manual_seed(n)
    lens = torch.randint(0, 40, (3001,), device="cuda", generator=g)
    rp = torch.zeros(3002, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    nnz = int(rp[-1])
    ci = torch.randint(k, (nnz,), device="cuda", generator=g).int()
    v = torch.randn(nnz, device="cuda", generator=g).to(dt)
    B = torch.randn(k, n, device="cuda", generator=g).to(dt)
    C = gpu_lib.spmm(rp, ci, v, B, alg="row_split", nnz=nnz)
    one = gpu_lib.spmm(rp, ci, v, B, alg="row_split", nnz=nnz, tuning=dict(column_slabs=1))
    assert torch.equal(C, one)
    assert np.isfinite(C.float().cpu().numpy()).all()
