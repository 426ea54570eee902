"""GPU parity of SDDMM over its lane layouts: every access width and alignment, several passes over
wide rows, row ends anywhere in a group, empty rows and rows that span many warps.

Small integers make every product and partial sum exact in float32, so float32 results must equal
the oracle's and 16-bit results its rounding."""
import numpy as np
import pytest

import oracle
from spmm_cases import csr_arrays
from test_gpu_merge import edge_lengths

pytestmark = pytest.mark.gpu

COMBOS = [("float32", "float32"), ("bfloat16", "float32"), ("bfloat16", "bfloat16"), ("float16", "float16")]


@pytest.mark.parametrize("n", [1, 3, 4, 8, 16, 31, 32, 33, 47, 64, 66, 96, 100, 127, 128, 129, 130, 192, 256, 260, 512, 640, 1024, 1040])
@pytest.mark.parametrize("storage,result", COMBOS)
def test_layouts_are_bitwise(gpu_lib, n, storage, result):
    import torch

    rng = np.random.default_rng(n)
    rp, ci, _ = csr_arrays(edge_lengths(rng), 7000, 9)
    m, dt = len(rp) - 1, getattr(torch, storage)
    dC = rng.integers(-3, 4, size=(m, n)).astype(np.float32)
    B = rng.integers(-4, 5, size=(7000, n)).astype(np.float32)
    d_rp, d_ci, d_dC, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, dC, B))
    out = gpu_lib.sddmm(d_rp, d_ci, d_dC.to(dt), d_B.to(dt), out_dtype=getattr(torch, result))
    ref = torch.from_numpy(oracle.sddmm(rp, ci, dC, B)).to(getattr(torch, result))
    assert torch.equal(out.cpu(), ref)


@pytest.mark.parametrize("n,pad", [(48, 1), (64, 2), (100, 1), (128, 2), (256, 4), (250, 2)])
def test_strides(gpu_lib, n, pad):
    """ldb and lddc above n, down to 4- and 8-byte alignment."""
    import torch

    rng = np.random.default_rng(n + pad)
    rp, ci, _ = csr_arrays(edge_lengths(rng), 7000, 10)
    dC = rng.integers(-3, 4, size=(len(rp) - 1, n + pad)).astype(np.float32)
    B = rng.integers(-4, 5, size=(7000, n + pad)).astype(np.float32)
    d_rp, d_ci, d_dC, d_B = (torch.from_numpy(x).cuda() for x in (rp, ci, dC, B))
    out = gpu_lib.sddmm(d_rp, d_ci, d_dC[:, :n], d_B[:, :n])
    ref = oracle.sddmm(rp, ci, np.ascontiguousarray(dC[:, :n]), np.ascontiguousarray(B[:, :n]))
    assert np.array_equal(out.cpu().numpy(), ref.astype(np.float32))


@pytest.mark.parametrize("n", [132, 180, 184, 252, 260, 388])
@pytest.mark.parametrize("k", [7000, 300_000])
def test_last_passes_are_bitwise(gpu_lib, n, k):
    """Widths whose last pass joins the one before it, always or where B is large."""
    import torch

    rng = np.random.default_rng(n)
    rp, ci, _ = csr_arrays(np.concatenate([rng.integers(0, 9, 600), [0, 300, 0, 31, 33]]).astype(np.int64), k, 9)
    g = torch.Generator(device="cuda").manual_seed(n)
    dC = rng.integers(-3, 4, size=(len(rp) - 1, n)).astype(np.float32)
    B = torch.randint(-4, 5, (k, n), device="cuda", generator=g).float()
    d_rp, d_ci, d_dC = (torch.from_numpy(x).cuda() for x in (rp, ci, dC))
    out = gpu_lib.sddmm(d_rp, d_ci, d_dC, B)
    rows = torch.repeat_interleave(torch.arange(len(rp) - 1, device="cuda"), (d_rp[1:] - d_rp[:-1]).long())
    assert torch.equal(out, (d_dC[rows] * B[d_ci.long()]).sum(1))


@pytest.mark.parametrize("n,storage,nnz", [(16, "float32", 3_600_000), (16, "float32", 3_599_999), (4, "bfloat16", 2_500_000),
                                           (8, "bfloat16", 7_000_000), (5, "float32", 185_000), (5, "float32", 195_000)])
def test_the_lines_between_lane_groups_and_warps(gpu_lib, n, storage, nnz):
    import torch

    g = torch.Generator(device="cuda").manual_seed(nnz)
    m, k, dt = 40_000, 5000, getattr(torch, storage)
    rp = (torch.arange(m + 1, device="cuda", dtype=torch.int64) * nnz // m).int()
    ci = torch.randint(k, (nnz,), device="cuda", generator=g).int()
    dC = torch.randint(-3, 4, (m, n), device="cuda", generator=g).to(dt)
    B = torch.randint(-4, 5, (k, n), device="cuda", generator=g).to(dt)
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), (rp[1:] - rp[:-1]).long())
    out = gpu_lib.sddmm(rp, ci, dC, B)
    assert torch.equal(out, (dC[rows].float() * B[ci.long()].float()).sum(1).to(dt))
