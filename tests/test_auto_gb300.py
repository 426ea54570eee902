"""The family that SPMM_ALG_AUTO_GB300 runs, and that the library names for it."""
import pytest

import paper_1803_08601_gb300 as pkg
from test_workspace import problem


@pytest.mark.gpu
@pytest.mark.parametrize("m,nnz,longest,n", [(4000, 20_000, 3000, 1), (4000, 20_000, 3000, 8), (4000, 20_000, 3000, 64),
                                             (600_000, 9_600_000, 1_000_000, 8), (600_000, 9_600_000, 1_000_000, 32),
                                             (900_000, 1_800_000, 2, 32), (30_000, 60_000, 2, 32),
                                             (30_000, 300_000, 10, 32), (30_000, 300_000, 10, 8)])
def test_a_call_runs_the_family_that_is_named(gpu_lib, m, nnz, longest, n):
    """By the bits and the launches of a forced call: 1 for the row split, 2 for the hybrid, 3 for merge.  The
    large skewed matrix at n = 8 has to stay with the hybrid."""
    import torch

    rp, ci, v, B = problem(torch, m, 1000, n, nnz)
    if longest > nnz // m:  # the first row takes what the others give up
        rp[1:] = (longest + torch.arange(m, device="cuda", dtype=torch.int64) * (nnz - longest) // (m - 1)).int()
    alg = gpu_lib.spmm_auto_gb300_alg(m, nnz, longest, n, gpu_lib.F32)
    if n == 8 and m == 600_000:
        assert alg == gpu_lib.ALG_ROW_SPLIT_HYBRID
    v = torch.randn(nnz, device="cuda")
    counts, C = [], []
    for a in (pkg.ALG_AUTO_GB300, alg):
        before = gpu_lib.spmm_launch_count()
        C.append(gpu_lib.spmm(rp, ci, v, B, alg=a, nnz=nnz, tuning=dict(max_row_len=longest)))
        counts.append(gpu_lib.spmm_launch_count() - before)
    assert counts[0] == counts[1] == {pkg.ALG_ROW_SPLIT: 1, pkg.ALG_ROW_SPLIT_HYBRID: 2, pkg.ALG_MERGE: 3}[alg]
    assert torch.equal(*C)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 4, 8, 16])
def test_a_workspace_for_the_selected_family_is_enough(gpu_lib, n):
    """Sized for the hybrid that the selector names, where the call runs merge if it allocates for itself."""
    import torch

    m, nnz, longest = 3_000_000, 400_000, 200_000  # full merge tiles take more than the hybrid
    rp, ci, v, B = problem(torch, m, 1000, n, nnz)
    rp[1:] = (longest + torch.arange(m, device="cuda", dtype=torch.int64) * (nnz - longest) // (m - 1)).int()
    named = gpu_lib.spmm_select_alg_gb300(m, nnz, longest, n, gpu_lib.F32)
    assert named == gpu_lib.ALG_ROW_SPLIT_HYBRID
    assert gpu_lib.spmm_auto_gb300_alg(m, nnz, longest, n, gpu_lib.F32) == gpu_lib.ALG_MERGE
    ws = torch.empty(gpu_lib.workspace_size(m, 1000, n, nnz, named), dtype=torch.uint8, device="cuda")
    hint = dict(max_row_len=longest)
    C = gpu_lib.spmm(rp, ci, v, B, alg="auto_gb300", nnz=nnz, tuning=hint, workspace=ws)
    assert torch.equal(C, gpu_lib.spmm(rp, ci, v, B, alg="merge", nnz=nnz))
    with pytest.raises(gpu_lib.SpMMError) as e:
        gpu_lib.spmm(rp, ci, v, B, alg="auto_gb300", nnz=nnz, tuning=hint, workspace=ws[:1024])
    assert e.value.status == gpu_lib.ERR_WORKSPACE


def test_the_hybrid_stays_where_it_is_ahead():
    """Both sides of the lines, at sizes where both families were timed."""
    pkg.build()
    F, H, M = pkg.F32, pkg.BF16, 1_000_000
    hybrid = [(400_000, 11_120_000, 40_000, 64, H), (200_000, 5_260_000, 20_000, 40, H), (300_000, 6_690_000, 30_000, 8, F),
              (M, 23_500_000, 100_000, 2, F), (500_000, 500_000, 1, 128, H), (50_000, 50_000, 1, 96, H),
              (800_000, 800_000, 1, 256, H), (1_200_000, 1_200_000, 1, 40, F), (500_000, M, 2, 48, F),
              (1_200_000, 2_400_000, 2, 128, F), (1_200_000, 2_400_000, 2, 192, F), (1_200_000, 1_200_000, 1, 64, F),
              (800_000, 1_600_000, 2, 32, F)]
    merge = [(100_000, 1_900_000, 10_000, 64, H), (200_000, 5_260_000, 20_000, 16, H), (200_000, 5_260_000, 20_000, 16, F),
             (M, 23_500_000, 100_000, 32, F), (M, 23_500_000, 100_000, 5, F), (M, 23_500_000, 100_000, 1, F),
             (500_000, 500_000, 1, 256, H), (800_000, 800_000, 1, 160, H), (M, 2 * M, 2, 100, H), (200_000, 200_000, 1, 48, F),
             (500_000, 500_000, 1, 128, F), (M, 2 * M, 2, 100, F), (800_000, 800_000, 1, 32, F)]
    for alg, cases in ((pkg.ALG_ROW_SPLIT_HYBRID, hybrid), (pkg.ALG_MERGE, merge)):
        for c in cases:
            assert pkg.spmm_select_alg_gb300(*c) == pkg.ALG_ROW_SPLIT_HYBRID, c
            assert pkg.spmm_auto_gb300_alg(*c) == alg, c
