"""The transpose of a pattern is queued on the caller's stream and its longest row read on another one:
results must not depend on the stream of the step, nor on who asks for the transpose."""
import numpy as np
import pytest

import oracle
from spmm_cases import csr_arrays

pytestmark = pytest.mark.gpu


def problem(torch, pkg, n=20):
    rng = np.random.default_rng(5)
    rp, ci, v = csr_arrays(rng.integers(0, 30, 4000), 3000, 2, int_vals=True)
    B = rng.integers(-4, 5, size=(3000, n)).astype(np.float32)
    dC = rng.integers(-3, 4, size=(4000, n)).astype(np.float32)
    d = [torch.from_numpy(x).cuda() for x in (rp, ci, v, B, dC)]
    refs = oracle.spmm_t(rp, ci, v, dC, 3000), oracle.sddmm(rp, ci, dC, B)
    return d, [r.astype(np.float32) for r in refs]


@pytest.mark.parametrize("side", [False, True])
def test_new_pattern_every_step(gpu_lib, side):
    import torch

    (rp, ci, v, B, dC), (ref_dB, ref_dv) = problem(torch, gpu_lib)
    stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for _ in range(5):
            A = gpu_lib.CSRMatrix(rp, ci, (4000, 3000))
            vals, x = v.clone().requires_grad_(True), B.clone().requires_grad_(True)
            dv, dB = torch.autograd.grad(gpu_lib.spmm_autograd(A, vals, x), (vals, x), dC)
            assert np.array_equal(dB.cpu().numpy(), ref_dB) and np.array_equal(dv.cpu().numpy(), ref_dv)


def test_queued_on_one_stream_used_on_another(gpu_lib):
    import torch

    (rp, ci, v, _, dC), (ref_dB, _) = problem(torch, gpu_lib)
    A = gpu_lib.CSRMatrix(rp, ci, (4000, 3000))
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        A.queue_transpose()
        A.queue_transpose()  # once is enough
    with torch.cuda.stream(second):
        dB = A.spmm_t(v, dC)
    torch.cuda.synchronize()
    assert np.array_equal(dB.cpu().numpy(), ref_dB)
    assert A.transpose_pattern()[3] == int(torch.bincount(ci.long(), minlength=3000).max())


@pytest.mark.parametrize("queued", [True, False])
def test_the_transpose_outlives_its_matrix_on_another_stream(gpu_lib, queued):
    """Memory of A^T, made on one stream, is not given out again while another stream still has to read it, after
    the last reference is gone.  Nothing is written to what is given out, whoever it belongs to."""
    import torch

    (rp, ci, v, _, dC), (ref_dB, _) = problem(torch, gpu_lib)
    A = gpu_lib.CSRMatrix(rp, ci, (4000, 3000))
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    gpu_lib.CSRMatrix(rp, ci, (4000, 3000)).spmm_t(v, dC)  # loads the kernels
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        if queued:
            A.queue_transpose()
        held = [x.untyped_storage().nbytes() for x in A.transpose_pattern()[:3]]
        taken = {x.data_ptr() for x in A.transpose_pattern()[:3]}
    with torch.cuda.stream(second):
        torch.cuda._sleep(200_000_000)  # about a tenth of a second
        dB = A.spmm_t(v, dC)
    del A
    with torch.cuda.stream(first):
        again = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in held for _ in range(3)]
    assert not second.query()
    assert not taken & {x.data_ptr() for x in again}
    torch.cuda.synchronize()
    assert np.array_equal(dB.cpu().numpy(), ref_dB)


def test_the_probe_takes_no_stream_of_torchs_pool(gpu_lib, monkeypatch):
    """torch hands the 32 streams of its pool out in turn: one taken here would be some caller's as well."""
    import torch

    (rp, ci, _, _, _), _ = problem(torch, gpu_lib)

    stream = torch.cuda.Stream

    def taken(*args, **kw):  # an object of a stream that is there names its id
        assert "stream_id" in kw, "a stream of the pool"
        return stream(*args, **kw)

    A = gpu_lib.CSRMatrix(rp, ci, (4000, 3000))
    monkeypatch.setattr(torch.cuda, "Stream", taken)
    A.queue_transpose()
    assert A.transpose_pattern()[3] == int(torch.bincount(ci.long(), minlength=3000).max())
