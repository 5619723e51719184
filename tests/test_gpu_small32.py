"""The FP32 single-CTA kernel (fst_small32.cuh) at the sizes where it can go wrong: every transform
length 2^10 .. 2^14 (first radix 1, 2, 4, 8), both ends of each length's range of N, odd N (the
middle sample), ranks of every shared-memory shape, odd batches, complex signals, in place, strided
rows, and the same signals through a ragged batch.  Against the FP64 oracle; tolerance 1e-5 of ||y||,
the FP32 tolerance of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402
from oracle import fst_oracle as O  # noqa: E402


@pytest.mark.parametrize("N,W,eps,K,batch,cplx", [
    (257, 0.2, 1e-6, None, 3, False), (512, 0.1, 1e-3, None, 1, True), (513, 0.25, 1e-8, None, 5, False),
    (1024, 1 / 64, 1e-8, None, 2, True), (1025, 0.2, 1e-6, None, 4, False), (2047, 0.25, 1e-12, None, 3, True),
    (2049, 0.1, 1e-6, None, 5, False), (3001, 0.25, 1e-6, None, 999, False), (4096, 1 / 16, 1e-6, None, 2, False),
    (4097, 0.2, 1e-6, None, 3, True), (8191, 0.05, 1e-4, None, 2, False), (8192, 0.25, 1e-8, None, 3, True),
    (700, 0.2, 1e-6, 185, 3, False), (700, 0.2, 1e-6, 230, 2, True)])
def test_small32_against_oracle(N, W, eps, K, batch, cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, K=K, eps=eps)
    o = O.make_plan(N, W, p.K, eps)
    assert p.r == o.r
    y = workloads.gaussian(batch, N, seed=N, complex_=cplx).to(torch.complex64 if cplx else torch.float32)
    nrm = np.linalg.norm(y.numpy(), axis=1)
    y64 = y.numpy().astype(np.complex128 if cplx else np.float64)
    ref = O.fast_project(o, y64.T).T
    yd = y.to("cuda")
    out = p.project(yd)
    assert np.all(np.linalg.norm(out.cpu().numpy() - ref, axis=1) < 1e-5 * nrm)
    wide = torch.zeros((batch, N + 3), dtype=y.dtype, device="cuda")
    wide[:, :N] = yd
    got = p.project(wide[:, :N], out=wide[:, :N])
    assert torch.equal(got, out) and torch.count_nonzero(wide[:, N:]) == 0
    b = p.apply_prolate(yd).cpu().numpy()
    z = (o.S_T @ (o.D[:, None] * (o.S_T.T @ y64.T))).T
    assert np.all(np.linalg.norm(b + z - ref, axis=1) < 1e-5 * nrm)
    if batch > 1:
        ys = [v.clone() for v in yd[:3]]
        outs = [torch.empty_like(v) for v in ys]
        F.fst_project_ragged([p.h] * len(ys), [v.data_ptr() for v in ys], [v.data_ptr() for v in outs],
                             F._dtype_code(y.dtype), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        for i, v in enumerate(outs):
            assert np.linalg.norm(v.cpu().numpy() - ref[i]) < 1e-5 * nrm[i]
