"""The shared-column kernels of T2^* y and T1 c (fst_lowrank.cuh) at their edges: the smallest N they
take, batches around the 16 vector columns of a block and the vectors of a round, real and complex
signals, low-rank sizes from the smallest to wide ones.  The FP64 path (generic kernels, pinned to the
oracle elsewhere) is the reference; FP32 rounding of sums over N = 2^7 .. 2^16 white-noise samples is
far below 2e-6 of the vector's norm, which is what is allowed (measured start: 2e-7)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402


@pytest.mark.parametrize("N,W,eps", [(64, 0.2, 1e-3), (128, 0.1, 1e-3), (256, 0.24, 0.3), (2048, 0.05, 1e-12), (32768, 0.21, 1e-6),
                                     (65536, 1 / 8, 1e-4)])
@pytest.mark.parametrize("batch,cplx", [(1, False), (1, True), (3, False), (8, True), (9, True), (16, False), (17, False),
                                        (33, True)])
def test_lowrank_against_fp64(N, W, eps, batch, cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, eps=eps)
    y = workloads.gaussian(batch, N, seed=3, complex_=cplx).to("cuda")
    ref = p.coeffs(y)
    y32 = y.to(torch.complex64 if cplx else torch.float32)
    got = p.coeffs(y32)
    nF = F.fst_coeffs_info(p.h)["nF"]
    for sl in (slice(0, nF), slice(nF, None)):
        d = (got[:, sl].to(torch.complex128) - ref[:, sl]).norm(dim=1)
        assert bool((d <= 2e-6 * ref[:, sl].norm(dim=1) + 1e-6).all()), (d / ref[:, sl].norm(dim=1)).max()
    assert torch.equal(p.coeffs(y32), got)
    x = p.expand(got)
    want = p.expand(got.to(torch.complex128))
    assert bool(((x.to(torch.complex128) - want).norm(dim=1) <= 2e-6 * want.norm(dim=1)).all())


@pytest.mark.parametrize("N,W,eps,batch,shared", [(128, 0.1, 1e-8, 3, True), (128, 0.2, 1e-6, 40, True), (128, 0.2, 1e-3, 146, False),
                                                  (128, 0.2, 1e-3, 147, True), (256, 0.1, 1e-8, 700, True),
                                                  (1024, 0.2, 1e-2, 64, False), (2048, 0.1, 1e-10, 50, True),
                                                  (4096, 0.2, 1e-6, 130, True), (4096, 0.2, 1e-6, 260, True)])
def test_expand_route_and_vectors_per_thread(N, W, eps, batch, shared):
    # the generic kernel for few short vectors with few columns; one, two and four vectors a thread
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, eps=eps)
    rH = F.fst_coeffs_info(p.h)["rH"]
    assert shared == (not (N <= 1024 and rH <= 8 and batch * rH <= 1024))
    y = workloads.gaussian(batch, N, seed=4, complex_=True).to("cuda")
    c = p.coeffs(y.to(torch.complex64))
    F.fst_profile_enable(True)
    x = p.expand(c)
    names = {r[0] for r in F.fst_profile_records()}
    F.fst_profile_enable(False)
    assert ("k_expand_gemm" in names) == shared
    want = p.expand(c.to(torch.complex128))
    assert bool(((x.to(torch.complex128) - want).norm(dim=1) <= 2e-6 * want.norm(dim=1)).all())
