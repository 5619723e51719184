"""fst_project_host over several chunks gives the bits of fst_project on the whole batch: FP64 at
both kinds of length (the partials of S_T^T y and the transform's split follow the whole call), FP32
on every form of the correction (tensor cores with a chunk of few rows, folded sums at P <= 32 and
at two-stage lengths, P = 8), odd batches, complex signals.  FST_HOST_CHUNK_MB=1 makes many chunks."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402


@pytest.mark.parametrize("N,W,eps,batch,dtype", [
    (4096, 1 / 16, 1e-6, 301, torch.float64), (2000, 0.2, 1e-8, 777, torch.float64), (1000, 0.1, 1e-6, 90, torch.complex128),
    (8192, 0.1, 1e-6, 75, torch.float64), (40000, 0.1, 1e-6, 30, torch.float64), (40000, 0.1, 1e-6, 7, torch.float64),
    (20011, 0.25, 1e-8, 21, torch.complex128), (65536, 1 / 8, 1e-4, 45, torch.float32), (65536, 1 / 8, 1e-4, 20, torch.complex64),
    (9001, 0.1, 1e-6, 99, torch.float32), (9001, 0.1, 1e-6, 60, torch.float32), (20003, 0.25, 1e-8, 101, torch.float32),
    (70000, 0.2, 1e-6, 70, torch.float32), (131072, 0.05, 1e-6, 33, torch.complex64), (3001, 0.25, 1e-6, 999, torch.float32)])
def test_host_chunks_bit_for_bit(monkeypatch, N, W, eps, batch, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, eps=eps)
    y = workloads.gaussian(batch, N, seed=N, complex_=dtype.is_complex).to(dtype)
    ref = p.project(y.cuda()).cpu()
    monkeypatch.setenv("FST_HOST_CHUNK_MB", "1")
    got = p.project_host(y.pin_memory())
    bad = (got != ref).any(dim=1)
    assert not bool(bad.any()), f"{int(bad.sum())} of {batch} signals differ"
