"""FP64 four-step kernels (fst_fast64.cuh) at the sizes where they can go wrong: every split of M =
2^10 .. 2^18 (P = 8, 16, 32; 32- to 8192-point rows), odd and ragged lengths, odd batches, complex
signals, ranks above one shared-memory round, in place, strided.  Against the FP64 oracle; tolerance
1e-12 of ||y||, the FP64 tolerance of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402
from oracle import fst_oracle as O  # noqa: E402


@pytest.mark.parametrize("N,W,eps,K,batch,cplx", [
    (511, 0.2, 1e-6, None, 3, False), (257, 0.1, 1e-3, None, 1, True), (1000, 1 / 64, 1e-8, None, 5, False),
    (2047, 0.25, 1e-8, None, 9, True), (4096, 1 / 16, 1e-6, None, 2, False), (4097, 0.2, 1e-6, None, 33, False),
    (8191, 0.05, 1e-4, None, 2, True), (9001, 0.1, 1e-6, None, 7, False), (20011, 0.25, 1e-8, None, 3, True),
    (8000, 0.1, 1e-6, None, 90, False), (16001, 0.1, 1e-6, None, 40, True),
    (65536, 1 / 8, 1e-4, None, 5, False), (100003, 0.03, 1e-6, None, 2, True), (600, 0.2, 1e-6, 40, 17, False)])
def test_fp64_against_oracle(N, W, eps, K, batch, cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, K=K, eps=eps)
    o = O.make_plan(N, W, p.K, eps)
    assert p.r == o.r
    y = workloads.gaussian(batch, N, seed=N, complex_=cplx)
    nrm = np.linalg.norm(y.numpy(), axis=1)
    ref = O.fast_project(o, y.numpy().T).T
    yd = y.to("cuda")
    out = p.project(yd)
    assert np.all(np.linalg.norm(out.cpu().numpy() - ref, axis=1) < 1e-12 * nrm)
    assert torch.equal(p.project(yd), out)
    wide = torch.zeros((batch, N + 5), dtype=y.dtype, device="cuda")
    wide[:, :N] = yd
    got = p.project(wide[:, :N], out=wide[:, :N])          # in place, strided rows
    assert torch.equal(got, out) and torch.count_nonzero(wide[:, N:]) == 0
    b = p.apply_prolate(yd).cpu().numpy()
    z = (o.S_T @ (o.D[:, None] * (o.S_T.T @ y.numpy().T))).T
    assert np.all(np.linalg.norm(b + z - ref, axis=1) < 1e-12 * nrm)


def test_fp64_in_a_stream_capture_without_workspace():
    # nothing can be allocated while a caller records a graph: a plan that has not run yet takes the
    # kernels that need no workspace
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, q = F.Plan(3000, 0.2, eps=1e-6), F.Plan(3000, 0.2, eps=1e-6)
    y = workloads.gaussian(3, 3000, seed=1).to("cuda")
    out = torch.empty_like(y)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.project(y, out=out)
    g.replay()
    torch.cuda.synchronize()
    ref = q.project(y)
    assert float((out - ref).norm()) < 1e-12 * float(y.norm())


def _captured(p, y):
    out = torch.empty_like(y)
    p.project(torch.zeros_like(y[:1]))          # first-call set-up happens before the recording
    torch.cuda.synchronize()
    n0 = F.fst_launch_count()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.project(y, out=out)
    return g, out, F.fst_launch_count() - n0


@pytest.mark.parametrize("batch,cplx", [(3, False), (2, True), (40, False)])
def test_fp64_short_signals_captured_without_the_workspace(batch, cplx):
    # single-CTA lengths: a caller's graph must not point at the plan's workspace, which a later
    # larger call frees, and must not depend on what the plan has run before
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p, q = F.Plan(3000, 0.2, eps=1e-6), F.Plan(3000, 0.2, eps=1e-6)
    y = workloads.gaussian(batch, 3000, seed=1, complex_=cplx).to("cuda")
    p.project(y)
    g, out, launches = _captured(p, y)
    assert launches == 1                        # the whole projection in one launch, no scratch
    big = workloads.gaussian(400, 3000, seed=2).to("cuda")
    p.project(big)                              # moves the workspace
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    first = out.clone()
    cold = torch.empty_like(y)
    gq = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gq):
        q.project(y, out=cold)
    gq.replay()
    torch.cuda.synchronize()
    assert torch.equal(first, cold)


def test_fp64_captured_whatever_ran_before():
    # longer lengths: a workspace left by a smaller call holds fewer pairs at a time, not other sums
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    y = workloads.gaussian(32, 8000, seed=5).to("cuda")
    outs = []
    for warm in (32, 16):
        p = F.Plan(8000, 0.2, eps=1e-6)
        p.project(y[:warm].clone())
        out = torch.empty_like(y)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.project(y, out=out)
        g.replay()
        torch.cuda.synchronize()
        outs.append((out, p))
    assert torch.equal(outs[0][0], outs[1][0])
    assert torch.equal(outs[0][0], outs[0][1].project(y))


@pytest.mark.parametrize("graphs", ["1", "0"])
def test_fp64_short_signals_on_a_full_device(monkeypatch, graphs):
    # the split kernels' workspace is not to be had: the kernel that needs none answers
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("FST_GRAPHS", graphs)
    p = F.Plan(4096, 1 / 16, eps=1e-6)
    y = workloads.gaussian(5, 4096, seed=8).to("cuda")
    F.fst_test_alloc_fail(1)
    try:
        got = p.project(y)
        again = p.project(y, out=torch.empty_like(y))   # with memory again: the split kernels
    finally:
        F.fst_test_alloc_fail(0)
    assert float((got - again).norm()) < 1e-12 * float(y.norm())


@pytest.mark.parametrize("N,W", [(4096, 1 / 16), (100003, 0.1)])
def test_fp64_rounding_against_long_double(N, W):
    # B y of a pair by FFTs in long double (64 or more bits of mantissa).  Kernels that form their twiddles as
    # products of a few small angles' roots are off by 3.8e-16 and 5.1e-16 here; a table entry per
    # factor has one rounding instead of up to three, so it may not be further off
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fft = pytest.importorskip("scipy.fft")
    L = np.longdouble
    if np.finfo(L).eps > 1e-18 or fft.rfft(np.ones(4, L)).dtype != np.clongdouble:
        pytest.skip("no extended precision")
    pi = L("3.14159265358979323846264338327950288")
    k = np.arange(1, N).astype(L)
    x = 2 * L(W) * k
    b = np.concatenate([[2 * L(W)], np.sin(pi * (x - 2 * np.floor(x / 2))) / (pi * k)])
    M = 1 << (2 * N - 1).bit_length()
    c = np.concatenate([b, np.zeros(M - 2 * N + 1, L), b[:0:-1]])
    y = workloads.gaussian(2, N, seed=N)
    B = fft.rfft(c)
    ref = np.stack([fft.irfft(B * fft.rfft(np.concatenate([v.astype(L), np.zeros(M - N, L)])), n=M)[:N] for v in y.numpy()])
    got = F.Plan(N, W, eps=1e-6).apply_prolate(y.cuda()).cpu().numpy()
    err = np.sqrt(((got - ref) ** 2).sum() / (ref ** 2).sum())
    assert err < (3.8e-16 if N == 4096 else 5.1e-16), err
