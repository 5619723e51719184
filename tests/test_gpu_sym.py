"""The folded rank-r correction (fst_sym.cuh) at its edges: odd N (the middle sample), N with every
remainder mod 4 (16-byte and single accesses), 1 to 130 rows (every block height and row-group count),
strided and unaligned rows, complex signals, in place, ranks from one column tile to several.  Against
the FP64 oracle; tolerance 1e-5 of ||y||, the FP32 tolerance of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402
from oracle import fst_oracle as O  # noqa: E402


@pytest.mark.parametrize("N,W,eps", [(9001, 0.2, 1e-1), (10002, 0.1, 1e-6), (20003, 0.25, 1e-8), (66000, 0.05, 1e-6),
                                     (70001, 0.2, 1e-12), (131074, 0.1, 1e-4)])
@pytest.mark.parametrize("batch,cplx", [(1, False), (1, True), (5, True), (9, False), (17, True), (33, False), (65, True)])
def test_folded_correction(N, W, eps, batch, cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, eps=eps)
    o = O.make_plan(N, W, p.K, eps)
    assert p.r == o.r
    y = workloads.gaussian(batch, N, seed=N + batch, complex_=cplx).to(torch.complex64 if cplx else torch.float32)
    nrm = np.linalg.norm(y.numpy(), axis=1)
    pick = sorted({0, batch // 2, batch - 1})
    ref = O.fast_project(o, y.numpy()[pick].astype(np.complex128 if cplx else np.float64).T).T
    yd = y.to("cuda")
    out = p.project(yd)
    assert np.all(np.linalg.norm(out.cpu().numpy()[pick] - ref, axis=1) < 1e-5 * nrm[pick])
    assert torch.equal(p.project(yd), out)
    flat = torch.zeros(batch * (N + 3) + 1, dtype=y.dtype, device="cuda")
    wide = flat[1:].view(batch, N + 3)[:, :N]            # odd stride and base
    wide.copy_(yd)
    got = p.project(wide, out=wide)                      # in place
    assert np.all(np.linalg.norm(got.cpu().numpy()[pick] - ref, axis=1) < 1e-5 * nrm[pick])


@pytest.mark.parametrize("N,W,eps,batch,cplx", [(40000, 0.25, 1e-8, 64, False), (65536, 0.2, 1e-8, 17, True),
                                                (8196, 0.2, 1e-9, 33, False)])
def test_tensor_core_correction_rank_33_to_64(N, W, eps, batch, cplx):
    # more than 32 addressable rows, N <= 65536, two column tiles of 32: the tcgen05 sums
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, W, eps=eps)
    o = O.make_plan(N, W, p.K, eps)
    assert p.r == o.r and 32 < p.r <= 64
    y = workloads.gaussian(batch, N, seed=batch, complex_=cplx).to(torch.complex64 if cplx else torch.float32)
    pick = sorted({0, batch // 2, batch - 1})
    ref = O.fast_project(o, y.numpy()[pick].astype(np.complex128 if cplx else np.float64).T).T
    yd = y.to("cuda")
    F.fst_profile_enable(True)
    out = p.project(yd)
    names = {r[0] for r in F.fst_profile_records()}
    F.fst_profile_enable(False)
    assert "k_corr_tc" in names
    nrm = np.linalg.norm(y.numpy(), axis=1)
    assert np.all(np.linalg.norm(out.cpu().numpy()[pick] - ref, axis=1) < 1e-5 * nrm[pick])
    assert torch.equal(p.project(yd), out)


@pytest.mark.parametrize("N", [8193, 16383])
@pytest.mark.parametrize("batch,cplx", [(48, False), (49, False), (32, True)])
def test_unaligned_rows_around_the_column_pass_rule(N, batch, cplx):
    # P = 8, rows no tensor map can address: own products up to 48 rows, folded sums above
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, 0.2, eps=1e-6)
    o = O.make_plan(N, 0.2, p.K, 1e-6)
    y = workloads.gaussian(batch, N, seed=batch, complex_=cplx).to(torch.complex64 if cplx else torch.float32)
    pick = [0, batch // 2, batch - 1]
    ref = O.fast_project(o, y.numpy()[pick].astype(np.complex128 if cplx else np.float64).T).T
    yd = y.to("cuda")
    F.fst_profile_enable(True)
    out = p.project(yd)
    names = {r[0] for r in F.fst_profile_records()}
    F.fst_profile_enable(False)
    assert ("k_sym_c" in names) == (batch * (2 if cplx else 1) > 48)
    nrm = np.linalg.norm(y.numpy(), axis=1)
    assert np.all(np.linalg.norm(out.cpu().numpy()[pick] - ref, axis=1) < 1e-5 * nrm[pick])


@pytest.mark.parametrize("batch", [1, 8])
def test_few_rows_sum_as_accurately_as_unfolded(batch):
    # chains of more than 64 products: U2^* y of N = 2^21 against FP64, no further off than the sums
    # over blocks of 2048 samples that the folded form replaced (2.1e-7 to 2.2e-7)
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N = 1 << 21
    p = F.Plan(N, 0.2, eps=1e-4)
    S = torch.as_tensor(p.export()["S_T"]).cuda()
    sd = torch.as_tensor(p.export(False)["D"]).cuda().abs().sqrt()
    num = den = 0.0
    for seed in range(16 // batch):
        y = workloads.gaussian(batch, N, seed=seed).float().cuda()
        ref = (y.double() @ S) * sd
        got = p.coeffs(y)[:, -p.r:].real.double()
        num += float((got - ref).norm()) ** 2
        den += float(ref.norm()) ** 2
    assert (num / den) ** 0.5 <= 2.2e-7


@pytest.mark.parametrize("N,eps,batch,own", [(8193, 1e-6, 16, False), (8193, 1e-6, 17, True), (20001, 1e-6, 32, False),
                                             (20001, 1e-6, 33, True), (32767, 1e-6, 48, True), (30001, 1e-6, 49, False),
                                             (40001, 1e-6, 40, False), (40001, 1e-3, 40, True)])
def test_unaligned_rows_by_column_count(N, eps, batch, own):
    # which of P = 8, 16, 32 keeps the column pass's own products, and that both forms agree with the oracle
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = F.Plan(N, 0.2, eps=eps)
    o = O.make_plan(N, 0.2, p.K, eps)
    y = workloads.gaussian(batch, N, seed=batch).float()
    pick = [0, batch // 2, batch - 1]
    ref = O.fast_project(o, y.numpy()[pick].astype(np.float64).T).T
    yd = y.to("cuda")
    F.fst_profile_enable(True)
    out = p.project(yd)
    names = {r[0] for r in F.fst_profile_records()}
    F.fst_profile_enable(False)
    assert ("k_sym_c" not in names) == own
    nrm = np.linalg.norm(y.numpy(), axis=1)
    assert np.all(np.linalg.norm(out.cpu().numpy()[pick] - ref, axis=1) < 1e-5 * nrm[pick])
