"""The plan's eigenvectors (forward recurrence with block exponents) at the sizes where it can go
wrong: one to a few entries, block edges of 8, long regions without oscillation (indices far from
2NW, where entries underflow), W next to 0 and 1/2.  Reference: dense eigenvectors of Slepian's
tridiagonal matrix.  Tolerance: an eigenvector of a backward stable method is off by at most
about eps ||T|| / gap; both sides take 8 eps ||T|| / gap."""
import numpy as np
import pytest

from paper_1611_04950_gb300 import fst as F


def _dense(N, W):
    n = np.arange(N, dtype=np.float64)
    c = 0.0 if W == 0.25 else np.cos(2 * np.pi * W)
    T = np.diag(((N - 1) / 2 - n) ** 2 * c)
    off = n[1:] * (N - n[1:]) / 2
    th, v = np.linalg.eigh(T + np.diag(off, 1) + np.diag(off, -1))
    return th[::-1], v[:, ::-1]


@pytest.mark.parametrize("N,W,K", [(1, 0.3, 1), (2, 0.2, 1), (3, 0.2, 1), (15, 0.1, 3), (16, 0.1, 3), (17, 0.1, 3),
                                   (33, 0.25, 16), (257, 1e-3, 0), (400, 0.499, 399), (800, 0.2, 3), (801, 0.2, 790),
                                   (1000, 1 / 64, 31)])
def test_vectors_against_dense(N, W, K):
    p = F.Plan(N, W, K=K, eps=1e-6, emulate=True)
    e = p.export()
    th, v = _dense(N, W)
    scale = np.abs(th).max() + 1e-300
    for j, l in enumerate(e["idx"]):
        s, ref = e["S_T"][:, j], v[:, l]
        gap = min([abs(th[l] - th[m]) for m in (l - 1, l + 1) if 0 <= m < N] + [scale])
        tol = 16 * 2.2e-16 * scale / gap + 1e-14
        assert np.abs(s - ref * np.sign(s @ ref)).max() <= tol
        ref_sum = s.sum() if l % 2 == 0 else (s * (N - 1 - 2 * np.arange(N))).sum()
        # (far above 2NW the sum vanishes and its sign is that of a rounding error)
        assert ref_sum > 0 or abs(ref_sum) < 1e-12 * N
        assert np.array_equal(s, (-1) ** int(l) * s[::-1])


def test_long_signal_rescaling():
    # eight steps of the Sturm recurrence grow by more than 2^256 from N = 2^18 on: the eigenvalues
    # lambda must straddle 1/2 around 2NW and the vectors be orthonormal (8 eps ||T|| / gap = 2e-9)
    p = F.Plan(1 << 18, 0.05, eps=1e-1, emulate=True)
    e = p.export()
    assert e["lam"][0] > 0.5 > e["lam"][-1] and np.all(np.diff(e["lam"]) < 0)
    assert np.abs(e["S_T"].T @ e["S_T"] - np.eye(p.r)).max() < 2e-9
