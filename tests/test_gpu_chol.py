"""The FP64 Cholesky of the MinSR solve (peps_chol.cu) through minsr_solve: sizes at the edges of its
64-row panels and 128-row update tiles, every split of the panel kernel, and badly scaled matrices."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2503_12557_gb300 import peps
    return peps


def _spd(n, seed, cond=1e6):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(n, 2 * n, generator=g, device="cuda", dtype=torch.float64)
    d = torch.logspace(0, -0.5 * np.log10(cond), n, device="cuda", dtype=torch.float64)
    A = A * d[torch.randperm(n, generator=g, device="cuda")][:, None]
    return A @ A.T / n, torch.randn(n, generator=g, device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("solve", [0, 2])
@pytest.mark.parametrize("n", [2, 3, 63, 64, 65, 66, 128, 130, 191, 193, 320, 513, 1300, 2500])
def test_solve_is_backward_stable(P, n, solve):
    T, b = _spd(n, n)
    h = P.PEPS(2, 2, 2, 2, 2, max_samples=1, solve=solve)
    lam = 1e-6 * float(T.diagonal().max())
    x, info = h.minsr_solve(T, b, lam=lam)
    assert h.last_status() == 0 and int(info[0]) == n
    M = T + lam * torch.eye(n, device="cuda", dtype=torch.float64)
    # Higham, Accuracy and Stability, th. 10.3-10.4: (M + dM) x = b with |dM| <= 4 n (3 n + 1) u |M|;
    # the factor's rows are scaled alike, so half of it, in the diagonally scaled norm
    d = M.diagonal().rsqrt()
    r = (b - M @ x) * d
    scale = (d[:, None] * M.abs() * d[None, :]).sum(1).max() * (x / d).abs().max()
    assert float(r.abs().max()) <= 4 * n * 2.0 ** -53 * float(scale) + 1e-300


def test_not_positive_definite_is_reported(P):
    T, b = _spd(300, 5)
    T[200, 200] = -1.0
    for solve in (0, 2):
        h = P.PEPS(2, 2, 2, 2, 2, max_samples=1, solve=solve)
        x, info = h.minsr_solve(T.clone(), b, lam=1e-9)
        h.last_status()
        assert int(info[0]) == -1 and h.last_warning and torch.all(x == 0)
