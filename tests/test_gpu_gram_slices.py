"""The digit-sliced tensor-core Gram (peps_gram_sl.cu) through minsr_gram: exact on integers at the
edges of its tiles and chunks, within its error bound of an extended-precision sum on badly
scaled rows, and with more columns than one panel of digits holds."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2503_12557_gb300 import peps
    return peps


def _gram(P, A, gram=0):
    h = P.PEPS(2, 2, 2, 2, 2, max_samples=1, gram=gram)
    T = h.minsr_gram(A if torch.is_tensor(A) else torch.as_tensor(A).cuda())
    assert h.last_status() == 0
    return T


@pytest.mark.parametrize("gram", [0, 2])
@pytest.mark.parametrize("ns,k", [(1, 1), (2, 31), (127, 32), (128, 33), (129, 64), (257, 1000), (384, 4097)])
def test_integers_are_exact(P, ns, k, gram):
    # |a| < 2^19 and K < 2^13: every entry of T is an integer below 2^53, exact in double
    A = np.random.default_rng(ns + k).integers(-2 ** 19, 2 ** 19, size=(ns, k)).astype(np.float64)
    T = _gram(P, A, gram).cpu().numpy()
    Ai = A.astype(np.int64)
    assert np.array_equal(T, (Ai @ Ai.T).astype(np.float64))


@pytest.mark.parametrize("ns,k,seed", [(5, 3, 1), (130, 700, 2), (64, 2049, 3)])
def test_scaled_rows_within_the_bound(P, ns, k, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((ns, k)) * 10.0 ** rng.uniform(-6, 0, size=(ns, k))
    A *= 2.0 ** rng.integers(-400, 400, size=(ns, 1))
    A[0] = 0.0
    A[1] *= 1e-5 / np.abs(A[1]).max()
    A[2, k // 2] = 1e3 * np.abs(A[2]).max()  # one entry far above the rest of its row
    T = _gram(P, A).cpu().numpy()
    assert np.array_equal(T, T.T)
    # rows scaled to a largest modulus of 1 (powers of two keep every digit), so that the
    # extended-precision reference stays in range; the scaling is undone in T exactly
    e = np.where(np.abs(A).max(1) > 0, np.frexp(np.abs(A).max(1))[1], 0)
    S = np.ldexp(A, -e[:, None])
    Ts = np.ldexp(np.ldexp(T, -e[:, None]), -e[None, :])
    ref = S.astype(np.longdouble) @ S.T.astype(np.longdouble)
    one = np.abs(S).sum(1)
    # digits: 2^-56 per entry of either row; dropped products: 6 2^-56 (1 + 2^-7) per column;
    # fixed point: two roundings per 32 columns at 2^-f, f >= 60 - log2(largest squared row norm)
    f = min(52.0, 60.0 - np.log2(max(1.0, (S ** 2).sum(1).max())))
    bound = 2.0 ** -56 * (one[:, None] + one[None, :]) + k * 7 * 2.0 ** -56 + 2 * (k / 32 + 1) * 2.0 ** -f
    bound = bound + 2.0 ** -52 * np.abs(ref)
    assert np.all(np.abs(Ts - ref) <= bound)


def test_subnormal_and_nonfinite_rows(P):
    rng = np.random.default_rng(4)
    A = rng.standard_normal((140, 50))
    A[3] *= 1e-310
    A[5, 7] = np.nan
    A[133, 0] = np.inf
    T = _gram(P, A).cpu().numpy()
    ok = np.ones(140, bool)
    ok[[5, 133]] = False
    assert np.all(np.isnan(T[~ok])) and np.all(np.isnan(T[:, ~ok]))
    ref = A[ok] @ A[ok].T
    # |T_ij| <= 50 * 16: both sums within 2^-44 of the exact one; row 3's products with the others are subnormal
    assert np.all(np.abs(T[ok][:, ok] - ref) <= 2.0 ** -40 * np.abs(ref).max())


def test_more_columns_than_one_panel(P):
    # 256 rows x 600 000 columns need 2.15 GB of digits, over the 2 GiB a panel may hold
    g = torch.Generator(device="cuda").manual_seed(6)
    A = torch.randn(200, 600000, generator=g, device="cuda", dtype=torch.float64)
    T = _gram(P, A)
    ref = A @ A.T
    # an FP64 dot product of K terms is within K 2^-53 |a||b| of the exact one
    n = A.norm(dim=1)
    assert torch.all((T - ref).abs() <= 600000 * 2.0 ** -52 * n[:, None] * n[None, :])
