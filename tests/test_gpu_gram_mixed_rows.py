"""The FP64-accurate Gram on rows of unlike shape: a row of equal-sized entries beside rows in which one
entry is a thousand times the others, whose scaled norms are far apart.

Bound, on rows scaled by powers of two to entries below 1 and squared norms below 2^8: a digit string
ends 2^-56 below the scale (2^-56 per entry of either row) and the result rounds once to double.  The two
other errors are sums of independent terms, taken at six standard deviations: the dropped digit products,
six a column (twelve on the diagonal, where they are equal in pairs) of uniform digits of variance
(256^2 - 1) / 12 at weight 2^-70, and one rounding per 32 columns of a uniform error in 2^-54.  An FP64
multiply-add sum in order has about this error.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gram", [0, 2])
@pytest.mark.parametrize("K", [4096, 21632])
def test_flat_and_spiky_rows(gram, K):
    from paper_2503_12557_gb300 import peps as P
    rng = np.random.default_rng(K)
    A = rng.standard_normal((24, K))
    A[0] = rng.choice([-1.0, 1.0], K) * rng.uniform(0.5, 1.0, K)
    for i in range(2, 24):
        A[i, rng.integers(K)] = 1e3 * rng.choice([-1.0, 1.0])
    h = P.PEPS(2, 2, 2, 2, 2, max_samples=1, gram=gram)
    T = h.minsr_gram(torch.as_tensor(A).cuda()).cpu().numpy()
    assert h.last_status() == 0
    h.close()
    e = np.frexp(np.abs(A).max(1))[1]
    S = np.ldexp(A, -e[:, None])
    t = np.maximum(0, (np.frexp((S ** 2).sum(1))[1] - 8 + 1) // 2)
    S, e = np.ldexp(S, -t[:, None]), e + t
    Ts = np.ldexp(np.ldexp(T, -e[:, None]), -e[None, :])
    ref = S.astype(np.longdouble) @ S.T.astype(np.longdouble)
    one = np.abs(S).sum(1)
    bound = 2.0 ** -56 * (one[:, None] + one[None, :]) + 2.0 ** -53 * np.abs(ref)
    bound = bound + 6 * np.sqrt(12 * K) * (256 ** 2 - 1) / 12 * 2.0 ** -70 + 6 * np.sqrt((K / 32 + 1) / 12) * 2.0 ** -54
    assert np.all(np.abs(Ts - ref) <= bound)
