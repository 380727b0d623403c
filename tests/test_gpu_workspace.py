"""Device memory at its limits, through the caller's allocator: refused allocations, smaller workspaces, and
calls after a failure."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2503_12557_gb300 import inputs as I

pytestmark = pytest.mark.gpu


class Limited:
    """Caller's allocator over torch's that refuses what `refuse(nbytes)` says."""

    def __init__(self, P, monkeypatch):
        self.sizes, self.refuse = [], lambda n: False

        def alloc(ctx, n):
            if self.refuse(int(n)):
                return None
            self.sizes.append(int(n))
            return P._torch_alloc(ctx, n)

        self.ref = P._Allocator(P._ALLOC_FN(alloc), P._FREE_FN(P._torch_free), None)
        monkeypatch.setattr(P, "_TORCH_ALLOCATOR", self.ref)


@pytest.fixture
def P():
    from paper_2503_12557_gb300 import build, peps
    build.build()
    return peps


def _minsr(P, h, ns, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    O = torch.randn(ns, h.Np, generator=g, device="cuda", dtype=h.odtype)
    e = torch.zeros(ns, 2, device="cuda", dtype=torch.float64)
    e[:, 0] = torch.randn(ns, generator=g, device="cuda", dtype=torch.float64)
    return h.minsr_step(O, e, lam=1e-3)[0].clone()


@pytest.mark.parametrize("gram", [0, 1])
def test_a_refused_growth_leaves_no_half_of_a_workspace(P, monkeypatch, gram):
    # the larger workspace fails at its k-th allocation; the smaller call that follows allocates anew
    lim = Limited(P, monkeypatch)
    h = P.PEPS(4, 4, 2, 2, 4, prec=0, max_samples=1, gram=gram)
    first = _minsr(P, h, 40)
    for k in range(14):
        calls = []

        def nth(n):
            calls.append(n)
            return len(calls) == k + 1

        lim.refuse = nth
        try:
            _minsr(P, h, 100)
        except RuntimeError as e:
            assert "PEPS_E_WORKSPACE" in str(e)
        lim.refuse = lambda n: False
        assert torch.equal(_minsr(P, h, 40), first)
    h.close()


def test_split_bf16_gram_of_more_columns_than_parameters(P):
    # minsr_gram takes any K: its operands are sized for the K of the call
    h = P.PEPS(2, 2, 2, 2, 2, max_samples=1, gram=1)
    A = torch.randn(130, 40 * h.Np + 3, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda",
                    dtype=torch.float64)
    T = h.minsr_gram(A)
    assert h.last_status() == 0
    n = A.norm(dim=1)
    # two BF16 parts of 8 bits each: 2^-16 of |a||b| dropped, FP32 sums of K terms
    bound = (2.0 ** -15 + A.shape[1] * 2.0 ** -23) * n[:, None] * n[None, :]
    assert torch.all((T - A @ A.T).abs() <= bound)
    h.close()


def test_noalloc_takes_what_fits_32_mib_without_the_scratch():
    # 536 samples of 4x4, D = 3, chi = 9 in FP64: parameters, environments and one CTA's buffers apart
    # from the row step's scratch are within 32 MiB
    from test_zz_no_alloc import _call, _noalloc_fn
    peps, f = _noalloc_fn()
    lat = I.Lattice(4, 4, 2, 3)
    theta = torch.as_tensor(I.peps_random(lat, 1, scale=0.5, bias=1.0)).cuda()
    S = torch.as_tensor(I.configs_uniform_sz0(lat, 536, 2)).cuda()
    rc, la, _, st = _call(peps, f, lat, 9, 0, theta, S)
    assert rc == 0
    h = peps.PEPS(4, 4, 2, 3, 9, prec=0, max_samples=536)
    h.set_params(theta)
    ref = h.amplitudes(S)
    assert float((la - ref[0]).abs().max()) <= 1e-10
    h.close()


@pytest.mark.parametrize("gram,solve,prec", [(0, 0, 0), (2, 2, 1), (0, 1, 1)])
def test_minsr_without_the_digit_and_factor_workspaces(P, monkeypatch, gram, solve, prec):
    # 600 rows: where neither workspace can be had, the n x n buffers that the solve leaves free hold them
    ns = 600
    n, K = ns, I.num_params(I.Lattice(6, 6, 2, 3))
    up = lambda x, a: (x + a - 1) // a * a  # noqa: E731
    digits = up(4 * n, 1024) + up(n, 128) * up(K, 32) * 14
    factor = up(14 * n * 64, 256) + (n + 63) // 64 * 64 * 65 * 8 + 4 * n + 256
    lim = Limited(P, monkeypatch)
    h = P.PEPS(6, 6, 2, 3, 9, prec=prec, max_samples=1, gram=gram, solve=solve)
    full = _minsr(P, h, ns)
    assert digits in lim.sizes and factor in lim.sizes
    rest = set(lim.sizes) - {digits, factor}
    h.close()
    lim.refuse = lambda b: b not in rest
    h = P.PEPS(6, 6, 2, 3, 9, prec=prec, max_samples=1, gram=gram, solve=solve)
    d = _minsr(P, h, ns)
    h.close()
    assert torch.equal(d, full)


def test_a_smaller_scratch_arena_gives_the_same_results(P, monkeypatch):
    lat = I.Lattice(6, 6, 2, 4)
    theta = torch.as_tensor(I.peps_random(lat, 1, scale=0.5, bias=1.0, alpha=1.5)).cuda()
    S = torch.as_tensor(I.configs_uniform_sz0(lat, 600, 2)).cuda()
    H = I.heisenberg(lat)
    store = 600 * 2 * 36 * 24 * 4 * 24 * 4
    lim = Limited(P, monkeypatch)
    h = P.PEPS(6, 6, 2, 4, 24, prec=1, max_samples=600)
    h.set_params(theta)
    full = h.evaluate(H, S)
    a = h.sample(S.clone(), P.MOVE_EXCHANGE, 1, seed=3, sweep0=0)[0].clone()
    h.close()
    arena = max(n for n in lim.sizes if n != store)
    lim.refuse = lambda n: n > arena // 3 and n != store
    h = P.PEPS(6, 6, 2, 4, 24, prec=1, max_samples=600)
    h.set_params(theta)
    r = h.evaluate(H, S)
    for k in ("logabs", "eloc", "O"):
        assert torch.equal(r[k], full[k])
    assert torch.equal(h.sample(S.clone(), P.MOVE_EXCHANGE, 1, seed=3, sweep0=0)[0], a)
    h.close()


def test_direct_sampling_after_a_refused_prepare(P, monkeypatch):
    lat = I.Lattice(4, 4, 2, 2)
    theta = torch.as_tensor(I.peps_random(lat, 1, scale=0.5, bias=1.0)).cuda()
    lim = Limited(P, monkeypatch)
    for k in range(4):
        h = P.PEPS(4, 4, 2, 2, 4, prec=0, max_samples=8)
        h.set_params(theta)
        h.direct_prepare(2)
        first = h.direct_sample(8, seed=1)[0].clone()
        calls = []

        def from_kth(n):
            calls.append(n)
            return len(calls) > k

        lim.refuse = from_kth
        try:
            h.direct_prepare(8)
        except RuntimeError as e:
            assert "PEPS_E_WORKSPACE" in str(e)
            with pytest.raises(RuntimeError, match="PEPS_E_ARG"):
                h.direct_sample(8, seed=1)
        lim.refuse = lambda n: False
        h.direct_prepare(2)
        assert torch.equal(h.direct_sample(8, seed=1)[0], first)
        h.close()
