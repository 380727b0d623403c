"""The row step and the sandwiches on the bonds that are not zero: states whose truncations keep a few
rows (the one-warp Jacobi, matrices in the scratch) and all of them (the block Jacobi, matrices in
the arena), at row lengths with and without a remainder, against the oracle; and results that do not
depend on how many threads and CTAs a batch of its size is given.

Tolerance: FP64 results agree with the oracle to 1e-10 (as in test_gpu_parity).
"""
import numpy as np
import pytest
import torch

from paper_2503_12557_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2503_12557_gb300 import build, peps
    build.build()
    return peps


# (Lx, Ly, D, chi, init): decaying legs leave few singular values, isotropic tensors all of them
SHAPES = [
    (4, 5, 2, 3, dict(scale=0.5, bias=1.0, alpha=1.5)),    # row length 6 < one chunk of eight
    (5, 4, 3, 7, dict(scale=0.5, bias=1.0, alpha=3.0)),    # row length 21
    (5, 5, 3, 7, dict(scale=1.0)),                         # 9 to 21 active rows
    (4, 6, 4, 16, dict(scale=0.5, bias=1.0, alpha=3.0)),   # the compiled shape, few active rows
    (4, 6, 4, 16, dict(scale=1.0)),                        # the same, every row active
    (4, 4, 5, 26, dict(scale=1.0)),                        # row length 130: the long-row Jacobi
]


@pytest.mark.parametrize("Lx,Ly,D,chi,init", SHAPES)
def test_bonds_vs_oracle(P, Lx, Ly, D, chi, init):
    from oracle import energy
    lat = I.Lattice(Lx, Ly, 2, D)
    th = I.peps_random(lat, 71, **init)
    S = I.configs_uniform_sz0(lat, 12, 72)
    H = I.heisenberg(lat)
    h = P.PEPS(Lx, Ly, 2, D, chi, prec=P.PREC_FP64, max_samples=12)
    h.set_params(torch.as_tensor(th).cuda())
    res = h.evaluate(H, torch.as_tensor(S).cuda())
    torch.cuda.synchronize()
    ref = energy.evaluate(th, S, lat, chi, H=H, want_O=True)
    ok = (np.asarray(ref["status"]) & 1) == 0
    assert ok.any()
    assert np.max(np.abs(res["logabs"].cpu().numpy() - ref["logabs"])[ok]) <= 1e-10
    el = res["eloc"].cpu().numpy()
    de = np.abs(el[:, 0] + 1j * el[:, 1] - ref["eloc"]) / np.maximum(1.0, np.abs(ref["eloc"]))
    assert np.max(de[ok]) <= 1e-10
    O, Or = res["O"].cpu().numpy(), ref["O"].real
    assert np.max((np.max(np.abs(O - Or), axis=1) / np.maximum(1.0, np.max(np.abs(Or), axis=1)))[ok]) <= 1e-10


@pytest.mark.parametrize("D,chi", [(4, 16), (3, 9), (4, 24)])
def test_results_do_not_depend_on_the_batch(P, D, chi):
    # 40 samples alone (large CTAs) and first in a batch of 1000 (small ones): the same bits
    lat = I.Lattice(4, 5, 2, D)
    th = torch.as_tensor(I.peps_random(lat, 73, scale=0.5, bias=1.0, alpha=1.5)).cuda()
    S = torch.as_tensor(I.configs_uniform_sz0(lat, 1000, 74)).cuda()
    H = I.heisenberg(lat)
    out = []
    for ns in (40, 1000):
        h = P.PEPS(lat.Lx, lat.Ly, 2, D, chi, prec=P.PREC_FP32, max_samples=ns)
        h.set_params(th)
        r = h.evaluate(H, S[:ns])
        C = S[:ns].clone()
        h.sample(C, P.MOVE_EXCHANGE, 2, seed=75, sweep0=0)
        out.append([r[k][:40].cpu() for k in ("logabs", "phase", "eloc", "O")] + [C[:40].cpu()])
    for a, b in zip(*out):
        assert torch.equal(a, b)
