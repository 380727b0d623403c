"""Observables do not depend on the scale of the PEPS tensors: every tensor times 2^k multiplies psi by
2^(k sites), leaves E_loc as it is and divides O by 2^k, also where a row of tensors multiplies to
1e-90 or 1e+90 and the squares of the truncated matrices' entries leave the double range.

Tolerance: a power of two changes no mantissa, so what may differ are roundings of the truncation's
scalar arithmetic; 1e-10, as against the oracle (test_gpu_parity), on samples whose truncation is
unique (status 0).
"""
import math

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


def _evaluate(P, lat, chi, theta, S, H):
    h = P.PEPS(lat.Lx, lat.Ly, 2, lat.D, chi, prec=P.PREC_FP64, max_samples=len(S))
    h.set_params(torch.as_tensor(theta).cuda())
    r = h.evaluate(H, torch.as_tensor(S).cuda())
    out = {k: v.cpu().numpy() for k, v in r.items()}
    h.close()
    return out


# (Ly, D, chi, init): at most 8 rows (the one-warp Jacobi) and more than it takes (the block form)
SHAPES = [(14, 2, 4, dict(scale=1.0)), (10, 4, 16, dict(scale=1.0))]


@pytest.mark.parametrize("Ly,D,chi,init", SHAPES)
@pytest.mark.parametrize("k", [-23, -27, -30, 30])
def test_scaled_tensors(P, Ly, D, chi, init, k):
    lat = I.Lattice(4, Ly, 2, D)
    theta = np.asarray(I.peps_random(lat, 81, **init))
    S = I.configs_uniform_sz0(lat, 6, 82)
    H = I.heisenberg(lat)
    a = _evaluate(P, lat, chi, theta, S, H)
    b = _evaluate(P, lat, chi, np.ldexp(theta, k), S, H)
    assert np.array_equal(a["status"], b["status"])
    ok = a["status"] == 0
    assert ok.any()
    assert np.max(np.abs(b["logabs"] - a["logabs"] - k * lat.nsites * math.log(2.0))[ok]) <= 1e-10
    assert np.array_equal(a["phase"][ok], b["phase"][ok])
    de = np.linalg.norm(b["eloc"] - a["eloc"], axis=1) / np.maximum(1.0, np.linalg.norm(a["eloc"], axis=1))
    assert np.max(de[ok]) <= 1e-10
    dO = np.max(np.abs(np.ldexp(b["O"], k) - a["O"]), axis=1) / np.maximum(1.0, np.max(np.abs(a["O"]), axis=1))
    assert np.max(dO[ok]) <= 1e-10
