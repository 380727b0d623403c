"""Handles of one scalar type share their kernels' dynamic shared-memory limit: creating a handle with a
smaller plan must not lower it for the others, in whatever order they are made."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, torch
from paper_2503_12557_gb300 import inputs as I, peps as P

def make(L, D, chi, prec):
    lat = I.Lattice(L, L, 2, D)
    h = P.PEPS(L, L, 2, D, chi, prec=prec, cplx=True, max_samples=4)
    h.set_params(torch.as_tensor(I.peps_random(lat, 1, scale=0.3, bias=1.0, complex_=True)).cuda())
    return h, torch.as_tensor(I.configs_uniform_sz0(lat, 4, 2)).cuda()

for prec in (P.PREC_FP32, P.PREC_FP64):
    big, S = make(4, 6, 36, prec)
    first = big.amplitudes(S)[0].clone()
    small, S2 = make(4, 4, 16, prec)      # a shape that real handles have compiled kernels for
    small.amplitudes(S2)
    again, _ = make(4, 6, 36, prec)
    assert torch.equal(again.amplitudes(S)[0], first)
    assert torch.equal(big.amplitudes(S)[0], first)
    for h in (big, small, again):
        h.close()
"""


def test_large_complex_handle_after_a_small_one():
    # in its own process: the limits outlive a handle, and earlier tests may have raised them
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
