"""A chain whose amplitude is not a number: u < |psi'/psi|^2 is false for every u, so no move is taken
(oracle/sampler.py: _accept), and the status says that the sample is not finite."""
import numpy as np
import pytest
import torch

from paper_2503_12557_gb300 import inputs as I
from oracle.sampler import _accept

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("move", ["flip", "exchange"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_no_move_from_a_non_finite_amplitude(prec, move, bad):
    from paper_2503_12557_gb300 import peps as P
    assert not _accept(0.0, 0.0, float("nan"))
    lat = I.Lattice(4, 4, 2, 2)
    theta = np.array(I.peps_random(lat, 91, scale=0.5, bias=1.0))
    blk = (I.site_offsets(lat)[1] - I.site_offsets(lat)[0]) // 2
    theta[:blk] = bad                       # site 0 in state 0
    S = torch.as_tensor(I.configs_uniform_sz0(lat, 16, 92)).cuda()
    S[:8, 0] = 0
    S[8:, 0] = 1
    h = P.PEPS(4, 4, 2, 2, 4, prec=prec, max_samples=16)
    h.set_params(torch.as_tensor(theta).cuda())
    before = S.clone()
    r = h.sample(S, P.MOVE_FLIP if move == "flip" else P.MOVE_EXCHANGE, 2, seed=5, sweep0=0)
    after, acc = r[0], r[1]
    assert torch.equal(after[:8], before[:8])
    assert torch.all(acc[:8] == 0)
    assert torch.all(after[8:, 0] == 1)     # and none moves there
    h.close()
