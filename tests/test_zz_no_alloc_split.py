"""The allocation-free update where its blocks share out the transfers and the
momentum pairs: one group of 128 sites, transfers that do not divide into the
steps dealt, one site at the largest frequency count."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs

from gpu_util import cuda, draw, ensure_built, oracle_full

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 8, 1, 1, 1), (8, 8, 2, 9, 1), (5, 5, 4, 7, 2), (1, 1, 64, 64, 1),
                                   (7, 7, 2, 4, 5)], ids=lambda s: "%dx%d_%d_%d_%d" % s)
def test_against_oracle(shape):
    Lx, Ly, Nw, Nwex, Nkex = shape
    torch, g4 = cuda(), ensure_built()
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 10.0, 2, 2, h=0.2)
    M, G0, s = draw(p, seed=12)
    s = np.array([1.0, -0.5])
    ref, S = oracle_full(p, M, G0, s)
    acc = torch.zeros(p.entries, dtype=torch.complex128, device="cuda")
    G0d = torch.from_numpy(G0).cuda()
    for r in range(2):
        g4.update_noalloc(p.Nc, p.Nw, p.Nwex, p.Nkex, M[r].cuda(), G0d, s[r], acc, lx=p.Lx)
    got = acc.cpu().numpy() / S
    assert oracle.errors(ref.reshape(-1), got)["L2"] <= 1e-11
