"""The allocation-free update against the oracle where its blocks can go wrong:
one site (256 planes per block), clusters whose Nc^2 entries exceed a block,
planes that do not divide it, transfer frequencies beyond one step of four and
up to the grid's size."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs

from gpu_util import cuda, draw, ensure_built, oracle_full

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 20, 7, 1), (5, 5, 5, 6, 13), (17, 1, 3, 6, 17),
                                   (16, 8, 1, 2, 9), (3, 2, 4, 8, 5), (4, 4, 8, 1, 16)],
                         ids=lambda s: "%dx%d_%d_%d_%d" % s)
def test_against_oracle(shape):
    Lx, Ly, Nw, Nwex, Nkex = shape
    torch, g4 = cuda(), ensure_built()
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 10.0, 3, 3, h=0.2)
    M, G0, s = draw(p, seed=11)
    s = np.array([1.0, -1.0, 0.75])
    ref, S = oracle_full(p, M, G0, s)
    acc = torch.zeros(p.entries, dtype=torch.complex128, device="cuda")
    G0d = torch.from_numpy(G0).cuda()
    for r in range(3):
        g4.update_noalloc(p.Nc, p.Nw, p.Nwex, p.Nkex, M[r].cuda(), G0d, s[r], acc, lx=p.Lx)
    got = acc.cpu().numpy() / S
    assert oracle.errors(ref.reshape(-1), got)["L2"] <= 1e-11
