"""The mixed path's G build at the edges of its 32-column blocks: fewer columns
than a block, a last block that is not full, blocks that span several momenta,
the largest frequency count, and a complex64 M on an 8-byte boundary; each
against the oracle, with the mixed path's bounds."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import TOL, check_entries, cuda, ensure_built, draw, exported_to_slabs, oracle_full

pytestmark = pytest.mark.gpu

SHAPES = [
    (1, 1, 1, 1, 1),      # two columns
    (2, 1, 3, 2, 2),      # 12 columns of two momenta in one block
    (3, 1, 5, 2, 2),      # 30
    (3, 3, 2, 3, 9),      # 36: eight momenta in the first block, a second block of four columns
    (5, 1, 17, 3, 2),     # 170 columns of 34 frequencies
    (1, 2, 64, 2, 2),     # 128 frequencies
]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("m_dtype", ["c128", "c64"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d_%d" % s[:3])
def test_against_oracle(shape, m_dtype, offset):
    torch = cuda()
    g4 = ensure_built()
    Lx, Ly, Nw, Nwex, Nkex = shape
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, 5, 3, m_dtype=m_dtype)
    M, G0, s = draw(p, seed=11)
    h = g4.G4.for_problem(p)
    G0d = torch.from_numpy(np.ascontiguousarray(G0)).cuda()
    for r in range(p.R):
        # one entry further into a buffer: complex64 rows then start at 8 mod 16 bytes
        buf = torch.empty(M[r].numel() + offset, dtype=M[r].dtype, device="cuda")
        view = buf[offset:].view(M[r].shape)
        view.copy_(M[r])
        h.compute_G(view, G0d, float(s[r]))
    got, S = h.finalize(allow_zero_sign=True)
    got = got.cpu().numpy()
    h.close()
    ref, Sref = oracle_full(p, M, G0, s)
    assert S == Sref
    assert oracle.errors(ref, got)["L2"] <= TOL["mixed"]
    ref_s, msel = exported_to_slabs(p, ref)
    got_s, _ = exported_to_slabs(p, got)
    check_entries(p, ref_s, got_s, msel, TOL["mixed"])
