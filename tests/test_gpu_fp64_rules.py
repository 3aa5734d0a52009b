"""The FP64 path's kernels on both sides of the rules that choose them: tiled or
one thread per entry (how much of the 16 x 16 frequency tiles lies on the grid),
tensor cores or not (few transfer momenta, few measurements), batches of one and
more, transfers beyond the grid."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import TOL, check_entries, draw, exported_to_slabs, oracle_full, run_lib

pytestmark = pytest.mark.gpu

SHAPES = [
    # Lx, Ly, Nw, Nwex, Nkex, R, batch: E from 2^18 on unless the last two
    (8, 4, 1, 2, 32, 3, 1), (8, 2, 2, 6, 16, 5, 5), (4, 4, 6, 2, 16, 4, 2), (4, 4, 7, 2, 8, 4, 4),
    (4, 4, 8, 1, 8, 3, 3), (3, 3, 14, 3, 3, 2, 1), (3, 3, 17, 2, 2, 6, 6), (16, 16, 1, 1, 2, 8, 8),
    (4, 2, 3, 2, 3, 9, 3), (2, 1, 2, 7, 2, 20, 20),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d_%d_%d_%d_%d_%d" % s)
@pytest.mark.parametrize("channel", ["ph_magnetic", "ph_density", "ph_transverse", "pp_updown"])
def test_against_oracle(shape, channel):
    Lx, Ly, Nw, Nwex, Nkex, R, batch = shape
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, R, batch, h=0.2)
    M, G0, s = draw(p, seed=15)
    s = np.linspace(-0.5, 1.5, R)
    ref, _ = oracle_full(p, M, G0, s, channel=channel)
    got, _, h = run_lib(p, M, G0, s, "fp64", channel=channel)
    h.close()
    assert oracle.errors(ref, got)["L2"] <= TOL["fp64"]
    ref_s, msel = exported_to_slabs(p, ref)
    got_s, _ = exported_to_slabs(p, got)
    check_entries(p, ref_s, got_s, msel, TOL["fp64"], channel=channel)
