"""The FP64 path's batch update on tensor cores (seven base-256 digits per
operand) against the oracle, at the edges of its tiles and chunks.

Tolerance 2e-14 (relative Frobenius).  Per product the digits lose at most
3 x 2^-55 of the product of the two operand rows' largest values (two 54-bit
roundings and the dropped levels); with rows whose largest value is at most
eight times their r.m.s. that is 64 x 3 x 2^-55 = 5e-15 of the r.m.s. product,
added over independent terms; the oracle's own FP64 sums of up to 130 terms
add at most 130 x 2^-53 = 1.4e-14."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs

from gpu_util import check_entries, draw, exported_to_slabs, oracle_full, run_lib

pytestmark = pytest.mark.gpu

TOL = 2e-14

CASES = [
    # Lx, Ly, Nw, Nwex, Nkex, R, batch, channel
    (3, 3, 9, 5, 7, 37, 16, "ph_magnetic"),       # one chunk for both spins, a ragged last batch
    (3, 3, 9, 5, 7, 17, 17, "ph_density"),        # two chunks
    (4, 2, 8, 3, 8, 64, 64, "ph_magnetic"),       # the largest batch
    (4, 2, 8, 3, 8, 50, 64, "ph_transverse"),     # spins exchanged, the second chunk partly filled
    (5, 1, 13, 16, 5, 40, 40, "pp_updown"),       # the widest window
    (5, 3, 6, 1, 15, 33, 33, "ph_density"),       # one transfer frequency
    (2, 1, 33, 7, 2, 64, 48, "pp_updown"),        # 66 frequencies, a batch off the chunk size
    (7, 3, 4, 2, 11, 20, 20, "ph_magnetic"),      # two row-momentum blocks at some tile shapes
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d_%d_%s" % (c[0], c[1], c[6], c[7]))
def test_against_oracle(case):
    Lx, Ly, Nw, Nwex, Nkex, R, batch, channel = case
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 10.0, R, batch, h=0.3)
    assert p.entries * min(R, batch) >= 4e6     # the path's threshold
    M, G0, s = draw(p, seed=3)
    s = s * np.linspace(0.5, 1.5, R)     # signs other than +-1
    ref, S = oracle_full(p, M, G0, s, channel=channel)
    got, S_dev, h = run_lib(p, M, G0, s, "fp64", channel=channel)
    h.close()
    err = oracle.errors(ref, got)
    print("L2 %.3e" % err["L2"])
    assert err["L2"] <= TOL, err
    ref_s, msel = exported_to_slabs(p, ref)
    got_s, _ = exported_to_slabs(p, got)
    check_entries(p, ref_s, got_s, msel, 1e-13, channel=channel)


@pytest.mark.parametrize("scale", [1e-30, 1e40, 1e130])
def test_range(scale):
    """M far from 1; 1e130 leaves the digits' exponent range and takes the plain kernels."""
    p = inputs.Problem(3, 3, 9, 5, 7, 10.0, 24, 24)
    M, G0, s = draw(p, seed=5)
    M = M * scale
    M[3] *= 1e-3
    ref, S = oracle_full(p, M, G0, s)
    got, S_dev, h = run_lib(p, M, G0, s, "fp64")
    h.close()
    unit = float(np.abs(ref).max())
    assert oracle.errors(ref / unit, got / unit)["L2"] <= TOL
