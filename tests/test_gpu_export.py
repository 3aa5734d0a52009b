"""The export's two kernels and the direct term's way into it at the edges of
their rules (8, 9, 12 and 13 transfers, clusters of up to twelve sites and more,
runs of 1, 4, 9 and 16 pairs that are shorter than a warp, chunks of pairs that
do not divide the cluster's), and host output in several blocks of an odd number
of n2 planes."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import TOL, check_entries, cuda, draw, ensure_built, exported_to_slabs, oracle_full, run_lib

pytestmark = pytest.mark.gpu

SHAPES = [
    # Lx, Ly, Nw, Nwex, Nkex
    (1, 1, 6, 13, 1), (1, 1, 9, 3, 1), (2, 1, 5, 9, 2), (2, 2, 7, 10, 3), (3, 1, 8, 1, 3),
    (3, 3, 4, 8, 9), (3, 3, 5, 9, 5), (4, 3, 3, 9, 7), (4, 3, 7, 12, 3), (4, 3, 7, 13, 3),
    (5, 4, 3, 6, 11), (4, 4, 9, 18, 2),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d_%d_%d_%d" % s)
@pytest.mark.parametrize("precision,kw", [("fp64", {}), ("mixed", {}), ("mixed", dict(channel="pp_updown"))],
                         ids=["fp64", "magnetic", "pp"])
def test_against_oracle(shape, precision, kw):
    Lx, Ly, Nw, Nwex, Nkex = shape
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, 3, 3, h=0.2)
    channel = kw.get("channel", "ph_magnetic")
    M, G0, s = draw(p, seed=13)
    s = np.array([1.0, -0.5, 1.25])
    ref, _ = oracle_full(p, M, G0, s, channel=channel)
    got, _, h = run_lib(p, M, G0, s, precision, **kw)
    h.close()
    assert oracle.errors(ref, got)["L2"] <= TOL[precision]
    ref_s, msel = exported_to_slabs(p, ref)
    got_s, _ = exported_to_slabs(p, got)
    check_entries(p, ref_s, got_s, msel, TOL[precision], channel=channel)


@pytest.mark.parametrize("Nwex", [9, 14])
def test_host_output_in_odd_blocks(Nwex):
    """More than one block of 1 GB: 39 and 7, and 25 and 21 n2 planes."""
    torch = cuda()
    g4 = ensure_built()
    p = inputs.Problem(4, 4, 23, Nwex, 16, 8.0, 2, 2)
    per = p.entries // p.Nw2 * 16
    assert (1 << 30) // per < p.Nw2 and ((1 << 30) // per) % 2 == 1
    M, G0, s = draw(p, seed=14)
    Md, G0d = M.cuda(), torch.from_numpy(np.ascontiguousarray(G0)).cuda()
    h = g4.G4.for_problem(p, precision="mixed")
    outs = []
    for dev in ("cuda", "cpu"):
        h.reset()
        for r in range(2):
            h.compute_G(Md[r], G0d, 1.0)
        out = torch.empty(p.entries, dtype=torch.complex128, device=dev)
        h.finalize(out)
        outs.append(out.cpu())
    h.close()
    assert torch.equal(outs[0], outs[1])
