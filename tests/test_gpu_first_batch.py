"""A run's first batch writes the accumulator instead of adding to a cleared
one.  A handle that still holds another run's values must give a new run's
result to the last bit, structural zeros included, whichever call comes first
after the reset: a batch, the export, a checkpoint, a restore or a grouped
accumulation."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import (TOL, check_entries, cuda, draw, ensure_built, exported_to_slabs, oracle_full,
                      run_lib)

pytestmark = pytest.mark.gpu

CASES = [
    # Lx, Ly, Nw, Nwex, Nkex, R, batch, kw
    (1, 1, 1, 3, 1, 3, 4, {}),                                   # Nwex > 2Nw
    (3, 3, 3, 5, 7, 9, 4, {}),                                   # Nkex < Nc
    (4, 2, 5, 4, 8, 6, 4, dict(channel="pp_updown")),
    (5, 1, 4, 2, 3, 6, 4, dict(channel="ph_transverse", deferred=True)),
    (2, 2, 9, 12, 4, 6, 4, dict(channel="ph_density", operands="tf32")),
    (4, 4, 2, 1, 16, 6, 6, dict(deferred=True)),
    (2, 2, 6, 6, 4, 6, 4, dict(wex_slab=(2, 3))),                # a slab of the transfers
    (2, 2, 4, 3, 4, 6, 4, dict(accum="f32pair")),
]


def dirty(p, kw):
    """A handle whose accumulator holds a run of large values."""
    M, G0, s = draw(p, seed=1)
    _, _, h = run_lib(p, M * 1e3, G0, s, "mixed", **kw)
    return h


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d_%d_%d" % c[:4])
def test_reset_leaves_nothing(case, tmp_path):
    torch = cuda()
    Lx, Ly, Nw, Nwex, Nkex, R, batch, kw = case
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, R, batch)
    M, G0, s = draw(p, seed=2)
    s = np.where(np.arange(R) == 1, -0.5, 1.0)
    h = dirty(p, kw)
    h.reset()
    got, S, h = run_lib(p, M, G0, s, "mixed", handle=h, **kw)
    want, _, h2 = run_lib(p, M, G0, s, "mixed", **kw)
    h2.close()
    assert np.array_equal(got, want)
    if "wex_slab" not in kw:
        channel = kw.get("channel", "ph_magnetic")
        ref, _ = oracle_full(p, M, G0, s, channel=channel)
        assert oracle.errors(ref, got)["L2"] <= TOL["mixed"]
        ref_s, msel = exported_to_slabs(p, ref)
        got_s, _ = exported_to_slabs(p, got)
        check_entries(p, ref_s, got_s, msel, TOL["mixed"], channel)
    # nothing staged: the export and a checkpoint are zero
    path = str(tmp_path / "zero.ckpt")
    h.reset()
    h.checkpoint(path)
    h.reset()
    out, S = h.finalize(allow_zero_sign=True)
    assert S == 0.0 and not bool(torch.any(out != 0))
    # a restore of the empty run into a handle with other values, then the run
    h.reset()
    h.restore(path)
    again, _, h = run_lib(p, M, G0, s, "mixed", handle=h, **kw)
    h.close()
    assert oracle.errors(want, again)["L2"] <= 1e-14


def test_grouped_first_batch():
    torch = cuda()
    g4 = ensure_built()
    ps = [inputs.Problem(2, 2, 3, 2, 4, 8.0, 8, 4), inputs.Problem(3, 1, 4, 3, 2, 8.0, 8, 4)]
    data = [draw(p, seed=4, problem_index=i) for i, p in enumerate(ps)]
    hs = [dirty(p, {}) for p in ps]
    G0s = [torch.from_numpy(np.ascontiguousarray(d[1])).cuda() for d in data]
    outs = []
    for run in range(2):     # the second run replays both graphs
        for h in hs:
            h.reset()
        for r0 in (0, 4):
            for h, (M, G0, s), g0 in zip(hs, data, G0s):
                for r in range(r0, r0 + 4):
                    h.compute_G(M[r].cuda(), g0, 1.0)
            g4.accumulate_group(hs)
        outs.append([h.finalize()[0].cpu().numpy() for h in hs])
    for i, (p, (M, G0, s)) in enumerate(zip(ps, data)):
        assert np.array_equal(outs[0][i], outs[1][i])
        ref, _ = oracle_full(p, M, G0, np.ones(8))
        assert oracle.errors(ref, outs[1][i])["L2"] <= TOL["mixed"]
        hs[i].close()
