"""g4_finalize to the device (the direct term's last window added on the way)
against the same run finalised to host memory (the window added to the
accumulator first, then blocks of n2 planes): the same sums in the same order,
so the same bits.  Sizes at the edges of the export's blocks: one momentum, n2
counts that are not a multiple of four, transfers that do not fill a block or a
group of sixteen, more transfers than one group, a partly filled last group."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import TOL, cuda, draw, oracle_full, run_lib

pytestmark = pytest.mark.gpu

CASES = [
    # Lx, Ly, Nw, Nwex, Nkex, R, batch, kw
    (1, 1, 1, 1, 1, 5, 4, {}),
    (1, 1, 3, 9, 1, 5, 4, {}),                            # Nwex > 2Nw, one momentum
    (3, 1, 5, 3, 3, 9, 4, dict(channel="ph_density")),
    (3, 3, 3, 5, 7, 9, 4, dict(direct_batches=1)),        # 15 transfers a group, three groups
    (4, 4, 3, 1, 16, 9, 4, {}),                           # eight momenta per block
    (4, 2, 5, 2, 7, 9, 4, dict(deferred=True)),           # a last block of three momenta
    (2, 2, 9, 18, 3, 5, 4, {}),                           # more than sixteen per momentum
    (5, 2, 3, 6, 9, 9, 4, dict(accum="f32pair")),
    (3, 2, 3, 7, 5, 9, 4, dict(channel="pp_updown")),     # no direct term
    (3, 2, 5, 10, 5, 9, 4, dict(precision="fp64")),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d_%d_%d" % c[:4])
def test_device_equals_host(case, tmp_path):
    torch = cuda()
    Lx, Ly, Nw, Nwex, Nkex, R, batch, kw = case
    kw = dict(kw)
    precision = kw.pop("precision", "mixed")
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, R, batch)
    M, G0, s = draw(p, seed=7)
    s = np.linspace(0.5, 1.5, R) * np.where(np.arange(R) % 3 == 1, -1, 1)
    got, S, h = run_lib(p, M, G0, s, precision, **kw)
    ref, Sref = oracle_full(p, M, G0, s, channel=kw.get("channel", "ph_magnetic"))
    assert oracle.errors(ref, got)["L2"] <= TOL[precision]
    host = torch.empty(p.entries, dtype=torch.complex128).pin_memory()
    want, _, h2 = run_lib(p, M, G0, s, precision, out=host, **kw)
    h2.close()
    assert np.array_equal(got.reshape(-1), want.reshape(-1))
    # a checkpoint taken after the finalised run still holds all of it
    path = str(tmp_path / "g4.ckpt")
    h.checkpoint(path)
    h.reset()
    h.restore(path)
    again, _ = h.finalize()
    h.close()
    assert np.array_equal(again.cpu().numpy().reshape(-1), got.reshape(-1))
