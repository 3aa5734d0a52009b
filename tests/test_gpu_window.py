"""A checkpoint after a full direct-term window holds no window: it goes into a
handle whose window is smaller."""
import numpy as np
import pytest

import oracle
from paper_2105_00027_gb300 import inputs
from gpu_util import TOL, cuda, draw, ensure_built, oracle_full

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deferred", [False, True])
def test_full_window_is_added_before_a_checkpoint(deferred, tmp_path):
    torch = cuda()
    g4 = ensure_built()
    p = inputs.Problem(2, 2, 4, 3, 4, 10.0, 72, 32)
    M, G0, s = draw(p, seed=3)
    Md, G0d = M.cuda(), torch.from_numpy(np.ascontiguousarray(G0)).cuda()
    a = g4.G4.for_problem(p, precision="mixed", direct_batches=2, deferred=deferred)   # 64 measurements
    b = g4.G4.for_problem(p, precision="mixed", direct_batches=1, deferred=deferred)   # 32
    for r in range(64):
        a.compute_G(Md[r], G0d, float(s[r]))
    a.checkpoint(tmp_path / "w.ckpt")
    b.restore(tmp_path / "w.ckpt")
    outs = []
    for h in (a, b):
        for r in range(64, 72):
            h.compute_G(Md[r], G0d, float(s[r]))
        outs.append(h.finalize()[0].cpu().numpy())
        h.close()
    assert np.array_equal(outs[0], outs[1])
    ref, _ = oracle_full(p, M, G0, s)
    assert oracle.errors(ref, outs[0])["L2"] <= TOL["mixed"]
