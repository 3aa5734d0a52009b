"""A deferred handle's first batch takes its operand scale from a read of M:
the bits an eager handle gets from the same batch, whatever the size of M, with
one G0 or one per measurement, and again after a reset."""
import numpy as np
import pytest

from paper_2105_00027_gb300 import inputs
from gpu_util import cuda, draw, run_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-6, 1.0, 3e5])
@pytest.mark.parametrize("m_dtype", ["c128", "c64"])
@pytest.mark.parametrize("own_g0", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1, 1), (3, 1, 5, 2, 2), (4, 2, 9, 3, 8)],
                         ids=lambda s: "%dx%d_%d" % s[:3])
def test_first_batch_equals_eager(shape, own_g0, m_dtype, scale):
    Lx, Ly, Nw, Nwex, Nkex = shape
    p = inputs.Problem(Lx, Ly, Nw, Nwex, Nkex, 8.0, 13, 16, m_dtype=m_dtype)
    M, G0, s = draw(p, seed=5)
    M = M * scale
    s = np.where(s < 0, -0.75, 1.0)
    want, _, h = run_lib(p, M, G0, s, "mixed", exchange="tensor_cores")
    h.close()
    got, _, h = run_lib(p, M, G0, s, "mixed", exchange="tensor_cores", deferred=True, own_g0=own_g0)
    assert np.array_equal(got, want)
    # other measurements after a reset: no scale is left over
    h.reset()
    want2, _, h2 = run_lib(p, M * 64, G0, s, "mixed", exchange="tensor_cores")
    h2.close()
    got2, _, h = run_lib(p, M * 64, G0, s, "mixed", handle=h, deferred=True, own_g0=own_g0)
    h.close()
    assert np.array_equal(got2, want2)
