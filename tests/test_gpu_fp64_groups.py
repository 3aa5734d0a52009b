"""The FP64 path's batch update on tensor cores: operands formed in several
groups of diagonals, slabs of the transfers, vertex input, and runs that are
saved and go on elsewhere.

Both forms' sums are compared entry by entry with a tolerance of 2e-14 of the
slab's largest entry: at most 2 x 20 terms per entry, each form within 40 x
2^-53 x (the sum of the products' moduli), which for the diagonal entries that
are largest is the entry itself up to a factor of two."""
import numpy as np
import pytest

from paper_2105_00027_gb300 import inputs
from gpu_util import check_entries, cuda, draw, ensure_built, exported_to_slabs, run_lib

pytestmark = pytest.mark.gpu

PLAIN = dict(mem_limit=1 << 40)     # a handle with a memory limit has the plain kernels alone


@pytest.mark.parametrize("channel", ["ph_magnetic", "ph_density", "ph_transverse", "pp_updown"])
def test_groups_of_diagonals(channel):
    """1143 diagonals of 3.5 MB each, 0.8 GB for them: several groups."""
    p = inputs.Problem(3, 3, 32, 2, 9, 10.0, 20, 64)
    M, G0, s = draw(p, seed=7)
    s = np.linspace(0.5, 1.5, 20)
    want, _, h = run_lib(p, M, G0, s, "fp64", channel=channel, **PLAIN)
    h.close()
    got, _, h = run_lib(p, M, G0, s, "fp64", channel=channel)
    h.close()
    ref_s, msel = exported_to_slabs(p, want)
    got_s, _ = exported_to_slabs(p, got)
    check_entries(p, ref_s, got_s, msel, 2e-14, channel=channel)


P0 = inputs.Problem(3, 3, 9, 5, 7, 10.0, 24, 8)


@pytest.mark.parametrize("channel", ["ph_magnetic", "pp_updown"])
def test_slab(channel):
    """Exact sums: a slab of the transfers has the whole handle's bits."""
    p = inputs.with_(P0, batch=24)
    M, G0, s = draw(p, seed=8)
    whole, _, h = run_lib(p, M, G0, s, "fp64", channel=channel)
    h.close()
    for first, count in ((0, 3), (2, 3)):
        h = ensure_built().G4.for_problem(p, precision="fp64", channel=channel, wex_slab=(first, count))
        h.profile()
        part, _, h = run_lib(p, M, G0, s, "fp64", channel=channel, handle=h)
        assert h.profile_read("exchange")[1] > 0     # the tensor-core form
        h.close()
        assert np.array_equal(part.reshape(count, -1), whole.reshape(p.Nwex, -1)[first:first + count])


def test_vertices():
    """A run fed from vertex configurations has the bits of one fed with their M."""
    torch = cuda()
    g4 = ensure_built()
    p = P0
    h = g4.G4.for_problem(p, precision="fp64")
    G0 = torch.from_numpy(np.ascontiguousarray(inputs.g0(p))).cuda()
    n = 12
    gen = torch.Generator(device="cuda").manual_seed(3)
    tau = (torch.rand(2 * n, generator=gen, dtype=torch.float64, device="cuda")) * p.beta
    site = torch.randint(0, p.Nc, (2 * n,), generator=gen, dtype=torch.int32, device="cuda")
    Xs = [torch.randn((2, n, n), generator=gen, dtype=torch.float64, device="cuda") for _ in range(p.R)]
    for X in Xs:
        h.compute_G_vertices(p.beta, n, n, tau, site, X, G0, 1.0)
    want, _ = h.finalize()
    Ms = [h.vertex_M(p.beta, n, n, tau, site, X) for X in Xs]
    h.reset()
    for M in Ms:
        h.compute_G(M, G0, 1.0)
    got, _ = h.finalize()
    h.close()
    assert torch.equal(got, want)


@pytest.mark.parametrize("begun", ["tensor", "plain"])
def test_restored_run_keeps_its_kernels(begun, tmp_path):
    """A run goes on bit for bit after a restore into a handle whose own choice
    may be the other form, until its next reset."""
    p = P0
    M, G0, s = draw(p, seed=9)
    kw = PLAIN if begun == "plain" else {}
    want, _, h = run_lib(p, M, G0, s, "fp64", **kw)
    h.close()
    other, _, h = run_lib(p, M, G0, s, "fp64", **({} if kw else PLAIN))
    h.close()
    assert not np.array_equal(want, other)      # the two forms differ in the last bits
    g4 = ensure_built()
    torch = cuda()
    G0d = torch.from_numpy(np.ascontiguousarray(G0)).cuda()
    h = g4.G4.for_problem(p, precision="fp64", **kw)
    for r in range(16):
        h.compute_G(M[r].cuda(), G0d, float(s[r]))
    h.checkpoint(tmp_path / "a.ckpt")
    h.close()
    h = g4.G4.for_problem(p, precision="fp64")
    h.restore(tmp_path / "a.ckpt")
    for r in range(16, 24):
        h.compute_G(M[r].cuda(), G0d, float(s[r]))
    got = h.finalize()[0].cpu().numpy()
    assert np.array_equal(got, want)
    h.reset()
    again, _, h = run_lib(p, M, G0, s, "fp64", handle=h)
    h.close()
    assert np.array_equal(again, want if begun == "tensor" else other)
