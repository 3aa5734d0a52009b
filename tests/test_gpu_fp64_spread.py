"""The FP64 path where the measurements of a batch, or their spins, differ in
size: every entry to FP64 accuracy of the products that are summed for it, not
of the largest values of the batch.

An entry's bound is 4 (2R + 8) 2^-53 S, S the sum of the moduli of its products
(2R exchange products and R direct ones): the reference, summed in FP64 in any
order, is off by at most sqrt(2) (2R + 4) 2^-53 S, the plain kernels by the
same, and the digit sums of rows within the allowed spread by less."""
import numpy as np
import pytest

from paper_2105_00027_gb300 import inputs
from gpu_util import cuda, draw, ensure_built

pytestmark = pytest.mark.gpu

R = 8
P = inputs.Problem(3, 3, 9, 5, 7, 10.0, R, R)


def reference(p, G, s, channel):
    """(G4, sum of the moduli of its products), exported layout, both over sum s."""
    import torch
    W, N, Nc = p.Nw2, p.N, p.Nc
    k = np.arange(Nc)
    kx, ky = k % p.Lx, k // p.Lx
    sg = torch.from_numpy(np.asarray(s)).cuda().reshape(-1, 1, 1)
    pp, trans = channel == "pp_updown", channel == "ph_transverse"
    ws = {"ph_magnetic": -1.0, "ph_density": 1.0}.get(channel)
    out = torch.zeros((2, p.Nwex, W, W, p.Nkex, Nc, Nc), dtype=torch.complex128, device="cuda")
    for q in range(p.Nkex):
        for m in range(p.Nwex):
            n = np.arange(W)
            f = m + W - 1 - n if pp else n + m
            kq = ((kx[q] - kx) % p.Lx + p.Lx * ((ky[q] - ky) % p.Ly) if pp
                  else (kx + kx[q]) % p.Lx + p.Lx * ((ky + ky[q]) % p.Ly))
            ok = torch.from_numpy(np.tile(f < W, Nc)).cuda()
            K = torch.from_numpy((kq[:, None] * W + np.minimum(f, W - 1)[None]).reshape(-1)).cuda()
            val = torch.zeros((N, N), dtype=torch.complex128, device="cuda")
            mod = torch.zeros((N, N), dtype=torch.float64, device="cuda")
            for sp in range(2):
                F = G[:, sp][:, K][:, :, K]
                F = F.transpose(1, 2) if pp else F
                X = G[:, 1 - sp if (pp or trans) else sp].transpose(1, 2)
                val += (X * F * (sg if pp else -sg)).sum(0)
                mod += (X.abs() * F.abs() * sg.abs()).sum(0)
            if ws is not None:
                C = G[:, 0] + ws * G[:, 1]
                j = torch.arange(N, device="cuda")
                a, b = C[:, K, j], C[:, j, K]
                val += (a[:, :, None] * b[:, None, :] * sg).sum(0)
                mod += (a.abs()[:, :, None] * b.abs()[:, None, :] * sg.abs()).sum(0)
            z = (ok[:, None] & ok[None, :])
            for i, x in enumerate((val * z, (mod * z).to(torch.complex128))):
                out[i, m, :, :, q] = x.reshape(Nc, W, Nc, W).permute(3, 1, 2, 0)
    return out[0] / float(np.sum(s)), out[1].real / abs(float(np.sum(s)))


def check(M, G0, s, channel):
    torch = cuda()
    g4 = ensure_built()
    Md, G0d = M.cuda(), torch.from_numpy(np.ascontiguousarray(G0)).cuda()
    G = torch.stack([g4.build_G(Md[r].contiguous(), G0d) for r in range(R)])
    ref, S = reference(P, G, s, channel)
    h = g4.G4.for_problem(P, precision="fp64", channel=channel)
    h.profile()
    for r in range(R):
        h.compute_G(Md[r], G0d, float(s[r]))
    got, _ = h.finalize()
    assert h.profile_read("exchange")[1] > 0     # the tensor-core form (unless its check leaves the batch)
    h.close()
    err = (got.reshape(ref.shape) - ref).abs()
    assert bool((err <= 4 * (2 * R + 8) * 2.0 ** -53 * S).all()), float((err / S.clamp_min(1e-300)).max())


@pytest.mark.parametrize("channel", ["ph_transverse", "pp_updown"])
@pytest.mark.parametrize("eps", [1.0, 1e-3, 1e-6, 1e-9])
def test_spin_imbalance(channel, eps):
    """One spin's G smaller than the other's."""
    M, G0, s = draw(P, seed=11)
    M, G0 = M.clone(), G0.copy()
    M[:, 1] /= eps
    G0[1] *= eps
    check(M, G0, np.linspace(0.5, 1.5, R), channel)


@pytest.mark.parametrize("channel", ["ph_magnetic", "ph_density", "ph_transverse", "pp_updown"])
@pytest.mark.parametrize("bits", [5, 20])
def test_large_values_in_different_measurements(channel, bits):
    """The rows of two halves of G are large in two different measurements."""
    M, G0, s = draw(P, seed=12)
    M = M.clone()
    M[1, :, :P.N // 2] *= 2.0 ** bits
    M[2, :, P.N // 2:] *= 2.0 ** bits
    check(M, G0, np.ones(R), channel)


def test_tiled_kernel_rounds_once_per_measurement():
    """The plain tiled kernel against the digit sums (error below 4e-17 S here)
    on one batch of 64 measurements.  A sum that is rounded once per measurement
    is off by at most 2^-53 |partial sum| each time, 0.41 of it in the mean; with
    partial sums growing evenly to S that is 0.41 x 2^-53 sqrt(64 / 3) S = 2.1e-16 S
    over independent roundings, in the mean over the entries.  (Twelve roundings
    per measurement, one per multiply-add, would be sqrt(12) times that bound.)"""
    torch = cuda()
    g4 = ensure_built()
    p = inputs.Problem(4, 4, 16, 4, 4, 20.0, 64, 64)
    M = torch.empty((64, 2, p.N, p.N), dtype=torch.complex128, device="cuda")
    inputs.fill_M_device(M, seed=7)
    G0 = torch.from_numpy(np.ascontiguousarray(inputs.g0(p))).cuda()
    outs = []
    for kw in ({}, dict(mem_limit=1 << 40)):     # with a memory limit: the plain kernels
        h = g4.G4.for_problem(p, precision="fp64", **kw)
        h.profile()
        for r in range(64):
            h.compute_G(M[r], G0, 1.0)
        outs.append(h.finalize()[0])
        assert (h.profile_read("exchange")[1] > 0) == (not kw)
        h.close()
    G = torch.stack([g4.build_G(M[r].contiguous(), G0) for r in range(64)])
    ref, S = reference(p, G, np.ones(64), "ph_magnetic")
    diag = lambda x: x.diagonal(dim1=1, dim2=2).diagonal(dim1=2, dim2=3)   # noqa: E731 n1 = n2, k1 = k2
    err, s = diag((outs[1] - outs[0]).abs().reshape(S.shape)), diag(S)
    rms = float(((err[s > 0] / s[s > 0]) ** 2).mean().sqrt())
    print("rms %.2e" % rms)
    assert rms <= 4.3e-16
