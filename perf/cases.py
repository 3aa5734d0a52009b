"""Performance cases: the G4 measurement step as a QMC program calls it.

A program makes one handle per G4 problem and keeps it; a pass is one run of
measurements through it: reset, one compute_G (or compute_G_vertices) per
measurement, finalize into the program's own output array.  The other kinds
are the vertex transform alone, several problems accumulated in grouped
launches, and the allocation-free update.  Sizes are the workloads of
``paper_2105_00027_gb300.inputs`` (and parts of them that leave room for
several states on one card), the tests' kind of odd clusters, and draws over
the same ranges.
"""
import math

import numpy as np
import torch

from paper_2105_00027_gb300 import g4, inputs

POOL_BYTES = 24 << 30   # distinct measurements kept on the device; longer runs cycle them


def listed():
    def run(name, Lx, Ly, Nw, Nwex, Nkex, beta, R, batch, **kw):
        c = dict(name=name, kind="run", Lx=Lx, Ly=Ly, Nw=Nw, Nwex=Nwex, Nkex=Nkex, beta=beta, R=R,
                 batch=batch, m_dtype="c128", precision="mixed", channel="ph_magnetic",
                 deferred=False, vertices=False)
        c.update(kw)
        return c

    return [
        # the smallest problem, in both precisions: 16 tiny launches and a finalize, all latency
        run("tiny_2x2_fp64", 2, 2, 4, 1, 1, 10.0, 16, 16, precision="fp64"),
        run("tiny_2x2_mixed", 2, 2, 4, 1, 1, 10.0, 16, 16),
        # the plain FP64 method on the 4x4 cluster, one batch of its 256 measurements
        run("c16_w64_fp64", 4, 4, 32, 8, 16, 20.0, 64, 64, precision="fp64"),
        # FP64 away from powers of two: 3x3 cluster, 34 frequencies, a subset of the
        # transfer momenta, density channel, a last batch that is not full
        run("c9_w34_fp64_density", 3, 3, 17, 5, 7, 5.0, 40, 16, precision="fp64",
            channel="ph_density"),
        # the same 4x4 problem on the mixed path, the whole run of 256 measurements
        run("c16_w64_mixed", 4, 4, 32, 8, 16, 20.0, 256, 64),
        # the paper's 6x6 cluster (four transfer frequencies), two batches, complex128 M
        run("c36_w64_mixed", 6, 6, 32, 4, 36, 20.0, 128, 64),
        # the 8x8 production form: complex64 M resident on the device, deferred staging,
        # batches of 128 (half the frequencies of the largest workload)
        run("c64_w32_deferred", 8, 8, 16, 4, 64, 40.0, 256, 128, m_dtype="c64", deferred=True),
        # a ragged problem in the paper's own channel (particle-particle): 5x3 cluster,
        # 50 frequencies, 11 of 15 transfer momenta, a last batch of 22
        run("c15_w50_pp", 5, 3, 25, 6, 11, 10.0, 150, 64, channel="pp_updown", m_dtype="c64"),
        # a run fed from vertex configurations (about 640 vertices per spin)
        run("c16_w64_vertices", 4, 4, 32, 8, 16, 20.0, 64, 64, vertices=True),
        # the vertex transform alone at the 8x8 size, about 5120 vertices per spin
        dict(name="vertex_M_c64_w64", kind="vertex_M", Lx=8, Ly=8, Nw=32, beta=40.0, U=4.0,
             precision="mixed"),
        # independent problems of uneven size in grouped launches, one round of batches
        # each: every cluster of 4, 8 and 16 sites with 16, 32 and 64 frequencies
        dict(name="group_c4_c16", kind="group", clusters="4,8,16", freqs="16,32,64", Nwex=4, R=64),
        # the allocation-free update at its largest size
        dict(name="noalloc_c16_w16", kind="noalloc", Lx=4, Ly=4, Nw=8, Nwex=4, Nkex=16, beta=10.0,
             R=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixed"] * 5 + ["fp64"] * 3 + ["vertices"] * 2 + ["vertex_M"] * 2 +
                      ["group", "noalloc"])
    while True:
        Lx, Ly = rng.randint(1, 8), rng.randint(1, 8)
        Nw = _log(rng, 2, 32)
        Nc, N = Lx * Ly, Lx * Ly * 2 * Nw
        Nwex = rng.randint(1, min(10, 2 * Nw))
        Nkex = Nc if rng.random() < 0.6 else rng.randint(1, Nc)
        beta = rng.choice([5.0, 10.0, 20.0, 40.0])
        E = N * N * Nwex * Nkex
        if kind == "noalloc":
            if N <= 256:
                return dict(kind=kind, Lx=Lx, Ly=Ly, Nw=Nw, Nwex=Nwex, Nkex=Nkex, beta=beta,
                            R=rng.randint(8, 32))
            continue
        if kind == "group":
            sizes = sorted(rng.sample([2, 4, 6, 8, 9, 12, 16], 3))
            freqs = sorted(rng.sample([8, 16, 20, 32, 46, 64], 2))
            return dict(kind=kind, clusters=",".join(map(str, sizes)),
                        freqs=",".join(map(str, freqs)), Nwex=rng.randint(1, 6),
                        R=rng.randint(16, 64))
        if kind == "vertex_M":
            if 64 <= N:
                return dict(kind=kind, Lx=Lx, Ly=Ly, Nw=Nw, beta=beta, U=rng.choice([2.0, 4.0, 6.0])
                            if Nc * beta <= 1200 else 4.0,
                            precision=rng.choice(["mixed", "mixed", "fp64"]) if Nc * beta <= 320
                            else "mixed")
            continue
        batch = rng.choice([8, 16, 32, 48, 64] if kind == "fp64" else [16, 40, 64, 64, 100, 128])
        R = max(8, _log(rng, 8, 256))
        if kind == "fp64" and not E * R <= 8e9:
            continue
        if kind == "vertices" and not (E * R <= 1e10 and R <= 64 and beta * Nc <= 400 and Nc > 1):
            continue
        if kind == "mixed" and not (E <= 6e8 and E * R <= 8e10 and N <= 2304):
            continue
        if N < 32:
            continue
        return dict(kind="run", Lx=Lx, Ly=Ly, Nw=Nw, Nwex=Nwex, Nkex=Nkex, beta=beta, R=R,
                    batch=batch, m_dtype=rng.choice(["c128", "c64"]),
                    precision="fp64" if kind == "fp64" else "mixed",
                    channel=rng.choice(["ph_magnetic"] * 3 + ["ph_density", "ph_transverse",
                                                              "pp_updown"]),
                    deferred=kind == "mixed" and rng.random() < 0.5,
                    vertices=kind == "vertices")


# ------------------------------------------------------------------ inputs

def _problem(c):
    return inputs.Problem(c["Lx"], c["Ly"], c["Nw"], c.get("Nwex", 1), c.get("Nkex", 1), c["beta"],
                          c.get("R", 1), c.get("batch", 1), m_dtype=c.get("m_dtype", "c128"))


def _group_problems(c):
    out = []
    for Nc in map(int, c["clusters"].split(",")):
        Lx, Ly = inputs.cluster_shape(Nc)
        for f in map(int, c["freqs"].split(",")):
            out.append(inputs.Problem(Lx, Ly, f // 2, c["Nwex"], Nc, (5.0, 10.0, 20.0)[len(out) % 3],
                                      c["R"], min(64, c["R"])))
    return out


def _signs(p, seed, index=0):
    s = inputs.signs(p, seed, index)
    if s.sum() == 0:
        s[:] = 1.0
    return s


def _pool(p):
    one = 2 * p.N * p.N * (16 if p.m_dtype == "c128" else 8)
    return max(1, min(p.R, POOL_BYTES // one))


def _M(p, seed, index=0):
    """The run's measurements: independent N(0, 1/N) real and imaginary parts."""
    dt = torch.complex128 if p.m_dtype == "c128" else torch.complex64
    M = torch.empty((_pool(p), 2, p.N, p.N), dtype=dt, device="cuda")
    return inputs.fill_M_device(M, seed=seed * 64 + index)


def _vertices(p, seed, U=4.0):
    """One vertex configuration on the device, spins sharing times and sites
    (the recipe of inputs.vertex_config)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.Generator(np.random.Philox(key=[seed, 0x5E]))
    n = max(1, int(round(inputs.vertices_per_spin(p, U) * (1.0 + 0.1 * (2.0 * rng.random() - 1.0)))))
    tau = torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * p.beta
    site = torch.randint(0, p.Nc, (n,), generator=g, dtype=torch.int32, device="cuda")
    X = torch.randn((2, n, n), generator=g, dtype=torch.float64, device="cuda") / math.sqrt(n)
    X.diagonal(dim1=1, dim2=2).add_(
        torch.rand((2, n), generator=g, dtype=torch.float64, device="cuda") + 0.5)
    return n, torch.cat([tau, tau]), torch.cat([site, site]), X


def _cfg_count(p):
    return min(p.R, 16)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "group":
        ps = _group_problems(c)
        return dict(case=c, ps=ps,
                    hs=[g4.G4.for_problem(p, precision="mixed") for p in ps],
                    Ms=[_M(p, seed, i) for i, p in enumerate(ps)],
                    G0s=[torch.from_numpy(inputs.g0(p)).cuda() for p in ps],
                    signs=[_signs(p, seed, i).tolist() for i, p in enumerate(ps)],
                    outs=[torch.empty(p.entries, dtype=torch.complex128, device="cuda") for p in ps])
    p = _problem(c)
    s = dict(case=c, p=p)
    if c["kind"] == "vertex_M":
        s["h"] = g4.G4(p.Nc, p.Nw, 1, 1, precision=c["precision"], batch=1, lx=p.Lx)
        s["cfg"] = _vertices(p, seed, c["U"])
        s["h"].reserve_vertices(s["cfg"][0])
        s["M"] = torch.empty((2, p.N, p.N), device="cuda",
                             dtype=torch.complex128 if c["precision"] == "fp64" else torch.complex64)
        return s
    s["G0"] = torch.from_numpy(inputs.g0(p)).cuda()
    s["signs"] = _signs(p, seed).tolist()
    s["out"] = torch.empty(p.entries, dtype=torch.complex128, device="cuda")
    if c["kind"] == "noalloc":
        s["M"] = _M(p, seed)
        return s
    s["h"] = g4.G4.for_problem(p, precision=c["precision"], channel=c["channel"],
                               deferred=c["deferred"])
    if c["vertices"]:
        s["cfgs"] = [_vertices(p, seed * 4099 + r) for r in range(_cfg_count(p))]
        s["h"].reserve_vertices(max(v[0] for v in s["cfgs"]))
    else:
        s["M"] = _M(p, seed)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    c = s["case"]
    if c["kind"] == "group":
        hs, ps = s["hs"], s["ps"]
        for h in hs:
            h.reset()
        for b in range(max(-(-p.R // p.batch) for p in ps)):
            for i, p in enumerate(ps):
                M = s["Ms"][i]
                for r in range(b * p.batch, min(p.R, (b + 1) * p.batch)):
                    hs[i].compute_G(M[r % M.shape[0]], s["G0s"][i], s["signs"][i][r])
            g4.accumulate_group(hs)
        return [h.finalize(o) for h, o in zip(hs, s["outs"])]
    p = s["p"]
    if c["kind"] == "vertex_M":
        n, tau, site, X = s["cfg"]
        return s["h"].vertex_M(p.beta, n, n, tau, site, X, M=s["M"])
    if c["kind"] == "noalloc":
        acc = s["out"]
        acc.zero_()
        for r, sg in enumerate(s["signs"]):
            g4.update_noalloc(p.Nc, p.Nw, p.Nwex, p.Nkex, s["M"][r % s["M"].shape[0]], s["G0"], sg,
                              acc, lx=p.Lx)
        return acc
    h, G0 = s["h"], s["G0"]
    h.reset()
    if c["vertices"]:
        for r, sg in enumerate(s["signs"]):
            n, tau, site, X = s["cfgs"][r % len(s["cfgs"])]
            h.compute_G_vertices(p.beta, n, n, tau, site, X, G0, sg)
    else:
        M = s["M"]
        for r, sg in enumerate(s["signs"]):
            h.compute_G(M[r % M.shape[0]], G0, sg)
    return h.finalize(s["out"])


# ------------------------------------------------------------------ work of a pass

def _transform_work(p, n, f64):
    """Grouped products and cluster transforms of both spins (vertices grouped by site)."""
    fft = 5.0 * max(1.0, math.log2(p.Nc)) * p.Nw2 * (n + p.N) * p.Nc
    flops = 2 * (4.0 * n * n * p.Nw2 + 8.0 * p.N * p.Nw2 * n + fft)
    return 2 * (8.0 * n * n + 12.0 * n), flops


def _run_work(p, channel, vertices):
    esz = 16 if p.m_dtype == "c128" else 8
    direct = 8.0 if channel in ("ph_magnetic", "ph_density") else 0.0
    w = {"bytes": 16.0 * p.entries + 32.0 * p.N, "flops": (16.0 + direct) * p.updates}
    if vertices:
        b, f = _transform_work(p, inputs.vertices_per_spin(p), False)
        w["bytes"] += p.R * b
        w["flops"] += p.R * f
    else:
        w["bytes"] += p.R * 2.0 * p.N * p.N * esz
        w["flops"] += p.R * 2.0 * 14.0 * p.N * p.N
    return w


def work(case):
    if case["kind"] == "group":
        ws = [_run_work(p, "ph_magnetic", False) for p in _group_problems(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    p = _problem(case)
    if case["kind"] == "vertex_M":
        b, f = _transform_work(p, inputs.vertices_per_spin(p, case["U"]), case["precision"] == "fp64")
        return {"bytes": b + 2.0 * p.N * p.N * (16 if case["precision"] == "fp64" else 8), "flops": f}
    if case["kind"] == "noalloc":
        return _run_work(p, "ph_magnetic", False)
    return _run_work(p, case["channel"], case["vertices"])


# ------------------------------------------------------------------ the same in 64 bits

def _exact_M(p, cfg):
    """Phi Mtau Phi^H / (beta Nc), both spins."""
    n, tau, site, X = cfg
    w = torch.from_numpy(inputs.matsubara(p.Nw, p.beta)).cuda()
    k = torch.from_numpy(inputs.momenta(p.Lx, p.Ly)).cuda()
    x = torch.stack([site[:n] % p.Lx, site[:n] // p.Lx]).double()
    ph = w[None, :, None] * tau[None, None, :n] - (k @ x)[:, None, :]
    Phi = torch.polar(torch.ones_like(ph), ph).reshape(p.N, n)
    return torch.stack([Phi @ X[s].to(torch.complex128) @ Phi.conj().T / (p.beta * p.Nc)
                        for s in range(2)])


def _exact_G4(p, channel, M_of, signs, normalise=True):
    """sum_r s_r [...] over the measurements, exported layout [m][n2][n1][q][k2][k1]."""
    Nc, W, N, NX, NK = p.Nc, p.Nw2, p.N, p.Nwex, p.Nkex
    pp, trans = channel == "pp_updown", channel == "ph_transverse"
    direct = channel in ("ph_magnetic", "ph_density")
    ws = -1.0 if channel == "ph_magnetic" else 1.0
    G0 = torch.from_numpy(inputs.g0(p)).cuda()
    k = np.arange(Nc)
    kx, ky = k % p.Lx, k // p.Lx

    def comb(q, sgn):   # k (+) q, or q (-) k
        return torch.from_numpy((sgn * kx + kx[q]) % p.Lx + p.Lx * ((sgn * ky + ky[q]) % p.Ly)).cuda()

    kk, nn = torch.arange(Nc, device="cuda")[:, None], torch.arange(W, device="cuda")
    # acc[q][m][k2][n2][k1][n1]
    acc = torch.zeros((NK, NX, Nc, W, Nc, W), dtype=torch.complex128, device="cuda")
    if direct:
        A = torch.zeros((NK, NX, len(signs), Nc, W), dtype=torch.complex128, device="cuda")
        B = torch.zeros_like(A)
    for r, sg in enumerate(signs):
        G = -(G0[:, :, None] * M_of(r).to(torch.complex128)) * G0[:, None, :]
        G.diagonal(dim1=1, dim2=2).add_(G0)
        G = G.reshape(2, Nc, W, Nc, W)
        Gt = G.permute(0, 3, 4, 1, 2).contiguous()          # [K2][K1] -> G(K1, K2)
        Gw = G[0] + ws * G[1]
        for q in range(NK):
            idx = comb(q, -1 if pp else 1)
            # the second factor, indexed like G(K2, K1)
            src = G.flip(2, 4) if pp else Gt
            F = (src[:, idx][:, :, :, idx]) * (sg if pp else -sg)
            for m in range(min(NX, W)):
                lo, hi = (slice(m, W), slice(0, W - m)) if pp else (slice(0, W - m), slice(m, W))
                out = acc[q, m][:, lo, :, lo]
                for s in range(2):
                    o = 1 - s if (pp or trans) else s
                    out.addcmul_(G[o][:, lo, :, lo], F[s][:, hi, :, hi])
                if direct:
                    # a(k1, n1) = G((k1 q, n1 + m), (k1, n1)), b(k2, n2) = G((k2, n2), (k2 q, n2 + m))
                    n = nn[:W - m]
                    A[q, m, r, :, :W - m] = Gw[idx[:, None], n + m, kk, n] * sg
                    B[q, m, r, :, :W - m] = Gw[kk, n, idx[:, None], n + m]
    if direct:
        for q in range(NK):
            for m in range(NX):
                acc[q, m] += (B[q, m].reshape(-1, N).T @ A[q, m].reshape(-1, N)).reshape(Nc, W, Nc, W)
        del A, B
    out = acc.permute(1, 3, 5, 0, 2, 4).contiguous()
    return out / float(np.sum(signs)) if normalise else out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "group":
        got = []
        for i, p in enumerate(_group_problems(c)):
            M, s = _M(p, seed, i), _signs(p, seed, i)
            got.append((_exact_G4(p, "ph_magnetic", lambda r: M[r % M.shape[0]], s).reshape(-1),
                        float(s.sum())))
        return got
    p = _problem(c)
    if c["kind"] == "vertex_M":
        return _exact_M(p, _vertices(p, seed, c["U"]))
    if p.updates > 3e11:
        return None
    s = _signs(p, seed)
    if c["kind"] == "run" and c["vertices"]:
        Ms = [_exact_M(p, _vertices(p, seed * 4099 + r)) for r in range(_cfg_count(p))]
        M_of = lambda r: Ms[r % len(Ms)]  # noqa: E731
    else:
        M = _M(p, seed)
        M_of = lambda r: M[r % M.shape[0]]  # noqa: E731
    channel = c.get("channel", "ph_magnetic")
    out = _exact_G4(p, channel, M_of, s, c["kind"] != "noalloc").reshape(-1)
    return out if c["kind"] == "noalloc" else (out, float(s.sum()))
