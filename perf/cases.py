"""The work that is timed: batched IESH trajectories and the library's other
entry points at the sizes a user runs them at.

Every dynamics case starts from a state the caller holds on the device
(positions, momenta, occupations, coefficients), hands it to the library,
advances it by a few steps and takes the new state back into device arrays,
so that one pass can be repeated on the same inputs.  `exact` restates each
path in plain 64-bit torch: dense Hamiltonians diagonalised by
torch.linalg.eigh, couplings as dense triple products, the step's exponential
as a Taylor series, determinant ratios by torch.linalg.solve.
"""
import math

import numpy as np
import torch

import iesh_inputs as W
import paper_2212_00518_gb300 as P
from paper_2212_00518_gb300 import eocc as E
from paper_2212_00518_gb300 import two as T

FS = W.FS_AU
MASK = 0xFFFFFFFF


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # a few trajectories of a small bath: the smallest calls, where the
        # time of a step is launches and latency
        dict(name="well20_fp64", kind="well", M=20, Ne=10, n=16, prec="fp64", dt=1.0, steps=20),
        # the measured configuration of the README: double well, M = 100
        dict(name="well100_fp64", kind="well", M=100, Ne=50, n=4096, prec="fp64", dt=1.0, steps=1),
        dict(name="well100_mixed", kind="well", M=100, Ne=50, n=4096, prec="mixed", dt=1.0, steps=8),
        # the large bath of the README, FP64 for a part of the batch
        dict(name="well200_fp64", kind="well", M=200, Ne=100, n=1024, prec="fp64", dt=1.0, steps=1),
        dict(name="well200_mixed", kind="well", M=200, Ne=100, n=8192, prec="mixed", dt=1.0, steps=2),
        # the paper's relaxation ensemble (Sec. III B): 1000 trajectories, long
        # steps, many hops
        dict(name="relax40_fp64", kind="relax", M=40, Ne=20, n=1000, prec="fp64", dt=100.0, steps=10),
        # one group of the uneven scattering batch: two leads, odd sizes, a
        # work list of live trajectories, trajectories that finish
        dict(name="scatter50_mixed", kind="scatter", M=50, Ne=25, n=1821, prec="mixed", dt=0.1 * FS, steps=16),
        # two adsorbate orbitals over six coordinates
        dict(name="two100_mixed", kind="two", M=100, Ne=51, n=4096, prec="mixed", dt=2.0, steps=4),
        # a batch held in page-locked host memory, advanced with its copies
        dict(name="host100_mixed", kind="host", M=100, Ne=50, n=4096, prec="mixed", dt=1.0, steps=4),
        # differentiable occupied-orbital energy, forward and backward
        dict(name="eocc300_fp64", kind="eocc", M=300, Ne=151, n=8192, prec="fp64"),
        dict(name="eocc300_fp32", kind="eocc", M=300, Ne=151, n=65536, prec="fp32"),
        # batched dense symmetric eigenproblems with eigenvectors
        dict(name="syev102_fp64", kind="syev", M=102, Ne=0, n=2048, prec="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["well", "well", "well", "relax", "scatter", "two", "two", "host", "eocc", "syev"])
    if kind == "syev":
        n = _log(rng, 8, 200)
        return dict(kind=kind, M=n, Ne=0, n=max(16, min(_log(rng, 64, 4096), int(2.2e9 / n ** 3))),
                    prec=rng.choice(["fp64", "fp32"]))
    if kind == "eocc":
        M = _log(rng, 20, 400)
        return dict(kind=kind, M=M, Ne=M // 2 + 1, n=max(16, min(_log(rng, 256, 32768), int(7e8 / M ** 2))),
                    prec=rng.choice(["fp64", "fp32"]))
    prec = rng.choice(["fp64", "mixed"]) if kind != "host" else "mixed"
    M = _log(rng, 10, 200) if kind in ("well", "host", "two") else _log(rng, 20, 120)
    Ne = min(112, max(1, int(round(M * rng.uniform(0.4, 0.6)))))
    steps = rng.randint(1, 4)
    dt = {"well": 1.0, "host": 1.0, "relax": 100.0, "scatter": 0.1 * FS, "two": 2.0}[kind]
    # at most the work of a third of the largest listed case of the precision
    # (the stiffer bands of the ensembles take several times the series terms)
    work = (M + 2) ** 2 * Ne * steps * (1.0 if kind in ("well", "host") else 4.0)
    most = (7e8 if prec == "fp64" else 2e10) / work
    return dict(kind=kind, M=M, Ne=Ne, n=max(16, min(_log(rng, 16, 8192), int(most))), prec=prec, dt=dt, steps=steps)


# ---------------------------------------------------------------- the inputs
def _model(case):
    if case["kind"] in ("well", "host"):
        return W.double_well(case["M"], case["Ne"])
    if case["kind"] == "relax":
        md = W.double_well_paper(case["M"])
        md["Ne"] = case["Ne"]
        return md
    if case["kind"] == "scatter":
        md = W.morse_image(case["M"], bias=0.1)
        md["Ne"] = case["Ne"]
        return md
    return W.two_orbital(M=case["M"], Ne=case["Ne"])


def _coefficients(occ, N, weight, gen):
    """Orthonormal electron columns [n][Ne][N] near the occupied orbitals, every
    amplitude nonzero: what a trajectory carries after some time."""
    n, Ne = occ.shape
    C = torch.complex(*(torch.randn(n, Ne, N, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2)))
    C.mul_(weight / math.sqrt(N))
    C.scatter_add_(2, occ[:, :, None], torch.ones(n, Ne, 1, dtype=torch.complex128, device="cuda"))
    L = torch.linalg.cholesky(C @ C.mH)
    return torch.linalg.solve_triangular(L, C, upper=False)


def _inputs(case, seed):
    """x, p, occ, C on the device."""
    kind, n, Ne = case["kind"], case["n"], case["Ne"]
    md = _model(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    N = case["M"] + (2 if kind == "two" else 1)
    occ = torch.arange(Ne, device="cuda").repeat(n, 1)
    if kind in ("well", "host"):
        kT = np.array([0.005, 0.0075, 0.01])[np.arange(n) % 3]
        x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], kT, seed)
    elif kind == "relax":
        x, p = W.thermal_harmonic(n, md["mass"], md["par"][0], 5 * 9.5e-4, seed)
        # electrons near the Fermi level rearranged, as at finite temperature
        jitter = torch.rand(n, N, device="cuda", generator=gen) * 0.15 * N
        occ = torch.topk(jitter + torch.arange(N, device="cuda"), Ne, dim=1, largest=False).indices.sort(1).values
    elif kind == "scatter":
        e = rng.uniform(W.ev(0.2), W.ev(1.5), n)
        # most on the way in at all distances, some about to leave
        x = W.angstrom(rng.uniform(1.6, 9.98, n))
        p = np.sqrt(2.0 * md["mass"] * e) * np.where(x > W.angstrom(9.5), 1.0, -1.0)
    else:
        s = np.sqrt(0.01 / (md["mass"] * md["omega"] ** 2))
        x = md["x0"][None, :] + rng.normal(0.0, s, (n, 6))
        p = rng.normal(0.0, np.sqrt(md["mass"] * 0.01), (n, 6))
        occ = torch.rand(n, N, device="cuda", generator=gen).argsort(1)[:, :Ne].sort(1).values
    C = _coefficients(occ, N, 0.3, gen)
    if case["prec"] != "fp64":
        C = C.to(torch.complex64)
    return md, torch.from_numpy(x).cuda(), torch.from_numpy(p).cuda(), occ.to(torch.int16).contiguous(), C.contiguous()


def _symmetric(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = case["M"]
    A = torch.randn(case["n"], n, n, dtype=torch.float64, device="cuda", generator=gen)
    A = 0.5 * (A + A.mT) + torch.diag(torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda") * math.sqrt(n))
    A = 0.5 * (A + A.mT)
    return A.contiguous() if case["prec"] == "fp64" else A.float().contiguous()


def _eocc_inputs(case, seed):
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    wl = W.eocc_workload(M=case["M"], B=case["n"], seed=5, Ne=case["Ne"])
    rng = np.random.default_rng(seed)
    x = torch.from_numpy(rng.normal(0.0, 0.3, (case["n"], 6))).to("cuda", dt)
    gE = torch.from_numpy(rng.normal(0.0, 1.0, case["n"])).to("cuda", dt)
    return wl, x, torch.from_numpy(wl["theta"]).to("cuda", dt), gE


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.seed = case, seed
    kind = case["kind"]
    if kind == "syev":
        s.A = _symmetric(case, seed)
        n, B = case["M"], case["n"]
        s.lam = torch.empty(B, n, dtype=s.A.dtype, device="cuda")
        s.V = torch.empty(B, n, n, dtype=s.A.dtype, device="cuda")
        s.info = torch.empty(B, dtype=torch.int32, device="cuda")
        need = P.iesh.load().iesh_syev_work_bytes(B, n, P.PREC_FP64 if case["prec"] == "fp64" else P.PREC_MIXED, 1)
        s.work = torch.empty(need, dtype=torch.uint8, device="cuda")
        return s
    if kind == "eocc":
        wl, s.x, s.theta, s.gE = _eocc_inputs(case, seed)
        s.model = E.EOccModel(wl)
        s.x.requires_grad_(True)
        s.theta.requires_grad_(True)
        return s
    md, s.x, s.p, s.occ, s.C = _inputs(case, seed)
    prec = P.PREC_FP64 if case["prec"] == "fp64" else P.PREC_MIXED
    n = case["n"]
    if kind == "two":
        s.ctx = T.TwoOrbitalContext(md, n, precision=prec)
    else:
        more = dict(z_done=W.angstrom(10.0), compact_every=4) if kind == "scatter" else {}
        s.ctx = P.Context(md, n, precision=prec, **more)
    s.out = dict(x=torch.empty_like(s.x), p=torch.empty_like(s.p), occ=torch.empty_like(s.occ),
                 C=torch.empty_like(s.C), status=torch.empty(n, dtype=torch.int32, device="cuda"))
    if kind == "host":
        s.ctx.set_state(s.x, s.p, s.occ, s.C)
        s.src = torch.from_numpy(s.ctx.checkpoint_save()).pin_memory()
        s.dst = torch.empty_like(s.src, pin_memory=True)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "syev":
        P.iesh.syev_batched(s.A, s.lam, s.V, s.info, s.work)
        return dict(lam=s.lam, V=s.V, info=s.info)
    if kind == "eocc":
        energy = E.eocc(s.x, s.theta, s.model)
        dx, dth = torch.autograd.grad(energy, (s.x, s.theta), s.gE)
        return dict(E=energy.detach(), dx=dx, dtheta=dth)
    if kind == "host":
        s.ctx.run_host(s.src, s.dst, s.case["dt"], s.case["steps"], seed=s.seed)
    else:
        s.ctx.set_state(s.x, s.p, s.occ, s.C)
        s.ctx.run(s.case["dt"], s.case["steps"], seed=s.seed)
    s.ctx.get_state(**s.out)
    return s.out


def work(case):
    n, Ne, M = case["n"], case["Ne"], case["M"]
    if case["kind"] == "syev":
        w = 8 if case["prec"] == "fp64" else 4
        return dict(bytes=n * w * (2 * M * M + M), flops=n * (4 / 3 + 4 / 3 + 3.0) * M ** 3)
    if case["kind"] == "eocc":
        w = 8 if case["prec"] == "fp64" else 4
        # one evaluation of every root's sums, and the gradients
        return dict(bytes=n * w * (6 + 1 + 1 + 6), flops=n * (6.0 * Ne * (M + 1) + 200))
    N = M + (2 if case["kind"] == "two" else 1)
    c = 16 if case["prec"] == "fp64" else 8
    # the unitary application, the determinant ratios, eigenpairs and couplings
    step = 8.0 * N * N * Ne + 8.0 * (N - Ne) * Ne * Ne + 8.0 / 3.0 * Ne ** 3 + 34.0 * N * N
    if case["kind"] == "host":  # the state's blob in and out
        return dict(bytes=2.0 * n * (c * N * Ne + 2 * Ne + 8 * 9 * N), flops=n * case["steps"] * step)
    return dict(bytes=2.0 * n * (c * N * Ne + 2 * Ne + 16), flops=n * case["steps"] * step)


# ------------------------------------------------------ plain 64-bit results
def _gauss_half(n, a, b):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (b - a) * x + 0.5 * (a + b), 0.5 * (b - a) * w


def _bath(md):
    lo, hi = md["band"]
    leads = md.get("leads") or [(md.get("mu", 0.0), md["M"] // 2, md["M"], 1.0)]
    e, w = [], []
    for mu, n_lo, n, frac in leads:
        for k, a, b in ((n_lo, lo, mu), (n - n_lo, mu, hi)):
            if k:
                ee, ww = _gauss_half(k, a, b)
                e.append(ee)
                w.append(ww * frac)
    e, w = np.concatenate(e), np.concatenate(w)
    o = np.argsort(e, kind="stable")
    return torch.from_numpy(e[o]).cuda(), torch.from_numpy(w[o]).cuda()


class _One:
    """One adsorbate orbital, one coordinate: x, p [n]."""

    def __init__(self, md):
        self.md, self.mass, self.P = md, md["mass"], md["par"]
        self.eps, w = _bath(md)
        self.z = math.sqrt(md["Gamma"] / (2 * math.pi)) * torch.sqrt(w)
        self.N = md["M"] + 1

    def at(self, x):
        """U0, dU0 [n][1], H [n][N][N], dH [n][1][N][N]."""
        P_, m, x = self.P, self.mass, x[:, 0]
        if self.md["kind"] == "harmonic":
            k = m * P_[0] ** 2
            U0, dU0 = 0.5 * k * x * x, k * x
            h, dh = 0.5 * k * (P_[1] ** 2 - 2 * P_[1] * x) + P_[2], torch.full_like(x, -k * P_[1])
            f, df = torch.ones_like(x), torch.zeros_like(x)
        else:
            De, x0, a, c, hinf, zim, ac, zc, sg = P_[:9]
            e = torch.exp(-a * (x - x0))
            U0, dU0 = De * (e - 1) ** 2 + c, -2 * a * De * (e - 1) * e
            r = torch.sqrt((x - zim) ** 2 + ac * ac)
            h, dh = hinf - 0.25 / r, 0.25 * (x - zim) / r ** 3
            f = torch.exp(-0.5 * ((x - zc) / sg) ** 2)
            df = -((x - zc) / sg ** 2) * f
        H = torch.diag_embed(torch.cat([h[:, None], self.eps.expand(len(x), -1)], 1))
        dH = torch.zeros_like(H)
        H[:, 0, 1:] = H[:, 1:, 0] = f[:, None] * self.z
        dH[:, 0, 0] = dh
        dH[:, 0, 1:] = dH[:, 1:, 0] = df[:, None] * self.z
        return U0, dU0[:, None], H, dH[:, None]

    def gauge(self, Q, Q_old, x):
        return Q * torch.where(Q[:, :1, :] < 0, -1.0, 1.0)


class _Two:
    """Two adsorbate orbitals, six coordinates: x, p [n][6]."""

    def __init__(self, md):
        self.md, self.mass = md, md["mass"]
        self.eps, w = _bath(md)
        self.w = torch.sqrt(w)
        self.N = md["M"] + 2
        self.th = [float(v) for v in md["theta"]]
        self.g = torch.tensor([self.th[2:8], self.th[8:14]], dtype=torch.float64, device="cuda")
        self.R = torch.as_tensor(md["R"], device="cuda")
        self.x0 = torch.as_tensor(md["x0"], device="cuda")

    def coupling(self, x):
        d = x - self.R
        return [self.md["Vbar"][a] * torch.exp(-0.5 * (d[:, 3 * a:3 * a + 3] ** 2).sum(1) / self.th[14 + a] ** 2)
                for a in range(2)]

    def at(self, x):
        n, k = len(x), self.mass * self.md["omega"] ** 2
        U0, dU0 = 0.5 * k * ((x - self.x0) ** 2).sum(1), k * (x - self.x0)
        h = x @ self.g.T + torch.tensor(self.th[:2], dtype=torch.float64, device="cuda")
        c = self.coupling(x)
        H = torch.diag_embed(torch.cat([h, self.eps.expand(n, -1)], 1))
        dH = torch.zeros(n, 6, self.N, self.N, dtype=torch.float64, device="cuda")
        for a in range(2):
            H[:, a, 2:] = H[:, 2:, a] = c[a][:, None] * self.w
            dH[:, :, a, a] = self.g[a]
            kap = -(x - self.R)[:, 3 * a:3 * a + 3] / self.th[14 + a] ** 2
            v = (kap * c[a][:, None])[:, :, None] * self.w
            dH[:, 3 * a:3 * a + 3, a, 2:] = v
            dH[:, 3 * a:3 * a + 3, 2:, a] = v
        return U0, dU0, H, dH

    def gauge(self, Q, Q_old, x):
        c = self.coupling(x)
        s = torch.where(c[0][:, None] * Q[:, 0] + c[1][:, None] * Q[:, 1] < 0, -1.0, 1.0)
        if Q_old is not None:
            ov = (Q_old * Q).sum(1)
            s = torch.where(ov.abs() >= 0.5, torch.sign(ov), s)
        return Q * s[:, None, :]


def _uniform(seed, n, step):
    """The hop uniforms of trajectories 0..n-1 at a step (Philox4x32-10)."""
    c = [torch.arange(n, dtype=torch.int64, device="cuda")] + [torch.full((n,), v, dtype=torch.int64, device="cuda")
                                                               for v in (0, step & MASK, step >> 32)]
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for r in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & MASK) ^ c[1] ^ k0, b & MASK, ((a >> 32) & MASK) ^ c[3] ^ k1, a & MASK]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return ((c[0] >> 5).double() * 67108864.0 + (c[1] >> 6).double()) / 9007199254740992.0


def _dynamics(model, case, seed, x, p, occ, C, z_done):
    """x, p [n][D], occ [n][Ne] int64, C [n][Ne][N] complex128, advanced."""
    dt, m, n, Ne, N = case["dt"], model.mass, case["n"], case["Ne"], model.N
    ar = torch.arange(n, device="cuda")[:, None]

    def electrons(x, occ, Q_old):
        _, dU0, H, dH = model.at(x)
        lam, Q = (v.cuda() for v in torch.linalg.eigh(H.cpu()))  # the host's LAPACK is the faster one here
        Q = model.gauge(Q, Q_old, x)
        Tm = Q.mT[:, None] @ (dH @ Q[:, None])  # [n][D][N][N]
        return lam, Q, Tm, dU0

    def force(Tm, dU0, occ):
        return -dU0 - torch.diagonal(Tm, dim1=2, dim2=3)[ar[:, :, None], torch.arange(Tm.shape[1], device="cuda")[None, :, None],
                                                        occ[:, None, :]].sum(2)

    def couple(Tm, lam, v):
        gap = lam[:, None, :] - lam[:, :, None]
        gap.diagonal(dim1=1, dim2=2).fill_(1.0)
        D = (Tm * v[:, :, None, None]).sum(1) / gap
        D.diagonal(dim1=1, dim2=2).zero_()
        return D

    lam, Q, Tm, dU0 = electrons(x, occ, None)
    F, v = force(Tm, dU0, occ), p / m
    done = torch.zeros(n, dtype=torch.bool, device="cuda")
    for step in range(case["steps"]):
        keep = (x, p, occ, C, lam, Q, Tm, dU0, F, v)
        D0, lam0 = couple(Tm, lam, v), lam
        p = p + 0.5 * dt * F
        x = x + dt * p / m
        lam, Q, Tm, dU0 = electrons(x, occ, Q)
        F = force(Tm, dU0, occ)
        p = p + 0.5 * dt * F
        v = p / m
        D1 = couple(Tm, lam, v)
        G = torch.complex(torch.diag_embed(0.5 * dt * (lam0 + lam)), -0.5 * dt * (D0 + D1)) * -1j
        mid = 0.25 * dt * (lam0 + lam)
        mid = (mid.max(1).values + mid.min(1).values)[:, None]  # the interval's middle, taken out of the series
        G.diagonal(dim1=1, dim2=2).add_(1j * mid)
        parts = max(1, math.ceil(float(G.abs().sum(2).max())))
        Y = C.mT.contiguous()
        for _ in range(parts):
            term = Y
            for k in range(1, 28):
                term = (G @ term) / (k * parts)
                Y = Y + term
        C = (Y * torch.exp(-1j * mid)[:, :, None]).mT.contiguous()
        # determinant ratios of every single excitation, and one hop at most
        Ct = C.mT
        S = Ct[ar, occ]
        Rm = torch.linalg.solve(S, Ct, left=False)  # [n][N][Ne]
        d = D1.gather(2, occ[:, None, :].expand(-1, N, -1))
        g = torch.clamp(-2.0 * dt * Rm.real * d, min=0.0).mT  # [n][Ne][N]
        g = g.scatter(2, occ[:, None, :].expand(-1, Ne, -1), 0.0).reshape(n, -1)
        over = g.cumsum(1) > _uniform(seed, n, step)[:, None]
        hop = over.any(1)
        at = over.to(torch.int8).argmax(1)
        a, to = at // N, at % N
        src = occ.gather(1, a[:, None])[:, 0]
        dE = (lam.gather(1, to[:, None]) - lam.gather(1, src[:, None]))[:, 0]
        if x.shape[1] == 1:
            p2 = p[:, 0] ** 2 - 2 * m * dE
            ok = hop & (p2 >= 0)
            pn = torch.where(p >= 0, 1.0, -1.0) * torch.sqrt(p2.clamp(min=0.0))[:, None]
        else:
            dv = Tm[ar[:, 0], :, to, src]  # along d_{m, s_a}: its length does not matter
            qa, qb = (dv * dv).sum(1), (dv * p).sum(1)
            disc = qb * qb - 2 * m * dE * qa
            ok = hop & (disc >= 0) & (qa > 0)
            root = torch.where(qb >= 0, 1.0, -1.0) * torch.sqrt(disc.clamp(min=0.0))
            pn = p + (-2 * m * dE / (qb + root))[:, None] * dv
        p = torch.where(ok[:, None], pn, p)
        occ = torch.where(ok[:, None], occ.scatter(1, a[:, None], to[:, None]).sort(1).values, occ)
        F, v = force(Tm, dU0, occ), p / m
        x, p, occ, C, lam, Q, Tm, dU0, F, v = (
            torch.where(done.reshape([n] + [1] * (o.dim() - 1)), o, w)
            for o, w in zip(keep, (x, p, occ, C, lam, Q, Tm, dU0, F, v)))
        if z_done > 0:
            done |= x[:, 0] > z_done
    return x, p, C


def _exact_eocc(case, seed):
    wl, x, theta, gE = _eocc_inputs(case, seed)
    x, th, gE = x.double(), theta.double(), gE.double()
    eps, w = _bath(dict(band=wl["band"], M=wl["M"]))
    R, V, Ne, n = torch.as_tensor(wl["R"], device="cuda"), wl["Vbar"], case["Ne"], case["n"]
    En = torch.empty(n, dtype=torch.float64, device="cuda")
    d = x - R
    r2 = torch.stack([(d[:, :3] ** 2).sum(1), (d[:, 3:] ** 2).sum(1)], 1)
    h = torch.stack([th[0] + x @ th[2:8], th[1] + x @ th[8:14]], 1)
    c = torch.as_tensor(V, device="cuda") * torch.exp(-0.5 * r2 / th[14:] ** 2)
    S, U = torch.empty(n, 2, dtype=torch.float64, device="cuda"), torch.empty(n, 2, dtype=torch.float64, device="cuda")
    for b in range(0, n, max(1, int(4e7 / (Ne * (wl["M"] + 1))))):
        sl = slice(b, min(n, b + max(1, int(4e7 / (Ne * (wl["M"] + 1))))))
        c0, c1, h0, h1 = c[sl, 0], c[sl, 1], h[sl, 0], h[sl, 1]
        c2 = c0 * c0 + c1 * c1
        hp, hm = (c0 * c0 * h0 + c1 * c1 * h1) / c2, (c1 * c1 * h0 + c0 * c0 * h1) / c2
        t = c0 * c1 * (h1 - h0) / c2
        # one arrowhead: the bath and |->, each with its weight
        pole, o = torch.cat([eps.expand(len(c2), -1), hm[:, None]], 1).sort(1)
        wt = torch.cat([c2[:, None] * w, (t * t)[:, None]], 1).gather(1, o)
        reach = torch.sqrt(wt.sum(1)) + (hp - pole[:, 0]).abs() + 1.0
        up = pole[:, :Ne]
        low = torch.cat([(pole[:, 0] - reach)[:, None], pole[:, :Ne - 1]], 1)
        gap = up - low

        def rest(base, tau):  # lam - h_+ - sum and its slope at lam = base + tau
            q = (base[:, :, None] - pole[:, None, :]) + tau[:, :, None]
            q = wt[:, None, :] / q
            return (base - hp[:, None]) + tau - q.sum(2)

        left = (rest(low, 0.5 * gap) >= 0) & (torch.arange(Ne, device="cuda") > 0)
        base = torch.where(left, low, up)
        lo, hi = torch.where(left, 0.0, -gap), torch.where(left, gap, 0.0)
        for _ in range(70):
            tau = 0.5 * (lo + hi)
            neg = rest(base, tau) < 0
            lo, hi = torch.where(neg, tau, lo), torch.where(neg, hi, tau)
        tau = 0.5 * (lo + hi)
        lam = base + tau
        q = (base[:, :, None] - pole[:, None, :]) + tau[:, :, None]
        qp = 1.0 / torch.sqrt(1.0 + (wt[:, None, :] / (q * q)).sum(2))
        qm = t[:, None] * qp / ((base - hm[:, None]) + tau)
        cc = torch.sqrt(c2)[:, None]
        Q = [(c0[:, None] * qp - c1[:, None] * qm) / cc, (c1[:, None] * qp + c0[:, None] * qm) / cc]
        En[sl] = lam.sum(1)
        for a, hh in ((0, h0), (1, h1)):
            S[sl, a] = (Q[a] ** 2).sum(1)
            U[sl, a] = (Q[a] ** 2 * (lam - hh[:, None])).sum(1)
        del q
    dx = S @ torch.stack([th[2:8], th[8:14]])
    dx = dx + 2 * torch.cat([U[:, :1] * -d[:, :3] / th[14] ** 2, U[:, 1:] * -d[:, 3:] / th[15] ** 2], 1)
    per = torch.cat([S, S[:, :1] * x, S[:, 1:] * x, 2 * U * r2 / th[14:] ** 3], 1)
    return dict(E=En, dx=gE[:, None] * dx, dtheta=(gE[:, None] * per).sum(0))


def exact(case, seed):
    kind = case["kind"]
    if kind == "eocc":
        return _exact_eocc(case, seed) if case["n"] * case["Ne"] * case["M"] < 1.2e9 else None
    if kind == "syev":
        if case["n"] * case["M"] ** 2 > 8e7:
            return None
        lam, Q = torch.linalg.eigh(_symmetric(case, seed).double().cpu())
        big = Q.abs().argmax(1, keepdim=True)
        return dict(lam=lam.cuda(), V=(Q * torch.sign(Q.gather(1, big))).mT.contiguous().cuda(), info=None)
    N = case["M"] + (2 if kind == "two" else 1)
    if case["n"] * N * N * (case["steps"] + 1) > 1.3e8 or case["n"] * N * N * (8 if kind == "two" else 1) > 4e8:
        return None  # dense eigenproblems of the whole batch at every step
    md, x, p, occ, C = _inputs(case, seed)
    model = _Two(md) if kind == "two" else _One(md)
    shape = x.shape
    z_done = W.angstrom(10.0) if kind == "scatter" else 0.0
    x, p, C = _dynamics(model, case, seed, x.reshape(case["n"], -1), p.reshape(case["n"], -1), occ.long(),
                        C.to(torch.complex128), z_done)
    return dict(x=x.reshape(shape), p=p.reshape(shape), occ=None, C=C, status=None)
