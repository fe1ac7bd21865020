"""Performance cases of the stochastic-LapH path on one GB300.

Each case is one call of a public entry point of paper_1104_3870_gb300.laph (or the
short sequence a user's program makes around it) on seeded synthetic inputs made on
the GPU.  Sizes come from the repository's workloads (4^3 x 8, 16^3 x 32, 24^3 x 128)
and from ordinary lattices in between.  exact() restates the same quantity in plain
torch / numpy FP64 and uses nothing of the package.
"""
import math

import numpy as np
import torch

from paper_1104_3870_gb300 import laph as L

XI, CSW = 3.5, 1.0           # anisotropy and clover coefficient of every workload
RHO, STOUT = 0.1, 10         # 4D stout steps that smooth the random links (stand-in for thermalisation)
C128 = torch.complex128
_CTX = {}


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _ctx():
    """One context (workspace, autotune cache) for the process, as a user's program keeps it."""
    if "c" not in _CTX:
        _CTX["c"] = L.Context(0)
    return _CTX["c"]


def _gen(seed, tag):
    return torch.Generator(device=_dev()).manual_seed(1000003 * (int(seed) % (1 << 40)) + tag)


def _randn(shape, g):
    return torch.complex(torch.randn(shape, generator=g, dtype=torch.float64, device=_dev()),
                         torch.randn(shape, generator=g, dtype=torch.float64, device=_dev()))


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the exact-distillation check lattice: a few sources of one time slice, where the
        # latency of a Krylov iteration counts and nothing else
        dict(name="solve_4x8", kind="solve", ns=4, nt=8, nrhs=8, m0=-0.04898, block=0, iters=60),
        # one source time of the 16^3 x 32 workload: 32 diluted sources (SF, LI8) in one call
        dict(name="solve_16x32", kind="solve", ns=16, nt=32, nrhs=32, m0=-0.0049, block=0, iters=190),
        # a slab of the 24^3 lattice with the block of 32 sources that the headline step solves
        dict(name="solve_24x32", kind="solve", ns=24, nt=32, nrhs=32, m0=0.005, block=32, iters=180),
        # the even-odd stencil on its own (its public entry): FP32 spinors, 32 right-hand sides, 24^3 slab
        dict(name="dslash_24x32", kind="dslash", ns=24, nt=32, nrhs=32, prec="fp32", mode="clovinv", parity=0),
        # true residuals of a set of solutions: K in FP64 on the full lattice
        dict(name="apply_16x32", kind="apply", ns=16, nt=32, nrhs=12, m0=-0.0049),
        # the 32 sources of one block of the headline step: Z4 noise, time-interlaced dilution
        dict(name="sources_24x128", kind="sources", ns=24, nt=128, nv=64, nrhs=32, tdil=16, ldil=8),
        # sink coefficients of one block of the headline step
        dict(name="sinks_24x128", kind="sinks", ns=24, nt=128, nv=64, nrhs=32),
        # sink coefficients of a few sources on a small lattice (ragged against every tile)
        dict(name="sinks_6x12", kind="sinks", ns=6, nt=12, nv=10, nrhs=5),
        # eigenvectors of every slice of the 16^3 x 32 workload
        dict(name="eigvecs_16x32", kind="eigvecs", ns=16, nt=32, nv=32),
        # pion correlator of one source time of the 16^3 x 32 workload (two lines, 32 projectors)
        dict(name="pion_16x32", kind="corr", channel="pion", nt=32, nv=32, nb=32, t0=8),
        # I = 2 two-pion correlator of one source time of the 24^3 x 128 workload (four lines)
        dict(name="pipi_24x128", kind="corr", channel="pipi", nt=128, nv=64, nb=32, t0=5),
        # momentum overlaps of the four smallest momenta on the 16^3 x 32 workload
        dict(name="overlaps_16x32", kind="overlaps", ns=16, nt=32, nv=32, nmom=4),
    ]


def _even(rng, lo, hi):
    return 2 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2))


def _whole(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "dslash", "apply", "sources", "sinks", "sinks", "eigvecs", "corr",
                       "overlaps"])
    if kind in ("solve", "dslash", "apply"):
        ns = rng.choice([4, 6, 8, 10, 12, 14, 16, 20, 24])
        nt = _even(rng, 4, 64)
        nrhs = rng.choice([_whole(rng, 1, 64), _whole(rng, 1, 64), 12, 16, 32, 64])
        while ns ** 3 * nt * nrhs > 24 ** 3 * 32 * 32 * (0.8 if kind == "solve" else 1.0):
            nt, nrhs = max(4, 2 * (nt // 4)), max(1, nrhs // 2)
        m0 = round(rng.uniform(0.02, 0.12), 4)
        if kind == "solve":
            return dict(kind=kind, ns=ns, nt=nt, nrhs=nrhs, m0=m0, block=rng.choice([0, 0, 32]),
                        iters=int(10 / (m0 + 0.05)))
        if kind == "apply":
            return dict(kind=kind, ns=ns, nt=nt, nrhs=min(nrhs, 48), m0=m0)
        return dict(kind=kind, ns=ns, nt=nt, nrhs=nrhs, prec=rng.choice(["fp32", "fp32", "fp64"]),
                    mode=rng.choice(["clovinv", "xpay", "apply"]), parity=rng.randrange(2))
    if kind == "sources":
        ldil = rng.choice([2, 4, 8])
        tdil = rng.choice([2, 4, 8])
        return dict(kind=kind, ns=rng.choice([4, 6, 8, 10, 12, 16, 20, 24]), nt=tdil * _even(rng, 2, 8),
                    nv=ldil * _whole(rng, 1, 8), nrhs=_whole(rng, 1, 32), tdil=tdil, ldil=ldil)
    if kind == "sinks":
        return dict(kind=kind, ns=rng.choice([4, 6, 8, 10, 12, 16, 20, 24]), nt=_even(rng, 4, 64),
                    nv=_whole(rng, 4, 112), nrhs=_whole(rng, 1, 40))
    if kind == "eigvecs":
        return dict(kind=kind, ns=rng.choice([4, 6, 8, 10]), nt=_even(rng, 4, 16), nv=_whole(rng, 4, 24))
    if kind == "corr":
        nt = _even(rng, 8, 128)
        return dict(kind=kind, channel=rng.choice(["pion", "rho", "scalar", "pipi"]), nt=nt, nv=8 * _whole(rng, 1, 8),
                    nb=4 * _whole(rng, 1, 8), t0=rng.randrange(nt))
    return dict(kind="overlaps", ns=rng.choice([4, 6, 8, 10, 12, 16]), nt=_even(rng, 4, 32), nv=_whole(rng, 4, 48),
                nmom=rng.choice([1, 2, 4, 7]))


# ------------------------------------------------------------------ lattice helpers (plain torch, FP64)
_AX = (3, 2, 1, 0)   # axis of x, y, z, t in [t, z, y, x, ...]


def _fwd(f, mu, lead=0):
    return torch.roll(f, -1, _AX[mu] + lead)


def _bwd(f, mu, lead=0):
    return torch.roll(f, 1, _AX[mu] + lead)


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _expm(a):
    """exp of small 3x3 matrices: Taylor series of a / 16, squared four times."""
    one = torch.eye(3, dtype=C128, device=a.device)
    x = a / 16.0
    e = one + x / 10.0
    for k in range(9, 0, -1):
        e = one + _mm(x, e) / k
    for _ in range(4):
        e = _mm(e, e)
    return e


def _raw_links(ns, nt, seed):
    """U = exp(0.4 i H), H Gaussian traceless Hermitian, [t, z, y, x, mu, 3, 3]."""
    a = _randn((nt, ns, ns, ns, 4, 3, 3), _gen(seed, 1))
    h = 0.5 * (a + _dag(a))
    h = h - h.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3.0 * torch.eye(3, dtype=C128, device=a.device)
    return _expm(0.4j * h)


def _stout(u, steps, ndir):
    """Stout smearing over the first ndir directions (staples among them only)."""
    for _ in range(steps):
        out = u.clone()
        for mu in range(ndir):
            um = u[..., mu, :, :]
            c = torch.zeros_like(um)
            for nu in range(ndir):
                if nu == mu:
                    continue
                un = u[..., nu, :, :]
                c += _mm(_mm(un, _fwd(um, nu)), _dag(_fwd(un, mu)))
                ub = _bwd(un, nu)
                c += _mm(_mm(_dag(ub), _bwd(um, nu)), _fwd(ub, mu))
            om = RHO * _mm(c, _dag(um))
            a = _dag(om) - om
            tr = a.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3.0
            out[..., mu, :, :] = _mm(_expm(-0.5 * (a - tr * torch.eye(3, dtype=C128, device=u.device))), um)
        u = out
    return u


def _links(ns, nt, seed):
    return _stout(_raw_links(ns, nt, seed), STOUT, 4).contiguous()


# Dirac matrices, gamma_mu = [[0, G], [G^dag, 0]], G_k = -i sigma_k, G_4 = 1
def _gammas():
    s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    g = []
    for b in [-1j * m for m in s] + [np.eye(2)]:
        m = np.zeros((4, 4), dtype=complex)
        m[:2, 2:], m[2:, :2] = b, b.conj().T
        g.append(m)
    return g


class _Dirac:
    """K of include/laph.h on [n, t, z, y, x, 4, 3] fields, plain torch."""

    def __init__(self, u, m0):
        self.gm = [torch.tensor(g, dtype=C128, device=u.device) for g in _gammas()]
        self.one = torch.eye(4, dtype=C128, device=u.device)
        self.w = (1 / XI, 1 / XI, 1 / XI, 1.0)
        a = torch.zeros(u.shape[:4] + (4, 3, 4, 3), dtype=C128, device=u.device)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                um, un = u[..., mu, :, :], u[..., nu, :, :]
                umm, unm, unn = _bwd(um, mu), _bwd(un, mu), _bwd(un, nu)
                q = _mm(_mm(_mm(um, _fwd(un, mu)), _dag(_fwd(um, nu))), _dag(un))
                q += _mm(_mm(_mm(un, _dag(_fwd(umm, nu))), _dag(unm)), umm)
                q += _mm(_mm(_mm(_dag(umm), _dag(_bwd(unm, nu))), _bwd(umm, nu)), unn)
                umn = _bwd(um, nu)
                q += _mm(_mm(_mm(_dag(unn), umn), _fwd(unn, mu)), _dag(um))
                f = (q - _dag(q)) / 8j
                f = f - f.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3 * torch.eye(3, dtype=C128, device=u.device)
                sg = 0.5j * (self.gm[mu] @ self.gm[nu] - self.gm[nu] @ self.gm[mu])
                wp = 0.5 * (1 + 1 / XI) if nu == 3 else 1 / XI
                a -= 0.5 * CSW * wp * torch.einsum("ab,tzyxij->tzyxaibj", sg, f)
        a = a.reshape(u.shape[:4] + (12, 12))
        self.a = a + (m0 + sum(self.w)) * torch.eye(12, dtype=C128, device=u.device)
        self.u = u.clone()
        self.u[-1, :, :, :, 3] *= -1.0      # antiperiodic in time

    def diag(self, f):
        return (self.a * f.flatten(-2).unsqueeze(-2)).sum(-1).unflatten(-1, (4, 3))

    def hop(self, f):
        out = torch.zeros_like(f)
        for mu in range(4):
            um = self.u[..., mu, :, :]
            a = torch.einsum("tzyxij,ntzyxsj->ntzyxsi", um, _fwd(f, mu, 1))
            b = _bwd(torch.einsum("tzyxji,ntzyxsj->ntzyxsi", um.conj(), f), mu, 1)
            out -= 0.5 * self.w[mu] * (torch.einsum("ab,ntzyxbc->ntzyxac", self.one - self.gm[mu], a)
                                       + torch.einsum("ab,ntzyxbc->ntzyxac", self.one + self.gm[mu], b))
        return out

    def __call__(self, f):
        return self.diag(f) + self.hop(f)

    def solve(self, b):
        """x with K x = b by restarted BiCGStab, one right-hand side."""
        x, r = torch.zeros_like(b), b.clone()
        bn = b.norm()
        for _ in range(8):
            if r.norm() <= 1e-15 * bn:
                break
            rh, p = r.clone(), r.clone()
            rho, d, stop = (rh.conj() * r).sum(), torch.zeros_like(b), max(1e-5 * float(r.norm()), 2e-16 * float(bn))
            for it in range(3000):
                v = self(p)
                al = rho / (rh.conj() * v).sum()
                s = r - al * v
                t = self(s)
                om = (t.conj() * s).sum() / (t.conj() * t).sum()
                d += al * p + om * s
                r = s - om * t
                if it % 10 == 9 and not float(r.norm()) > stop:
                    break
                new = (rh.conj() * r).sum()
                p = r + (new / rho) * (al / om) * (p - om * v)
                rho = new
            x = x + d
            r = b - self(x)
        return x


def _waves(ns, count, dev):
    """The lowest plane waves of a slice, [count, z, y, x]."""
    ks = sorted(((a, b, c) for a in range(-2, 3) for b in range(-2, 3) for c in range(-2, 3)),
                key=lambda k: (k[0] ** 2 + k[1] ** 2 + k[2] ** 2, k))[:count]
    i = torch.arange(ns, device=dev, dtype=torch.float64)
    return torch.stack([torch.exp(2j * math.pi / ns * (k[0] * i[None, None, :] + k[1] * i[None, :, None]
                                                      + k[2] * i[:, None, None])) for k in ks])


def _smooth_sources(case, seed):
    """gamma_4 V P rho with plane waves for V: one spin, every fourth slice, smooth in space."""
    ns, nt, n, dev = case["ns"], case["nt"], case["nrhs"], _dev()
    w = _waves(ns, 27, dev) / math.sqrt(3.0 * ns ** 3)
    out = torch.zeros((n, nt, ns, ns, ns, 4, 3), dtype=C128, device=dev)
    code = torch.randint(0, 4, (n, nt, 27, 3), generator=_gen(seed, 2), device=dev)
    z4 = torch.tensor([1, 1j, -1, -1j], dtype=C128, device=dev)[code]
    for i in range(n):
        t0 = (i // 4) % min(4, nt)
        out[i, t0::4, :, :, :, i % 4] = torch.einsum("tkc,kzyx->tzyxc", z4[i, t0::4], w)
    return out


def _evecs(ns, nt, nv, seed):
    """Unit vectors in place of the eigenvectors, [nt, nv, V3, 3]."""
    v = _randn((nt, nv, ns ** 3, 3), _gen(seed, 3))
    return v / v.flatten(2).norm(dim=2)[..., None, None]


def _sinks_sol(case, seed):
    """Solutions that fall off in time from their source slice, [nrhs, V, 4, 3]."""
    ns, nt, n = case["ns"], case["nt"], case["nrhs"]
    x = _randn((n, nt, ns ** 3, 4, 3), _gen(seed, 4))
    t = torch.arange(nt, device=x.device, dtype=torch.float64)
    for i in range(n):
        x[i] *= torch.exp(-0.15 * torch.minimum((t - i) % nt, (i - t) % nt))[:, None, None, None]
    return x


def _blist(case):
    if case["kind"] == "sources":
        ntot = case["tdil"] * 4 * case["ldil"]
        return [(5 + i) % ntot for i in range(case["nrhs"])]
    nl = case["nb"] // 4
    return [(case["t0"] * 4) * nl + i for i in range(case["nb"])]


def _halves(case):
    return (case["nt"] * case["ns"] ** 3 // 2, 12, case["nrhs"])


_MODES = {"clovinv": L.HOP_CLOVINV, "xpay": L.HOP_CLOVINV_XPAY, "apply": L.HOP_APPLY}
_PRECS = {"fp64": L.PREC_FP64, "fp32": L.PREC_FP32}
_CHANNELS = {"pion": L.CH_PION, "rho": L.CH_RHO, "scalar": L.CH_SCALAR, "pipi": L.CH_PIPI_I2}


def _half_fields(case, seed):
    dt = C128 if case["prec"] == "fp64" else torch.complex64
    g = _gen(seed, 5)
    return [_randn(_halves(case), g).to(dt) for _ in range(1 if case["mode"] == "clovinv" else 2)]


def _lines(case, seed):
    """Sink coefficients (falling off in time) and noise codes of the correlator's lines."""
    n = 4 if case["channel"] == "pipi" else 2
    nt, nv, nb, dev = case["nt"], case["nv"], case["nb"], _dev()
    g = _gen(seed, 6)
    t = (torch.arange(nt, device=dev, dtype=torch.float64) - case["t0"]) % nt
    f = torch.exp(-0.1 * torch.minimum(t, nt - t))[None, :, None, None]
    coef = [(_randn((nb, nt, 4, nv), g) * f).contiguous() for _ in range(n)]
    codes = [torch.randint(0, 4, (nt, 4, nv), generator=g, device=dev).to(torch.uint8) for _ in range(n)]
    return coef, codes


def _moms(case):
    return [(0, 0, 1), (0, 1, 1), (1, 1, 1), (0, 0, 2), (0, -1, 0), (1, 0, -2), (2, 1, 0)][: case["nmom"]]


# ------------------------------------------------------------------ the measured interface
def prepare(case, seed):
    k, dev = case["kind"], _dev()
    s = dict(case=case, ctx=_ctx())
    if k == "corr":
        s["lat"] = L.lattice(4, case["nt"], XI)
        s["coef"], s["codes"] = _lines(case, seed)
        s["dil"] = L.dilution((L.DIL_FULL, 0), (L.DIL_FULL, 0), (L.DIL_INTERLACE, case["nb"] // 4))
        s["b"], s["out"] = _blist(case), torch.empty(case["nt"], dtype=C128, device=dev)
        return s
    ns, nt = case["ns"], case["nt"]
    s["lat"] = L.lattice(ns, nt, XI)
    if k in ("solve", "apply", "dslash"):
        s["u"] = _links(ns, nt, seed)
    if k == "solve":
        s["rhs"] = _smooth_sources(case, seed)
        s["sol"] = torch.empty_like(s["rhs"])
    elif k == "apply":
        s["in"] = _randn((case["nrhs"], nt, ns, ns, ns, 4, 3), _gen(seed, 7))
        s["out"] = torch.empty_like(s["in"])
    elif k == "dslash":
        s["f"] = _half_fields(case, seed)
        s["out"] = torch.empty_like(s["f"][0])
    elif k == "eigvecs":
        u = _raw_links(ns, nt, seed)
        s["u"] = _stout(_stout(u, STOUT, 4), 2, 3).contiguous()
        s["evals"] = torch.empty((nt, case["nv"]), dtype=torch.float64, device=dev)
        s["evecs"] = torch.empty((nt, case["nv"], ns ** 3, 3), dtype=C128, device=dev)
    else:
        s["v"] = _evecs(ns, nt, case["nv"], seed)
        if k == "sources":
            s["noise"] = int(seed) % 50000
            s["dil"] = L.dilution((L.DIL_INTERLACE, case["tdil"]), (L.DIL_FULL, 0), (L.DIL_INTERLACE, case["ldil"]))
            s["b"] = _blist(case)
            s["out"] = torch.empty((case["nrhs"], nt, ns, ns, ns, 4, 3), dtype=C128, device=dev)
            s["codes"] = torch.empty((nt, 4, case["nv"]), dtype=torch.uint8, device=dev)
        elif k == "sinks":
            s["sol"] = _sinks_sol(case, seed)
            s["out"] = torch.empty((case["nrhs"], nt, 4, case["nv"]), dtype=C128, device=dev)
        else:
            s["mom"] = _moms(case)
            s["out"] = torch.empty((case["nmom"], nt, case["nv"], case["nv"]), dtype=C128, device=dev)
    return s


def run(s):
    c, ctx, lat = s["case"], s["ctx"], s["lat"]
    k = c["kind"]
    if k == "solve":
        prm = L.solver_params(tol=1e-10, rhs_block=c["block"])
        L.dirac_solve_batch(ctx, lat, s["u"], c["m0"], CSW, s["rhs"], s["sol"], c["nrhs"], prm)
        return [s["sol"][: _checked(c)], s["sol"][_checked(c):]]
    if k == "apply":
        L.laph_dirac_apply(ctx, lat, s["u"], c["m0"], CSW, s["in"], s["out"], c["nrhs"])
        return s["out"]
    if k == "dslash":
        z = s["f"][1] if c["mode"] != "clovinv" else None
        L.laph_dslash_eo(ctx, lat, s["u"], 0.02, CSW, c["parity"], _MODES[c["mode"]], _PRECS[c["prec"]], s["f"][0], z,
                         s["out"], c["nrhs"])
        return s["out"]
    if k == "eigvecs":
        L.laph_eigvecs(ctx, lat, s["u"], c["nv"], s["evals"], s["evecs"])
        return [s["evals"], s["evecs"]]
    if k == "sources":
        L.laph_make_sources(ctx, lat, s["v"], c["nv"], s["noise"], 7, s["dil"], s["b"], s["out"], s["codes"])
        return [s["out"], s["codes"]]
    if k == "sinks":
        L.laph_sinks(ctx, lat, s["v"], c["nv"], s["sol"], c["nrhs"], s["out"])
        return s["out"]
    if k == "corr":
        L.correlate(ctx, lat, _CHANNELS[c["channel"]], c["t0"], c["nv"], s["dil"], s["b"], s["coef"], s["codes"],
                    s["out"])
        return s["out"]
    L.laph_mom_overlaps(ctx, lat, s["v"], c["nv"], s["mom"], s["out"])
    return s["out"]


def work(case):
    """Inputs read once, outputs written once; flops of the operator (1824 per site and
    right-hand side of a hop with its site term) or of the contraction (8 per complex multiply-add)."""
    k = case["kind"]
    if k == "corr":
        nt, nv, nb = case["nt"], case["nv"], case["nb"]
        n = {"pion": 1, "scalar": 1, "rho": 3, "pipi": 4}[case["channel"]]
        flops = 8.0 * nt * nb * nb * 4 * nv * n + (16.0 * nt * nb ** 3 if case["channel"] == "pipi" else 0)
        lines = 4 if case["channel"] == "pipi" else 2
        return dict(bytes=lines * (16.0 * nb * nt * 4 * nv + 4.0 * nv * nt) + 16.0 * nt, flops=flops)
    v = case["ns"] ** 3 * case["nt"]
    if k in ("solve", "apply", "dslash"):
        n, links = case["nrhs"], 16.0 * 36 * v
        if k == "dslash":
            el = 16.0 if case["prec"] == "fp64" else 8.0
            return dict(bytes=links + el * 6 * v * n * (2 if case["mode"] == "clovinv" else 3), flops=912.0 * v * n)
        steps = 2 * case["iters"] if k == "solve" else 1
        return dict(bytes=links + 16.0 * 24 * v * n, flops=1824.0 * v * n * steps)
    nv = case["nv"]
    ev = 16.0 * 3 * v * nv
    if k == "eigvecs":
        m = 2 * nv + 32   # a Krylov space of this dimension with order-16 filters, and its orthogonalisation
        return dict(bytes=16.0 * 36 * v + ev, flops=v * (16.0 * m * 500 + 8.0 * 3 * m * m))
    if k == "sources":
        used = case["nrhs"] / (case["tdil"] * case["ldil"])
        return dict(bytes=ev * min(1.0, used) + 16.0 * 12 * v * case["nrhs"], flops=2.0 * 3 * v * nv * used)
    if k == "sinks":
        n = case["nrhs"]
        return dict(bytes=ev + 16.0 * 12 * v * n + 16.0 * n * case["nt"] * 4 * nv, flops=8.0 * 12 * v * nv * n)
    return dict(bytes=ev + 16.0 * case["nmom"] * case["nt"] * nv * nv, flops=8.0 * 3 * v * nv * nv * case["nmom"])


# ------------------------------------------------------------------ 64-bit values
def _checked(case):
    """Right-hand sides of a solve whose exact solution is worked out (one by one)."""
    return min(case["nrhs"], 2 if case["ns"] ** 3 * case["nt"] <= 16 ** 3 * 32 else 1)


def _exact_dslash(case, seed):
    ns, nt, n, p = case["ns"], case["nt"], case["nrhs"], case["parity"]
    K = _Dirac(_links(ns, nt, seed), 0.02)
    f = [x.to(C128) for x in _half_fields(case, seed)]
    i = torch.arange(ns, device=_dev())
    t = torch.arange(nt, device=_dev())
    odd = ((t[:, None, None, None] + i[:, None, None] + i[:, None] + i) % 2).reshape(-1)
    here = torch.nonzero(odd == p).flatten()
    there = torch.nonzero(odd != p).flatten()
    out = torch.empty_like(f[0])
    for a in range(0, n, 4):   # a few right-hand sides at a time
        full = torch.zeros((min(4, n - a), nt * ns ** 3, 12), dtype=C128, device=_dev())
        full[:, there] = f[0][:, :, a:a + 4].permute(2, 0, 1)
        h = K.hop(full.reshape(-1, nt, ns, ns, ns, 4, 3)).reshape(full.shape)[:, here]
        site = K.a.reshape(-1, 12, 12)[here]
        if case["mode"] == "apply":
            y = h + torch.einsum("sij,nsj->nsi", site, f[1][:, :, a:a + 4].permute(2, 0, 1))
        else:
            y = torch.linalg.solve(site, h.permute(1, 2, 0)).permute(2, 0, 1)
            if case["mode"] == "xpay":
                y = f[1][:, :, a:a + 4].permute(2, 0, 1) - y
        out[:, :, a:a + 4] = y.permute(1, 2, 0)
    return out


def _philox_codes(n, key0):
    """Low two bits of word 0 of Philox4x32-10(counter (i, 0, 0, 0), key (key0, 0x4C415048))."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64)] + [np.zeros(n, dtype=np.uint64)] * 3
    k0, k1 = np.uint64(key0), np.uint64(0x4C415048)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ k0, b & m32, (a >> np.uint64(32)) ^ c[3] ^ k1, a & m32]
    return (c[0] & np.uint64(3)).astype(np.uint8)


def _exact_sources(case, seed):
    ns, nt, nv, dev = case["ns"], case["nt"], case["nv"], _dev()
    codes = torch.from_numpy(_philox_codes(nt * 4 * nv, (7 << 16) | int(seed) % 50000).reshape(nt, 4, nv)).to(dev)
    rho = torch.tensor([1, 1j, -1, -1j], dtype=C128, device=dev)[codes.long()]
    v = _evecs(ns, nt, nv, seed)
    out = torch.zeros((case["nrhs"], nt, ns ** 3, 4, 3), dtype=C128, device=dev)
    for i, b in enumerate(_blist(case)):
        bl, bs, bt = b % case["ldil"], b // case["ldil"] % 4, b // (4 * case["ldil"])
        y = torch.einsum("tnxc,tn->txc", v[bt::case["tdil"], bl::case["ldil"]], rho[bt::case["tdil"], bs, bl::case["ldil"]])
        out[i, bt::case["tdil"], :, (bs + 2) % 4] = y      # gamma_4 swaps the spin pairs
    return [out.reshape(-1, nt, ns, ns, ns, 4, 3), codes]


def _exact_sinks(case, seed):
    v, x = _evecs(case["ns"], case["nt"], case["nv"], seed), _sinks_sol(case, seed)
    out = torch.empty((case["nrhs"], case["nt"], 4, case["nv"]), dtype=C128, device=_dev())
    for t in range(case["nt"]):
        out[:, t] = torch.einsum("nk,ika->ian", v[t].flatten(1).conj(), x[:, t].transpose(2, 3).flatten(1, 2))
    return out


def _exact_eigvecs(case, seed):
    ns, nt, nv = case["ns"], case["nt"], case["nv"]
    if ns > 8:
        return None
    u = _stout(_stout(_raw_links(ns, nt, seed), STOUT, 4), 2, 3)
    n = 3 * ns ** 3
    evals, evecs = [], []
    for t in range(nt):
        eye = torch.eye(n, dtype=C128, device=_dev()).reshape(n, 1, ns, ns, ns, 3)
        lap = 6.0 * eye
        for mu in range(3):
            um = u[t:t + 1, ..., mu, :, :]
            lap = lap - torch.einsum("tzyxij,ntzyxj->ntzyxi", um, _fwd(eye, mu, 1))
            lap = lap - _bwd(torch.einsum("tzyxji,ntzyxj->ntzyxi", um.conj(), eye), mu, 1)
        w, y = torch.linalg.eigh(lap.reshape(n, n).transpose(0, 1).cpu())
        y = y[:, :nv].transpose(0, 1).to(_dev())
        a = y.abs()
        j = (a >= a.max(dim=1, keepdim=True).values * (1 - 1e-8)).to(torch.uint8).argmax(dim=1)
        lead = y[torch.arange(nv, device=y.device), j]
        evals.append(w[:nv].to(_dev()))
        evecs.append((y * (lead.conj() / lead.abs())[:, None]).reshape(nv, ns ** 3, 3))
    return [torch.stack(evals), torch.stack(evecs)]


def _exact_corr(case, seed):
    nt, nv, t0, nl = case["nt"], case["nv"], case["t0"], case["nb"] // 4
    coef, codes = _lines(case, seed)
    dev = _dev()
    z4 = torch.tensor([1, 1j, -1, -1j], dtype=C128, device=dev)
    rho = []
    for c in codes:
        r = torch.zeros((case["nb"], 4, nv), dtype=C128, device=dev)
        for i in range(case["nb"]):
            r[i, i // nl, i % nl::nl] = z4[c[t0, i // nl, i % nl::nl].long()]
        rho.append(r)
    gm = [torch.tensor(g, dtype=C128, device=dev) for g in _gammas()]
    g5 = gm[0] @ gm[1] @ gm[2] @ gm[3]

    def sink(a, b, w):
        return torch.einsum("btxn,xy,ctyn->tbc", coef[a].conj(), w, coef[b])

    def source(a, b, w):
        return -torch.einsum("bxn,xy,cyn->bc", rho[a].conj(), w, rho[b])

    def meson(a, b, c):
        w = (g5 @ gm[3]).conj().T @ c
        return -(sink(a, b, w) * source(a, b, w).conj()).sum((1, 2))

    if case["channel"] == "pion":
        out = meson(0, 1, gm[3] @ g5)
    elif case["channel"] == "scalar":
        out = meson(0, 1, gm[3])
    elif case["channel"] == "rho":
        out = sum(meson(0, 1, gm[3] @ gm[k]) for k in range(3)) / 3.0
    else:
        c = gm[3] @ g5
        w = (g5 @ gm[3]).conj().T @ c
        x = torch.einsum("tad,tcb,ab,cd->t", sink(0, 3, w), sink(2, 1, w), source(0, 1, w).conj(), source(2, 3, w).conj())
        out = meson(0, 1, c) * meson(2, 3, c) - x
    return torch.roll(out, -t0)


def _exact_overlaps(case, seed):
    ns, nt = case["ns"], case["nt"]
    v = _evecs(ns, nt, case["nv"], seed)
    i = torch.arange(ns, device=_dev(), dtype=torch.float64)
    out = []
    for p in _moms(case):
        ph = torch.exp(-2j * math.pi / ns * (p[0] * i + p[1] * i[:, None] + p[2] * i[:, None, None])).reshape(-1)
        out.append(torch.stack([v[t].flatten(1).conj() @ (v[t] * ph[None, :, None]).flatten(1).T for t in range(nt)]))
    return torch.stack(out)


def exact(case, seed):
    k = case["kind"]
    if k == "solve":
        K = _Dirac(_links(case["ns"], case["nt"], seed), case["m0"])
        b = _smooth_sources(case, seed)
        return [torch.cat([K.solve(b[i:i + 1]) for i in range(_checked(case))]), None]
    if k == "apply":
        K = _Dirac(_links(case["ns"], case["nt"], seed), case["m0"])
        f = _randn((case["nrhs"], case["nt"]) + 3 * (case["ns"],) + (4, 3), _gen(seed, 7))
        return torch.cat([K(f[i:i + 2]) for i in range(0, case["nrhs"], 2)])
    return {"dslash": _exact_dslash, "sources": _exact_sources, "sinks": _exact_sinks, "eigvecs": _exact_eigvecs,
            "corr": _exact_corr, "overlaps": _exact_overlaps}[k](case, seed)
