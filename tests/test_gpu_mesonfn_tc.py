"""correlate() through the tensor-core meson functions (mesonfn_tc.cu) against the coefficient-space
sums in numpy, at the edges of its kernels: K = 4 N_v below and above a sub-chunk and a drain, tiles of
64 rows, source matrices with one nonzero per row (full spin and LapH interlace dilution) and dense
ones (no spin or LapH dilution), nb above the shared-memory pi pi kernel (nb = 80), and NaN inputs.

Tolerance: a meson function is within dM = 8 (4 N_v) 2^-52.5 max|a| max|b| of the exact sum (entry
rounding and dropped digit pairs, both parts); this goes linearly through the correlator sums, whose
FP64 rounding adds at most 1e-13 of the sum of moduli."""
import numpy as np
import pytest

import synth
from oracle.gamma import GAMMA
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

G5 = GAMMA[0] @ GAMMA[1] @ GAMMA[2] @ GAMMA[3]
C = {"pion": [GAMMA[3] @ G5], "rho": [GAMMA[3] @ g for g in GAMMA[:3]], "scalar": [GAMMA[3]], "pipi": [GAMMA[3] @ G5]}


def _proj(kind, J, N, b, i):
    return [True, i == b, (J * i) // N == b, i % max(J, 1) == b][kind]


def _count(kind, J, N):
    return [1, N, J, J][kind]


def _inputs(channel, nt, nv, dil, nb, t0, seed):
    nlines = 4 if channel == "pipi" else 2
    nS, nL = _count(*dil[1], 4), _count(*dil[2], nv)
    total = _count(*dil[0], nt) * nS * nL
    bT = next(b for b in range(_count(*dil[0], nt)) if _proj(*dil[0], nt, b, t0))
    bs = [(bT * nS * nL + i) % total for i in range(nb)]
    coef = [synth.random_complex((nb, nt, 4, nv), seed=seed + k) for k in range(nlines)]
    rng = np.random.default_rng(seed)
    codes = [rng.integers(0, 4, (nt, 4, nv)).astype(np.uint8) for _ in range(nlines)]
    rho = []
    for c in codes:
        r = np.zeros((nb, 4, nv), dtype=complex)
        for i, b in enumerate(bs):
            for a in range(4):
                for n in range(nv):
                    if (_proj(*dil[0], nt, b // (nL * nS), t0) and _proj(*dil[1], 4, b // nL % nS, a)
                            and _proj(*dil[2], nv, b % nL, n)):
                        r[i, a, n] = 1j ** c[t0, a, n]
        rho.append(r)
    return bs, coef, codes, rho


def _run(channel, nt, nv, dil, bs, t0, coef, codes):
    L = lib()
    ch = {"pion": L.CH_PION, "rho": L.CH_RHO, "scalar": L.CH_SCALAR, "pipi": L.CH_PIPI_I2}[channel]
    out = empty((nt,), dev(coef[0]).dtype)
    L.correlate(context(), L.lattice(4, nt, 3.5), ch, t0, nv, L.dilution(*dil), bs, [dev(c) for c in coef],
                [dev(c) for c in codes], out)
    return host(out)


@pytest.mark.parametrize("channel,nt,nv,dil,nb", [
    ("pion", 2, 1, ((1, 0), (1, 0), (0, 0)), 4),
    ("rho", 4, 7, ((1, 0), (0, 0), (0, 0)), 1),
    ("scalar", 4, 24, ((3, 2), (3, 2), (3, 8)), 16),
    ("pipi", 4, 16, ((1, 0), (1, 0), (3, 8)), 32),
    ("pipi", 2, 10, ((1, 0), (0, 0), (0, 0)), 3),
    ("pipi", 2, 160, ((1, 0), (1, 0), (3, 20)), 80),
])
def test_correlate_tensor_core(channel, nt, nv, dil, nb):
    t0 = 1
    bs, coef, codes, rho = _inputs(channel, nt, nv, dil, nb, t0, 91)
    got = _run(channel, nt, nv, dil, bs, t0, coef, codes)
    g5g4 = G5 @ GAMMA[3]
    dm = 8.0 * 4 * nv * 2.0 ** -52.5 * max(np.abs(c).max() for c in coef) ** 2

    def snk(a, b, c):
        return np.einsum("btxn,xy,ctyn->tbc", coef[a].conj(), g5g4.conj().T @ c, coef[b], optimize=True)

    def src(a, b, c):
        return -np.einsum("bxn,xy,cyn->bc", rho[a].conj(), g5g4.conj().T @ c, rho[b], optimize=True)

    def meson(a, b, c):
        m, s = snk(a, b, c), src(a, b, c).conj()
        return -(m * s).sum((1, 2)), ((dm + 1e-13 * np.abs(m)) * np.abs(s)).sum((1, 2))

    if channel == "pipi":
        c = C["pipi"][0]
        (c12, e12), (c34, e34) = meson(0, 1, c), meson(2, 3, c)
        m14, m32, s12, s34 = snk(0, 3, c), snk(2, 1, c), src(0, 1, c), src(2, 3, c)
        x = np.einsum("tad,tcb,ab,cd->t", m14, m32, s12.conj(), s34.conj(), optimize=True)
        ex = [np.einsum("tad,tcb,ab,cd->t", np.abs(m14) + p, np.abs(m32) + q, np.abs(s12), np.abs(s34), optimize=True)
              for p, q in ((0, 0), (dm, dm))]
        ref = c12 * c34 - x
        tol = np.abs(c12) * e34 + np.abs(c34) * e12 + e12 * e34 + (ex[1] - ex[0]) + 1e-13 * ex[0]
    else:
        parts = [meson(0, 1, c) for c in C[channel]]
        ref, tol = sum(p[0] for p in parts) / len(parts), sum(p[1] for p in parts) / len(parts)
    assert np.all(np.abs(got - np.roll(ref, -t0)) <= np.roll(tol, -t0) + 1e-15)


@pytest.mark.parametrize("channel", ["pion", "pipi"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_correlate_non_finite_stays_on_its_slice(channel, bad):
    nt, nv, nb, dil, t0 = 4, 8, 8, ((1, 0), (1, 0), (3, 2)), 2
    bs, coef, codes, rho = _inputs(channel, nt, nv, dil, nb, t0, 7)
    coef[1][3, 3, 2, 5] = bad
    got = _run(channel, nt, nv, dil, bs, t0, coef, codes)
    finite = np.isfinite(got)
    assert not finite[1] and finite[[0, 2, 3]].all()     # slice 3 is dt = 1
