"""The exact-slice GEMM on rows and columns at the ends of the FP64 range, where the fixed point over a
power of two per row has no room, and overlaps of vectors with NaN: row 0 of the eigenvectors, one
solution or one line is scaled, the rest is of size one, so that the products are ordinary FP64 numbers.

Tolerance: every entry is compared after the scale is taken out of it, so it is that of ordinary rows:
8 K 2^-52.5 max|a| max|b| (entry rounding and dropped digit pairs, both parts)."""
import numpy as np
import pytest
import torch

import synth
from oracle import laph as olaph
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_mesonfn_tc import _inputs, _run

pytestmark = [pytest.mark.gpu, requires_gpu]


def _overlaps(v, nv, ns, nt, mom):
    L = lib()
    out = empty((len(mom), nt, nv, nv), torch.complex128)
    L.laph_mom_overlaps(context(), L.lattice(ns, nt, 3.5), dev(v), nv, mom, out)
    return host(out)


def _overlaps_ref(v, ns, mom):
    i = np.arange(ns)
    out = []
    for p in mom:
        ph = np.exp(-2j * np.pi / ns * (p[0] * i + p[1] * i[:, None] + p[2] * i[:, None, None])).reshape(-1)
        out.append(np.einsum("tnxc,x,tmxc->tnm", v.conj(), ph, v))
    return np.array(out)


@pytest.mark.parametrize("power", [-950, -1000, -1020])
def test_overlaps_of_a_tiny_vector(power):
    ns, nt, nv, mom = 4, 2, 5, [(0, 0, 1), (1, 0, -1)]
    v = synth.random_complex((nt, nv, ns ** 3, 3), seed=1)
    ref = _overlaps_ref(v, ns, mom)
    w = v.copy()
    w[:, 0] *= 2.0 ** power
    got = _overlaps(w, nv, ns, nt, mom)
    got[:, :, 0, 1:] *= 2.0 ** -(power // 2)
    got[:, :, 0, 1:] *= 2.0 ** -(power - power // 2)
    got[:, :, 1:, 0] *= 2.0 ** -(power // 2)
    got[:, :, 1:, 0] *= 2.0 ** -(power - power // 2)
    K = 3 * ns ** 3
    bound = 8 * K * 2.0 ** -52.5 * np.abs(v).max() ** 2 + 400 * K * 2.0 ** (-1074 - power)   # subnormal terms of the sum
    sel = np.ones((nv, nv), dtype=bool)
    sel[0, 0] = False
    assert np.abs(got - ref)[:, :, sel].max() <= bound
    assert np.all(np.abs(got[:, :, 0, 0]) <= 1e-300)


def test_overlaps_of_a_huge_vector():
    """The phase takes a part of the largest FP64 numbers out of range, in FP64 and here."""
    ns, nt, nv, mom, big = 8, 2, 3, [(1, 0, 0)], 2.0 ** 1023
    w = 1e-3 * synth.random_complex((nt, nv, ns ** 3, 3), seed=2)
    w[:, 0, 1, 0] = 1.99 + 1.99j                      # at x = 1, where the phase is e^(-i pi / 4)
    ref = _overlaps_ref(w, ns, mom)
    x = w.copy()
    x[:, 0] = x[:, 0] * big
    got = _overlaps(x, nv, ns, nt, mom)
    assert not np.isfinite(got[:, :, :, 0]).any()
    got[:, :, 0, 1:] /= big
    assert np.abs(got - ref)[:, :, :, 1:].max() <= 8 * 3 * ns ** 3 * 2.0 ** -52.5 * 3 * np.abs(w[:, 1:]).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_overlaps_with_a_vector_that_is_not_finite(bad):
    ns, nt, nv, mom = 4, 2, 5, [(0, 0, 1), (1, 0, -1)]
    v = synth.random_complex((nt, nv, ns ** 3, 3), seed=3)
    ref = _overlaps_ref(v, ns, mom)
    v[1, 2, 17, 1] = bad
    got = _overlaps(v, nv, ns, nt, mom)
    hit = np.zeros(got.shape, dtype=bool)
    hit[:, 1, 2] = hit[:, 1, :, 2] = True
    assert np.array_equal(~np.isfinite(got), hit)
    assert np.abs(got - ref)[~hit].max() <= 8 * 3 * ns ** 3 * 2.0 ** -52.5 * np.abs(v[0]).max() ** 2 * 2


@pytest.mark.parametrize("power", [-950, -1000, -1020])
def test_sinks_of_a_tiny_solution(power):
    L = lib()
    ns, nt, nv, nrhs = 4, 2, 6, 3
    V, X = synth.random_complex((nt, nv, ns ** 3, 3), seed=4), synth.random_spinor(ns, nt, seed=5, nrhs=nrhs)
    ref = olaph.sinks(V, X)
    Y = X.copy()
    Y[1] *= 2.0 ** power
    out = empty((nrhs, nt, 4, nv), torch.complex128)
    L.laph_sinks(context(), L.lattice(ns, nt, 3.5), dev(V), nv, dev(Y), nrhs, out)
    got = host(out)
    got[1] *= 2.0 ** -(power // 2)
    got[1] *= 2.0 ** -(power - power // 2)
    K = 3 * ns ** 3
    bound = 8 * K * 2.0 ** -52.5 * np.abs(V).max() * np.abs(X).max() + 400 * K * 2.0 ** (-1074 - power)
    assert np.abs(got - ref).max() <= bound


def test_correlator_of_a_tiny_line():
    nt, nv, nb, dil, t0, power = 4, 8, 8, ((1, 0), (1, 0), (3, 2)), 2, -1000
    bs, coef, codes, _ = _inputs("pion", nt, nv, dil, nb, t0, 11)
    ref = _run("pion", nt, nv, dil, bs, t0, coef, codes)
    got = _run("pion", nt, nv, dil, bs, t0, [coef[0] * 2.0 ** power, coef[1]], codes)
    assert np.abs(got * 2.0 ** 500 * 2.0 ** (-power - 500) - ref).max() <= 1e-13 * np.abs(ref).max()
