"""The exact-slice tensor-core GEMM behind laph_sinks at the edges of its tiles: rows n around 64,
columns 4 nrhs around 64, K = 3 ns^3 below one sub-chunk's multiple and above one 512-real-k drain.

Tolerance: an entry is rounded by at most 2^-56 of its scale (at most twice the largest entry of its
row or column, per real part), and the digit pairs left out are below 1.2 * 7 * 2^12 * 2^-68 per real
product, so a part of a coefficient is within 2 K * 4 max|V| max|X| * 2^-52.5 of the exact sum; the
FP64 reference adds its own rounding, at most K 2^-52 sum |V||X| (and far less in practice)."""
import numpy as np
import pytest

import synth
from oracle import laph as olaph
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nv,nrhs", [(2, 1, 1), (2, 7, 16), (4, 63, 17), (4, 64, 15), (6, 65, 16), (8, 128, 3)])
def test_exact_gemm_tile_edges(ns, nv, nrhs):
    L = lib()
    nt, K = 2, 3 * ns ** 3
    V = synth.random_complex((nt, nv, ns ** 3, 3), seed=31 + nv)
    X = synth.random_spinor(ns, nt, seed=32 + nrhs, nrhs=nrhs)
    coef = empty((nrhs, nt, 4, nv), dev(X).dtype)
    L.laph_sinks(context(), L.lattice(ns, nt, 3.5), dev(V), nv, dev(X), nrhs, coef)
    ref = olaph.sinks(V, X)
    scale = np.einsum("tnxc,itxac->itan", np.abs(V), np.abs(X).reshape(nrhs, nt, ns ** 3, 4, 3))
    vmax = max(np.abs(V.real).max(), np.abs(V.imag).max())
    xmax = max(np.abs(X.real).max(), np.abs(X.imag).max())
    bound = 8.0 * K * vmax * xmax * 2.0 ** -52.5 + K * 2.0 ** -52 * scale
    assert np.all(np.abs(host(coef) - ref) <= 2 * bound)
