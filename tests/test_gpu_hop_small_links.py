"""The FP64 hop on links and hop weights far below one: fields of scaled SU(3) links, one small link
among ordinary ones, spatial weights of a large anisotropy (a source whose neighbours in space see nothing
else), a slice whose time links are zero (an open boundary), and one small column.

Tolerance: FP64 arithmetic on 48 products, 1e-14 of the largest entry that the same neighbours give at
the site and, for scaled links, of the scaled result."""
import numpy as np
import pytest
import torch

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import MODES, from_eo, reference, to_eo

pytestmark = [pytest.mark.gpu, requires_gpu]

NS, NT = 4, 6


def _hop(u, xi, p, x):
    L = lib()
    out = empty(x.shape, torch.complex128)
    L.laph_dslash_eo(context(), L.lattice(NS, NT, xi), dev(u), 0.02, 1.0, p, MODES["apply"], L.PREC_FP64, dev(x),
                     dev(np.zeros_like(x)), out, x.shape[2])
    return host(out)


def _ref(u, xi, p, x):
    return reference(WilsonClover(u, 0.02, 1.0, xi), NS, NT, p, "apply", x, np.zeros_like(x))


@pytest.mark.parametrize("scale", [1.0, 0.3, 1e-2, 1e-6, 1e-9, 1e-200])
def test_scaled_links(scale):
    u = scale * gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)
    x = synth.random_complex((NS ** 3 * NT // 2, 12, 3), seed=4)
    for p in (0, 1):
        got, ref = _hop(u, 3.5, p, x), _ref(u, 3.5, p, x)
        assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()


@pytest.mark.parametrize("part", ["matrix", "row", "column"])
def test_one_small_link(part):
    """Only the neighbour behind the small link carries a field, so its product stands alone at a site."""
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=8), 0.1, 2, spatial_only=False)
    t, z, y, x0 = 1, 2, 1, 3
    sel = {"matrix": (slice(None), slice(None)), "row": (1, slice(None)), "column": (slice(None), 1)}[part]
    u[t, z, y, x0, 3][sel] *= 1e-8
    x = np.zeros((2, NT, NS, NS, NS, 4, 3), dtype=complex)
    x[0, t, z, y, x0] = synth.random_complex((4, 3), seed=1)           # seen through U^dag at t + 1
    x[1, t + 1, z, y, x0] = synth.random_complex((4, 3), seed=2)       # seen through U at t
    for r, (site, q) in enumerate(((t + 1, t), (t, t + 1))):
        p = (site + z + y + x0) % 2
        eo = to_eo(x, 1 - p, NS, NT)
        got, ref = (from_eo(f, p, NS, NT)[r, site, z, y, x0] for f in (_hop(u, 3.5, p, eo), _ref(u, 3.5, p, eo)))
        # colour by colour: a small row or column makes one colour small
        assert np.all(np.abs(got - ref).max(0) <= 1e-14 * np.abs(ref).max(0))


@pytest.mark.parametrize("xi", [3.5, 16.0, 1e4, 1e8])
def test_weights_of_a_large_anisotropy(xi):
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=9), 0.1, 2, spatial_only=False)
    x = np.zeros((1, NT, NS, NS, NS, 4, 3), dtype=complex)
    x[0, 2] = synth.random_complex((NS, NS, NS, 4, 3), seed=3)          # one slice: slice 2 sees space only
    for p in (0, 1):
        eo = to_eo(x, 1 - p, NS, NT)
        got, ref = (from_eo(f, p, NS, NT)[0, 2] for f in (_hop(u, xi, p, eo), _ref(u, xi, p, eo)))
        assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()


def test_open_boundary_in_time():
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=10), 0.1, 2, spatial_only=False)
    u[-1, :, :, :, 3] = 0.0
    x = synth.random_complex((NS ** 3 * NT // 2, 12, 2), seed=5)
    for p in (0, 1):
        got, ref = _hop(u, 3.5, p, x), _ref(u, 3.5, p, x)
        assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()
