"""NaN and infinities in the FP64 hop: what the clover blocks or an operand bring in reaches exactly the
outputs that FP64 arithmetic would give it.

Blocks: a mass or clover coefficient that is not finite makes every entry of A x non-finite (each row has
a non-finite diagonal, or all of its entries are NaN), and csw = 0 with m0 = -(1 + 3 / xi) makes A = 0, whose
inverse is NaN throughout.  Operands: an entry (spin a, any colour) of a neighbour enters the two half
spinors u -+ G d that hold spin a, all colours of each through the link, and with a block inverse the whole
chirality; an entry of the site term's operand enters the six rows of its chirality (apply) or its own
component (xpay).  Masks are compared component by component, so there is no tolerance."""
import numpy as np
import pytest
import torch

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import MODES, from_eo, reference, to_eo

pytestmark = [pytest.mark.gpu, requires_gpu]

NS, NT, XI = 4, 6, 4.0   # 1 / xi is exact, so that m0 = -1.75 cancels the hop weights exactly
# the spin that shares a half spinor with spin a in direction mu (G_1 and G_2 swap the lower pair)
PARTNER = [[3, 2, 1, 0], [3, 2, 1, 0], [2, 3, 0, 1], [2, 3, 0, 1]]


def _links():
    return gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)


def _hop(u, m0, csw, mode, p, x, z):
    L = lib()
    out = empty(x.shape, torch.complex128)
    L.laph_dslash_eo(context(), L.lattice(NS, NT, XI), dev(u), m0, csw, p, MODES[mode], L.PREC_FP64, dev(x),
                     None if mode == "clovinv" else dev(z), out, x.shape[2])
    return host(out)


@pytest.mark.parametrize("modes,m0,csw", [
    (("clovinv", "xpay"), -(1.0 + 3.0 / XI), 0.0),
    (("clovinv", "xpay", "apply"), np.nan, 1.0),
    (("apply",), np.inf, 1.0),
    (("clovinv", "xpay", "apply"), 0.1, np.nan),
])
def test_blocks_that_are_not_finite(modes, m0, csw):
    u = _links()
    vh, nr = NS ** 3 * NT // 2, 2
    x, z = synth.random_complex((vh, 12, nr), seed=4), synth.random_complex((vh, 12, nr), seed=5)
    x[::3] = 0.0
    for mode in modes:
        for p in (0, 1):
            got = _hop(u, m0, csw, mode, p, x, z)
            assert not np.isfinite(got).any()


def test_apply_with_a_mass_that_is_not_finite():
    L = lib()
    x = synth.random_spinor(NS, NT, seed=6, nrhs=2)
    out = empty(x.shape, torch.complex128)
    L.laph_dirac_apply(context(), L.lattice(NS, NT, XI), dev(_links()), float("nan"), 1.0, dev(x), out, 2)
    assert not np.isfinite(host(out)).any()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["in", "z"])
@pytest.mark.parametrize("mode", list(MODES))
def test_operands_that_are_not_finite(mode, where, bad):
    if mode == "clovinv" and where == "z":
        return
    u = _links()
    K = WilsonClover(u, 0.02, 1.0, XI)
    vh, nr = NS ** 3 * NT // 2, 3
    cb, spin, col, r = 10, 1, 1, 1
    for p in (0, 1):
        x, z = synth.random_complex((vh, 12, nr), seed=4), synth.random_complex((vh, 12, nr), seed=5)
        clean_x, clean_z = x.copy(), z.copy()
        (x if where == "in" else z)[cb, 3 * spin + col, r] = bad
        (clean_x if where == "in" else clean_z)[cb, 3 * spin + col, r] = 0.0
        got = _hop(u, 0.02, 1.0, mode, p, x, z)
        hit = np.zeros((vh, 4, 3, nr), dtype=bool)
        if where == "in":
            f = np.zeros((vh, 12, nr), dtype=complex)
            f[cb, :, r] = 1.0
            full = from_eo(f, 1 - p, NS, NT)
            for mu, ax in enumerate((4, 3, 2, 1)):        # x, y, z, t of [nr][t][z][y][x]
                for s in (1, -1):
                    near = to_eo(np.ascontiguousarray(np.roll(full, s, ax)), p, NS, NT).reshape(vh, 4, 3, nr)[:, 0, 0] != 0
                    for a in (spin, PARTNER[mu][spin]):
                        hit[:, a][np.broadcast_to(near[:, None], (vh, 3, nr))] = True
            if mode != "apply":
                for h in (0, 2):
                    any_ = hit[:, h:h + 2].any((1, 2))
                    hit[:, h:h + 2] = np.broadcast_to(any_[:, None, None], (vh, 2, 3, nr))
        elif mode == "apply":
            hit[cb, 0:2, :, r] = True
        else:
            hit[cb, spin, col, r] = True
        hit = hit.reshape(vh, 12, nr)
        assert np.array_equal(~np.isfinite(got), hit)
        ref = reference(K, NS, NT, p, mode, clean_x, clean_z)
        assert np.abs(got[~hit] - ref[~hit]).max() <= 1e-13 * np.abs(ref).max()
