"""The fixed-point FP64 hop (dslash_fix.cu) where its number format matters: operands spread over many
orders of magnitude between sites, very small and very large fields, zero spinors, NaN and infinities
(the FP64 kernel takes over), and an anisotropy whose hop weights are not below one (likewise).

Tolerance: at a site every error scales with the largest entry M of the neighbour spinors and of the
site term's operand: an entry is cut at 2^-58 and a sum rounded at 2^-57 of up to 2 M, 48 of them meet in
an output of row norm |A^-1| (or |A|) <= 12 max|entry|; 1e-14 * 12 max|entry| M leaves a factor of ten."""
import numpy as np
import pytest
import torch

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import MODES, from_eo, parity_sites, reference, to_eo

pytestmark = [pytest.mark.gpu, requires_gpu]

NS, NT, M0, CSW = 4, 6, 0.02, 1.0


def _hop(xi, u, mode, p, x, z):
    L = lib()
    out = empty(x.shape, torch.complex128)
    L.laph_dslash_eo(context(), L.lattice(NS, NT, xi), dev(u), M0, CSW, p, MODES[mode], L.PREC_FP64, dev(x),
                     None if mode == "clovinv" else dev(z), out, x.shape[2])
    return host(out)


def _neighbour_max(x, p):
    """max |entry| over the eight neighbour spinors of every site of parity p, [cb][1][nr]."""
    m = np.abs(from_eo(x, 1 - p, NS, NT)).max((-1, -2))                     # [nr][t][z][y][x]
    n = np.max([np.roll(m, s, ax) for ax in (1, 2, 3, 4) for s in (1, -1)], axis=0)
    full = np.broadcast_to(n[..., None, None], n.shape + (4, 3))
    return to_eo(np.ascontiguousarray(full), p, NS, NT)


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("kind,xi", [("spread", 3.5), ("tiny", 3.5), ("huge", 3.5), ("sparse", 3.5), ("spread", 0.4)])
def test_fixed_point_hop_ranges(mode, kind, xi):
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, M0, CSW, xi)
    vh, nr = NS ** 3 * NT // 2, 5
    rng = np.random.default_rng(3)
    x, z = synth.random_complex((vh, 12, nr), seed=4), synth.random_complex((vh, 12, nr), seed=5)
    if kind == "spread":
        x *= 10.0 ** rng.uniform(-25, 5, (vh, 1, nr))
        z *= 10.0 ** rng.uniform(-25, 5, (vh, 1, nr))
    elif kind == "tiny":
        x, z = 1e-250 * x, 1e-250 * z
    elif kind == "huge":
        x, z = 1e250 * x, 1e250 * z
    else:
        x[rng.random((vh, 12, nr)) < 0.9] = 0.0
        z[rng.random((vh, 1, nr)).repeat(12, 1) < 0.5] = 0.0
    for p in (0, 1):
        got, ref = _hop(xi, u, mode, p, x, z), reference(K, NS, NT, p, mode, x, z)
        a = K.a.reshape(-1, 12, 12)[parity_sites(NS, NT, p)]
        top = np.abs(a).max() if mode == "apply" else np.abs(np.linalg.inv(a)).max()
        M = _neighbour_max(x, p) * max(1.0, 1.0 / xi)
        if mode != "clovinv":
            M = np.maximum(M, np.abs(z).max(1, keepdims=True))
        assert np.all(np.abs(got - ref) <= 1e-14 * 12 * max(top, 1.0) * M)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["in", "z"])
def test_fixed_point_hop_non_finite(bad, where):
    """A non-finite entry reaches exactly the outputs it reaches in the oracle's arithmetic."""
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, M0, CSW, 3.5)
    vh, nr = NS ** 3 * NT // 2, 3
    x, z = synth.random_complex((vh, 12, nr), seed=4), synth.random_complex((vh, 12, nr), seed=5)
    (x if where == "in" else z)[10, 4, 1] = bad
    got = _hop(3.5, u, "apply", 0, x, z)
    hit = np.zeros((vh, 12, nr), dtype=bool)
    if where == "in":
        f = np.zeros((vh, 12, nr))
        f[10, :, 1] = 1.0
        hit[:] = (_neighbour_max(f.astype(complex), 0) > 0.5)
    else:
        hit[10, :, 1] = True
    assert np.isfinite(got[~hit]).all()
    assert not np.isfinite(got[hit]).all()
    clean_x, clean_z = x.copy(), z.copy()
    (clean_x if where == "in" else clean_z)[10, 4, 1] = 0.0
    ref = reference(K, NS, NT, 0, "apply", clean_x, clean_z)
    assert np.abs(got[~hit] - ref[~hit]).max() <= 1e-13 * np.abs(ref).max()
