"""The clover blocks and their inverses (clover.cu) against the oracle's site matrices: rough SU(3)
links (the fixed-point products at full range), links that are not bounded by one (the FP64 path), a
mass that cancels the diagonal, so that A has small L D L^dag pivots (the pivoted inverse), and ns = 2,
where both neighbours in a direction are the same site.

laph_dslash_eo in FP64: apply mode on a zero hop operand gives A z, clovinv gives A^{-1} D x.
Tolerance: A is 64-bit accurate, rel <= 1e-14; an inverse loses cond(A): rel <= 1e-14 cond(A) + 1e-13."""
import numpy as np
import pytest
import torch

import synth
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import CSW, MODES, XI, parity_sites, reference

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,eps,scale,m0", [
    (4, 6, 2.0, 1.0, -0.05), (2, 4, 2.0, 1.0, 0.3), (6, 4, 0.4, 1.0, -0.05),
    (4, 4, 1.0, 1.3, 0.1), (4, 4, 2.0, 1.0, -(1.0 + 3.0 / XI)),
])
def test_clover_blocks(ns, nt, eps, scale, m0):
    L = lib()
    u = scale * synth.random_su3_field(ns, nt, seed=5, eps=eps)
    K = WilsonClover(u, m0, CSW, XI)
    vh, nr = ns ** 3 * nt // 2, 3
    x = synth.random_complex((vh, 12, nr), seed=6)
    zero = np.zeros_like(x)
    for p in (0, 1):
        a = K.a.reshape(-1, 12, 12)[parity_sites(ns, nt, p)]
        out = empty(x.shape, torch.complex128)
        L.laph_dslash_eo(context(), L.lattice(ns, nt, XI), dev(u), m0, CSW, p, MODES["apply"], L.PREC_FP64, dev(zero),
                         dev(x), out, nr)
        ref = np.einsum("sij,sjn->sin", a, x)
        assert np.abs(host(out) - ref).max() <= 1e-14 * np.abs(a).sum(2).max() * np.abs(x).max()
        L.laph_dslash_eo(context(), L.lattice(ns, nt, XI), dev(u), m0, CSW, p, MODES["clovinv"], L.PREC_FP64, dev(x),
                         None, out, nr)
        ref = reference(K, ns, nt, p, "clovinv", x, zero)
        cond = np.linalg.cond(a).max()
        assert np.linalg.norm(host(out) - ref) <= (1e-14 * cond + 1e-13) * np.linalg.norm(ref)
