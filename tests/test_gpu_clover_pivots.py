"""The inverse of clover blocks whose diagonal is far smaller than their other entries: a constant
colour-diagonal field in the (x, z) plane and a mass that cancels the hop weights up to d = 1e-9, so that
A = d + s2 x G with |G| up to 0.2 is indefinite and well conditioned, while an elimination along the diagonal
starts with the pivot d.

Tolerance: as for every inverse, rel <= 1e-14 cond(A) + 1e-13 (cond(A) is about 2)."""
import numpy as np
import pytest
import torch

import synth
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import MODES, parity_sites, reference

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("d", [1e-9, 1e-4, 0.03])
def test_inverse_of_indefinite_blocks(d, sign):
    L = lib()
    ns, nt, xi = 6, 4, 4.0
    m0 = -1.75 + sign * d
    u = np.broadcast_to(np.eye(3, dtype=complex), (nt, ns, ns, ns, 4, 3, 3)).copy()
    for z in range(ns):   # a sixth of a turn per plaquette: periodic, and no colour without a field
        u[:, z, :, :, 0] = np.diag(np.exp(2j * np.pi / ns * z * np.array([1, 1, -2])))
    K = WilsonClover(u, m0, 1.0, xi)
    vh, nr = ns ** 3 * nt // 2, 3
    x = synth.random_complex((vh, 12, nr), seed=6)
    for p in (0, 1):
        a = K.a.reshape(-1, 12, 12)[parity_sites(ns, nt, p)]
        cond = np.linalg.cond(a).max()
        assert cond < 10
        out = empty(x.shape, torch.complex128)
        L.laph_dslash_eo(context(), L.lattice(ns, nt, xi), dev(u), m0, 1.0, p, MODES["clovinv"], L.PREC_FP64, dev(x), None,
                         out, nr)
        ref = reference(K, ns, nt, p, "clovinv", x, np.zeros_like(x))
        assert np.linalg.norm(host(out) - ref) <= (1e-14 * cond + 1e-13) * np.linalg.norm(ref)
