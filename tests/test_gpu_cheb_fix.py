"""Eigenpairs through the fixed-point Chebyshev chain (cheb_fix.cu) where it can go wrong: rough links at
full range, ns = 2 (both neighbours of a direction are one site), slices that are no multiple of a block, and
links that are not bounded by one, which take the FP64 kernel.

Tolerance: the residuals converge to 12e-13 (12 x the default 1e-13); an eigenvalue is within its vector's
residual squared over the gap plus FP64 rounding of ||-Delta|| <= 14, so abs <= 1e-12 without degeneracy, and the
vectors satisfy ||-Delta y - mu y|| <= 2e-12 with the matrix formed here."""
import numpy as np
import pytest
import torch

import synth
from oracle.laplacian import slice_matrix
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nv,eps,scale", [(2, 4, 3, 2.0, 1.0), (4, 2, 5, 2.0, 1.0), (6, 4, 9, 0.6, 1.0),
                                                (10, 2, 7, 0.6, 1.0), (4, 2, 5, 0.6, 1.2)])
def test_eigenpairs(ns, nt, nv, eps, scale):
    L = lib()
    u = scale * synth.random_su3_field(ns, nt, seed=11, eps=eps)
    evals, evecs = empty((nt, nv), torch.float64), empty((nt, nv, ns ** 3, 3), torch.complex128)
    L.laph_eigvecs(context(), L.lattice(ns, nt, 1.0), dev(u), nv, evals, evecs)
    mu, v = host(evals), host(evecs).reshape(nt, nv, -1)
    for t in range(nt):
        m = slice_matrix(u, t)
        ref = np.linalg.eigvalsh(m.toarray() if hasattr(m, "toarray") else m)[:nv]
        assert np.abs(mu[t] - ref).max() <= 1e-12
        r = (m @ v[t].T).T - mu[t][:, None] * v[t]
        assert np.linalg.norm(r, axis=1).max() <= 2e-12
