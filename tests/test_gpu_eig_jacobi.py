"""The cluster Jacobi of the eigensolver where its split can go wrong: few slices (eight blocks a slice), enough for
four, two and one block, odd and even Krylov dimensions, and blocks that own no row of the eigenvector matrix.

Tolerance: residuals as the eigensolver's contract (12e-13; 2e-12 with the matrix formed here), eigenvalues
abs <= 1e-12 against the dense solver."""
import numpy as np
import pytest
import torch

import synth
from oracle.laplacian import slice_matrix
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nv,m", [(2, 2, 1, 14), (4, 2, 6, 39), (4, 20, 6, 42), (4, 40, 5, 37), (4, 78, 4, 36),
                                        (2, 154, 2, 17), (6, 2, 24, 130)])
def test_krylov_dims(ns, nt, nv, m):
    L = lib()
    u = synth.random_su3_field(ns, nt, seed=8, eps=1.2)
    evals, evecs = empty((nt, nv), torch.float64), empty((nt, nv, ns ** 3, 3), torch.complex128)
    L.laph_eigvecs(context(), L.lattice(ns, nt, 1.0), dev(u), nv, evals, evecs, L.EigParams(krylov_dim=m, seed=12345))
    mu, v = host(evals), host(evecs).reshape(nt, nv, -1)
    for t in range(0, nt, max(1, nt // 8)):
        a = slice_matrix(u, t)
        r = (a @ v[t].T).T - mu[t][:, None] * v[t]
        assert np.linalg.norm(r, axis=1).max() <= 2e-12
        assert np.abs(mu[t] - np.linalg.eigvalsh(a.toarray())[:nv]).max() <= 1e-12
