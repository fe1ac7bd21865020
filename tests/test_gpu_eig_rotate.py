"""The restart GEMM of the eigensolver on the tensor cores: column counts on both sides of a tile of 64, Krylov
dimensions that are no multiple of the 16 of a sub-chunk, row counts below and above a tile.

Tolerance: as the eigensolver's contract, residuals <= 12e-13 (2e-12 with the matrix formed here), and
orthonormal vectors to 1e-11 (restarts keep the basis orthonormal to its residuals)."""
import numpy as np
import pytest
import torch

import synth
from oracle.laplacian import slice_matrix
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nv,m", [(2, 2, 15), (4, 10, 33), (6, 40, 101), (6, 62, 139), (8, 6, 31)])
def test_restart_gemm(ns, nv, m):
    L = lib()
    nt = 2
    u = synth.random_su3_field(ns, nt, seed=3, eps=1.2)
    evals, evecs = empty((nt, nv), torch.float64), empty((nt, nv, ns ** 3, 3), torch.complex128)
    L.laph_eigvecs(context(), L.lattice(ns, nt, 1.0), dev(u), nv, evals, evecs, L.EigParams(krylov_dim=m, seed=12345))
    mu, v = host(evals), host(evecs).reshape(nt, nv, -1)
    for t in range(nt):
        a = slice_matrix(u, t)
        r = (a @ v[t].T).T - mu[t][:, None] * v[t]
        assert np.linalg.norm(r, axis=1).max() <= 2e-12
        assert np.abs(v[t].conj() @ v[t].T - np.eye(nv)).max() <= 1e-11
