"""The source kernel at the edges of its tiles: slices of 8, 216, 512 and 1000 sites (a part of a tile, a
ragged last tile, one whole block, a block and a part), and more slices than a second grid dimension holds.
Every slice is checked, the ones that the time projector leaves out against exact zeros.

Tolerance: a sum of N_v terms +-v, +-iv in FP64, abs <= 1e-15 N_v max|v|."""
import numpy as np
import pytest
import torch

import synth
from oracle import noise as onoise
from oracle.dilution import full_projector_diag
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nv,dil,bs", [
    (2, 4, 5, ((1, 0), (1, 0), (1, 0)), [0, 37, 79]), (6, 6, 7, ((3, 2), (0, 0), (0, 0)), [1, 0]),
    (8, 2, 4, ((0, 0), (1, 0), (3, 2)), [0, 3, 7]), (10, 4, 6, ((2, 2), (3, 2), (2, 3)), [11, 4]),
    (2, 65540, 1, ((3, 4), (1, 0), (0, 0)), [2, 13]),
])
def test_sources_every_slice(ns, nt, nv, dil, bs):
    L = lib()
    v = synth.random_complex((nt, nv, ns ** 3, 3), seed=4)
    rhs = empty((len(bs), nt, ns ** 3, 4, 3), torch.complex128)
    rhs.fill_(7.0)
    L.laph_make_sources(context(), L.lattice(ns, nt, 1.0), dev(v), nv, 2, 5, L.dilution(*dil), bs, rhs, None)
    rho = onoise.z4_values(onoise.z4_codes(nt, nv, 2, 5))
    got = host(rhs)
    for i, b in enumerate(bs):
        p = full_projector_diag(dil, nt, nv, b).reshape(nt, 4, nv)
        y = np.einsum("tan,tnxc->txac", p * rho, v)[:, :, [2, 3, 0, 1]]
        assert np.abs(got[i] - y).max() <= 1e-15 * nv * np.abs(v).max()
        assert not got[i][~p.any((1, 2))].any()
