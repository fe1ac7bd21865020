"""The source kernel over its choices: blocks of 64, 128, 256 and 512 sites (by the number of slices that are not
zero), and lists of the projector's vectors that are empty, just full and longer than one list (192).

Tolerance: a sum of N_v terms +-v, +-iv in FP64, abs <= 1e-15 N_v max|v|."""
import numpy as np
import pytest
import torch

import synth
from oracle import noise as onoise
from oracle.dilution import full_projector_diag
from tests.gpu_util import context, dev, empty, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nv,dil,nb", [
    (6, 2, 9, ((0, 0), (0, 0), (3, 3)), 3),
    (10, 8, 5, ((0, 0), (1, 0), (0, 0)), 24), (10, 8, 5, ((0, 0), (1, 0), (0, 0)), 50),
    (10, 8, 5, ((0, 0), (1, 0), (0, 0)), 90), (10, 8, 5, ((0, 0), (1, 0), (0, 0)), 200),
    (6, 2, 191, ((0, 0), (0, 0), (0, 0)), 1), (6, 2, 192, ((0, 0), (0, 0), (0, 0)), 1),
    (6, 2, 193, ((0, 0), (1, 0), (1, 0)), 3), (8, 2, 400, ((3, 2), (0, 0), (3, 2)), 4), (6, 2, 600, ((0, 0), (1, 0), (2, 3)), 5),
])
def test_sources_shapes(ns, nt, nv, dil, nb):
    L = lib()
    v = dev(synth.random_complex((nt, nv, ns ** 3, 3), seed=4))
    total = len(full_projector_list(dil, nt, nv))
    bs = [(5 * i + 1) % total for i in range(nb)]
    rhs = empty((nb, nt, ns ** 3, 4, 3), torch.complex128)
    rhs.fill_(7.0)
    L.laph_make_sources(context(), L.lattice(ns, nt, 1.0), v, nv, 2, 5, L.dilution(*dil), bs, rhs, None)
    rho = onoise.z4_values(onoise.z4_codes(nt, nv, 2, 5))
    for i, b in enumerate(bs):
        p = full_projector_diag(dil, nt, nv, b).reshape(nt, 4, nv)
        y = torch.einsum("tan,tnxc->txac", dev(p * rho), v)[:, :, [2, 3, 0, 1]]
        assert float((rhs[i] - y).abs().max()) <= 1e-15 * nv * float(v.abs().max())


def full_projector_list(dil, nt, nv):
    counts = [{0: 1, 1: n, 2: j, 3: j}[k] for (k, j), n in zip(dil, (nt, 4, nv))]
    return range(counts[0] * counts[1] * counts[2])
