"""The partial sums of a large exact-slice GEMM: the batch goes in passes whose partial sums stay below
512 MB, whatever the number of tiles (here 7936 of 128 KB, 1 GB), with the same results.

Tolerance: 8 K 2^-52.5 max|a| max|b|, as for every exact-slice GEMM."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import dev, empty, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def test_overlaps_of_many_tiles_in_bounded_memory():
    L = lib()
    ns, nt, nv = 4, 128, 65
    mom = [(i % 5 - 2, i // 5 - 2, i % 3) for i in range(30)]     # 31 column tiles, 2 row tiles, 128 slices
    v = dev(synth.random_complex((nt, nv, ns ** 3, 3), seed=1))
    out = empty((len(mom), nt, nv, nv), torch.complex128)
    ctx = L.Context(0)
    small = empty((1, nt, nv, nv), torch.complex128)
    L.laph_mom_overlaps(ctx, L.lattice(ns, nt, 3.5), v, nv, mom[:1], small)   # the small buffers
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    L.laph_mom_overlaps(ctx, L.lattice(ns, nt, 3.5), v, nv, mom, out)
    torch.cuda.synchronize()
    grown = before - torch.cuda.mem_get_info()[0]
    assert grown <= (512 << 20) + (64 << 20)
    i = torch.arange(ns, device="cuda", dtype=torch.float64)
    w = v.reshape(nt, nv, -1)
    bound = 8 * 3 * ns ** 3 * 2.0 ** -52.5 * float(w.abs().max()) ** 2
    for k, p in enumerate(mom):
        ph = torch.exp(-2j * np.pi / ns * (p[0] * i + p[1] * i[:, None] + p[2] * i[:, None, None])).reshape(-1)
        ref = torch.einsum("tnk,tmk->tnm", w.conj(), w * ph.repeat_interleave(3))
        assert float((out[k] - ref).abs().max()) <= bound
