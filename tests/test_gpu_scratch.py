"""Calls on a device that is nearly full: buffers that only a faster path needs are left out, and the call is
not refused.  The FP64 hop of 256 right-hand sides on 16^3 x 16 wants 1.6 GB for its operand in fixed
point; with 1 GB left it takes the FP64 kernel.

Tolerance: the two kernels agree to 1e-13 of the largest entry, as each does with the oracle."""
import pytest
import torch

import synth
from tests.gpu_util import dev, lib, requires_gpu
from tests.test_gpu_dslash import MODES

pytestmark = [pytest.mark.gpu, requires_gpu]


def test_hop_on_a_nearly_full_device():
    L = lib()
    ns, nt, nr = 16, 16, 256
    u = dev(synth.random_su3_field(ns, nt, seed=7, eps=0.6))
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((ns ** 3 * nt // 2, 12, nr, 2), generator=g, dtype=torch.float64, device="cuda")
    x = torch.view_as_complex(x)
    ref, out = torch.empty_like(x), torch.empty_like(x)

    def hop(ctx, dst, n):
        L.laph_dslash_eo(ctx, L.lattice(ns, nt, 3.5), u, 0.02, 1.0, 0, MODES["clovinv"], L.PREC_FP64, x, None, dst, n)
        torch.cuda.synchronize()

    roomy, tight = L.Context(0), L.Context(0)
    hop(roomy, ref, nr)
    roomy.close()
    hop(tight, out, 1)                   # the operator's own arrays
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        hop(tight, out, nr)
    finally:
        del fill
        torch.cuda.empty_cache()
        tight.close()
    assert float((out - ref).abs().max()) <= 1e-13 * float(ref.abs().max())
