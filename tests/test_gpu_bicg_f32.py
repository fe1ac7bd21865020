"""The streamed inner solver (bicg_f32.cu and the stencil's fused products) over its right-hand-side
counts: packed and unpacked updates (even and odd nr), the generic products (nr not 32, 64 or 128), and
the stencil's with one, two and four groups of 32 right-hand sides, some of which are zero.

Every solve must meet 1e-10 on the oracle's own K (5 % for its rounding) without the CG fallback."""
import numpy as np
import pytest

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nrhs", [(8, 10, 1), (6, 10, 33), (6, 8, 32), (4, 8, 65), (4, 8, 96), (6, 6, 64), (4, 8, 128)])
def test_streamed_solve_right_hand_sides(ns, nt, nrhs):
    L = lib()
    m0 = 0.05
    u = gauge.stout(synth.random_su3_field(ns, nt, seed=91), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, m0, 1.0, 3.5)
    b = synth.random_spinor(ns, nt, seed=92, nrhs=nrhs)
    zero = list(range(7, nrhs, 13))
    b[zero] = 0.0
    sol = empty(b.shape, dev(b).dtype)
    reps = L.dirac_solve_batch(context(), L.lattice(ns, nt, 3.5), dev(u), m0, 1.0, dev(b), sol, nrhs,
                               L.solver_params(rhs_block=nrhs))
    x = host(sol)
    for i in range(nrhs):
        assert reps[i].status == 0 and reps[i].fallback_used == 0
        if i in zero:
            assert np.all(x[i] == 0.0)
        else:
            assert np.linalg.norm(b[i] - K.apply(x[i])) <= 1.05e-10 * np.linalg.norm(b[i])
