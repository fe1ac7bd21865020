"""The streamed inner solver where its right-hand sides stop one after another: sources that converge at
different iterations (b, K b, K K b and zeros) in one block, polled after every iteration and rarely.  What a right-hand side gets does not depend on when
the others stop, so solutions and iteration counts are the same bits from call to call and for both
polling intervals; every solve meets 1e-10 on the oracle's own K (5 % for its rounding)."""
import numpy as np
import pytest

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ns,nt,nrhs", [(4, 8, 96), (6, 8, 33)])
def test_right_hand_sides_that_stop_at_different_iterations(ns, nt, nrhs):
    L = lib()
    m0 = 0.05
    u = gauge.stout(synth.random_su3_field(ns, nt, seed=93), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, m0, 1.0, 3.5)
    b = synth.random_spinor(ns, nt, seed=94, nrhs=nrhs)
    for i in range(nrhs):
        if i % 5 == 1:
            b[i] = K.apply(b[i])                  # rough solutions: fewer iterations than rough sources
        elif i % 5 == 2:
            b[i] = K.apply(K.apply(b[i]))
        elif i % 5 == 3:
            b[i] = 0.0
    out = []
    for every in (1, 1, 50):
        sol = empty(b.shape, dev(b).dtype)
        reps = L.dirac_solve_batch(context(), L.lattice(ns, nt, 3.5), dev(u), m0, 1.0, dev(b), sol, nrhs,
                                   L.solver_params(rhs_block=nrhs, check_every=every))
        out.append((host(sol), [r.iters for r in reps]))
        assert all(r.status == 0 and r.fallback_used == 0 for r in reps)
    assert len(set(out[0][1])) > 3
    for x, iters in out[1:]:
        assert iters == out[0][1] and np.array_equal(x, out[0][0])
    for i in range(nrhs):
        assert np.linalg.norm(b[i] - K.apply(out[0][0][i])) <= 1.05e-10 * np.linalg.norm(b[i])
