"""The one-kernel inner solver (bicg_small.cu) at the edges of its shapes: one CTA to clusters of 16,
128, 256 and 512 threads, lattices that leave lanes and whole CTAs without sites, a zero and a
non-finite right-hand side beside ordinary ones.

The solve must meet its tolerance by the oracle's own K (1e-10 on the true residual, with 5 % for the
oracle's rounding) without the CG fallback, and take about as many iterations as the streamed solver
does for the same sources (a block above the one-kernel limit): within a third."""
import numpy as np
import pytest

import synth
from oracle import gauge
from oracle.dirac import WilsonClover
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _solve(L, ns, nt, u, m0, b):
    sol = empty(b.shape, dev(b).dtype)
    reps = L.dirac_solve_batch(context(), L.lattice(ns, nt, 3.5), dev(u), m0, 1.0, dev(b), sol, len(b),
                               L.solver_params(rhs_block=len(b)), allow_not_converged=True)
    return host(sol), reps


@pytest.mark.parametrize("ns,nt,nrhs", [(2, 2, 3), (2, 6, 1), (4, 4, 5), (4, 8, 2), (6, 4, 3), (6, 6, 2), (6, 10, 1), (8, 8, 2)])
def test_small_solve_shapes(ns, nt, nrhs):
    L = lib()
    m0 = 0.05
    u = gauge.stout(synth.random_su3_field(ns, nt, seed=81), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, m0, 1.0, 3.5)
    b = synth.random_spinor(ns, nt, seed=82, nrhs=nrhs)
    x, reps = _solve(L, ns, nt, u, m0, b)
    for i in range(nrhs):
        assert reps[i].status == 0 and reps[i].fallback_used == 0
        assert np.linalg.norm(b[i] - K.apply(x[i])) <= 1.05e-10 * np.linalg.norm(b[i])
    many = np.repeat(b, 70 // nrhs + 1, axis=0)      # above every limit: the streamed solver
    _, ref = _solve(L, ns, nt, u, m0, many)
    for i in range(nrhs):
        it = ref[i * (70 // nrhs + 1)].iters
        assert abs(reps[i].iters - it) <= max(6, it // 3), (reps[i].iters, it)


def test_small_solve_zero_and_non_finite_sources():
    L = lib()
    ns, nt, m0 = 4, 6, 0.05
    u = gauge.stout(synth.random_su3_field(ns, nt, seed=83), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, m0, 1.0, 3.5)
    b = synth.random_spinor(ns, nt, seed=84, nrhs=4)
    b[1] = 0.0
    b[2, 3, 1, 0, 2, 1, 1] = np.nan
    x, reps = _solve(L, ns, nt, u, m0, b)
    assert np.all(x[1] == 0.0) and reps[1].status == 0
    assert reps[2].status == L.LAPH_ERR_NOT_CONVERGED and np.isnan(reps[2].true_resid)
    for i in (0, 3):
        assert reps[i].status == 0
        assert np.linalg.norm(b[i] - K.apply(x[i])) <= 1.05e-10 * np.linalg.norm(b[i])
