"""Operands of the FP64 hop at the lower end of the FP64 range, and zeros of both signs.

Tolerance: an output of entries of size 1e-300 keeps the 1e-14 of the largest entry that ordinary operands
keep, and is rounded to a multiple of the least subnormal, 48 times on its way in the reference
(48 * 5e-324); a field of zeros gives zeros."""
import numpy as np
import pytest
import torch

import synth
from oracle import gauge
from tests.gpu_util import context, dev, empty, host, lib, requires_gpu
from tests.test_gpu_dslash import MODES, reference
from oracle.dirac import WilsonClover

pytestmark = [pytest.mark.gpu, requires_gpu]

NS, NT, XI, M0 = 4, 6, 3.5, 0.02


def _hop(u, mode, p, x, z):
    L = lib()
    out = empty(x.shape, torch.complex128)
    L.laph_dslash_eo(context(), L.lattice(NS, NT, XI), dev(u), M0, 1.0, p, MODES[mode], L.PREC_FP64, dev(x),
                     None if mode == "clovinv" else dev(z), out, x.shape[2])
    return host(out)


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("power", [-940, -990, -1015])
def test_tiny_operands(mode, power):
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)
    K = WilsonClover(u, M0, 1.0, XI)
    x, z = (synth.random_complex((NS ** 3 * NT // 2, 12, 2), seed=s) for s in (4, 5))
    tiny = 2.0 ** power
    for p in (0, 1):
        ref = reference(K, NS, NT, p, mode, x, z)
        got = _hop(u, mode, p, tiny * x, tiny * z)
        up = 2.0 ** (-power // 2)                    # 2^-power itself may be out of range
        assert np.abs(got * up * 2.0 ** (-power - (-power // 2)) - ref).max() <= (
            1e-14 * np.abs(ref).max() + 200 * 2.0 ** (-1074 - power))


@pytest.mark.parametrize("mode", list(MODES))
def test_negative_zeros(mode):
    u = gauge.stout(synth.random_su3_field(NS, NT, seed=7), 0.1, 2, spatial_only=False)
    x = np.zeros((NS ** 3 * NT // 2, 12, 3), dtype=complex)
    x[..., 0] = complex(-0.0, -0.0)
    x[::2, :, 1] = complex(-0.0, -0.0)
    for p in (0, 1):
        assert np.all(_hop(u, mode, p, x, x) == 0.0)


def test_one_colour_stays_one_colour():
    """On unit links a field of one colour, with zeros of either sign in the others, stays of one colour."""
    u = np.broadcast_to(np.eye(3, dtype=complex), (NT, NS, NS, NS, 4, 3, 3)).copy()
    x = np.zeros((NS ** 3 * NT // 2, 4, 3, 2), dtype=complex)
    x[:, :, 1] = complex(-0.0, -0.0)
    x[:, :, 0] = synth.random_complex((NS ** 3 * NT // 2, 4, 2), seed=4)
    x = x.reshape(-1, 12, 2)
    for p in (0, 1):
        got = _hop(u, "apply", p, x, x).reshape(-1, 4, 3, 2)
        assert np.abs(got[:, :, 0]).max() > 0.1 and np.all(got[:, :, 1:] == 0.0)
