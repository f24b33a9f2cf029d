"""The whole-step kernel of 32^3 cells (a cluster per band) against the oracle: the
64-atom cell under a pulse and with the time-reversal-symmetric step, few atoms off
the grid points (boxes that wrap, empty rows, one and several classes per axis), narrow
boxes, atoms in more classes than it takes (the slab kernels), and a restart
mid-run bit for bit.  Bars: the single-precision ones of the other parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import (FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, compare, gpu_run, oracle_run, random_subsim)

pytestmark = pytest.mark.gpu

PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
KICK = W.Kick(k0=0.01, direction=(0.0, 0.6, 0.8))
_MIXED = np.array([[0.1, 0.2, 0.3], [0.1, 0.7, 0.3], [0.55, 0.2, 0.9], [0.97, 0.03, 0.9], [0.55, 0.7, 0.01]])
_NINE = np.array([[0.1 * i + 0.03, 0.5, 0.25] for i in range(9)])


def _cell(bands, atoms, **kw):
    c = W.cell_tiny(atoms="pair", n=(32, 32, 32), a=(20.5, 20.0, 21.0), n_bands=bands)
    return c.replace(atom_frac=np.asarray(atoms, dtype=np.float64), **kw)


CASES = [
    (lambda: W.cell_b(n_bands=2), (1, 1, 2), PULSE, "taylor4"),
    (lambda: W.cell_b(n_bands=2), (1, 1, 1), KICK, "etrs"),
    (lambda: _cell(3, [[0.1, 0.2, 0.3]]), (2, 1, 1), KICK, "taylor4"),
    (lambda: _cell(3, _MIXED, proj_half=6.5), (1, 2, 1), PULSE, "taylor4"),
    (lambda: _cell(2, _NINE, proj_half=7.0), (1, 1, 1), KICK, "taylor4"),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_step32c_vs_oracle(case):
    make, mp, field, propagator = CASES[case]
    cell = make()
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.06, 2, field, seed=260 + case)
    P, g = gpu_run(cell, [s], precision="fp32", propagator=propagator)
    P.close()
    compare(g[0], oracle_run(cell, s, propagator=propagator), FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)


@pytest.mark.parametrize("field", [KICK, PULSE])
def test_step32c_restart_bitwise(field):
    cell = W.cell_b(n_bands=3)
    s = random_subsim(cell, (1, 2, 1), (0.25, 0.5, 0.125), 0.06, 4, field, seed=270)
    P1, _ = gpu_run(cell, [s], precision="fp32", steps=2)
    mid, step = P1.get_state(0)
    P1.propagate(2)
    P2, _ = gpu_run(cell, [s], precision="fp32", steps=0)
    P2.load_state(0, mid, step)
    P2.propagate(2)
    np.testing.assert_array_equal(P1.get_state(0)[0], P2.get_state(0)[0])
    np.testing.assert_array_equal(P1.density(0), P2.density(0))
    np.testing.assert_array_equal(P1.current(0)[0][3:], P2.current(0)[0][3:])
    P1.close()
    P2.close()
