"""Phase tables formed from factors (single precision): atoms outside the cell's edges,
on its faces and off the grid, boxes wider and narrower than half the cell, axes of
unequal length, fields along one axis and along all three, against the oracle at the
bars of the other single-precision parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu

ALONG_Z = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.0, 0.0, 1.0))
ALONG_ALL = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, -0.5, 0.8))
_OUT = np.array([[-0.3, 1.4, 0.0], [0.55, -1.25, 2.5]])
CASES = [
    ((16, 16, 16), _OUT, 8.0, ALONG_Z),
    ((16, 16, 16), np.array([[0.0, 0.5, 0.97], [0.999, 0.03125, 0.5]]), 3.0, ALONG_ALL),
    ((10, 13, 17), _OUT, 9.0, ALONG_ALL),
    ((32, 16, 16), np.array([[0.11, 0.51, 0.49], [-0.02, 0.77, 1.0]]), 16.0, ALONG_Z),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_factored_phases_vs_oracle(case):
    from oracle import dynamics, kpoints
    n, atoms, half, field = CASES[case]
    cell = W.cell_tiny(atoms="pair", n=n, a=tuple(0.72 * v for v in n), n_bands=4).replace(atom_frac=atoms,
                                                                                          proj_half=half)
    s = random_subsim(cell, (2, 1, 2), (0.25, 0.5, 0.125), 0.04, 3, field, seed=310 + case)
    P, g = gpu_run(cell, [s], precision="fp32")
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 3, dynamics.field_samples(field, s["dt"], 3),
                           ops=dynamics.Operators(cell), keep_state=False)
    compare(g[0], o, FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
