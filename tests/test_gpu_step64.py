"""The double-precision whole-step kernel of 8^3 and 16^3 grids against the oracle
where its paths differ: one and several passes over the z groups, groups whose
minimum image jumps inside the cell or not at all, other stencil widths, no
projectors, a field that changes every step (fresh projections per step), and
runs just below and at the number of orbitals from which it is taken.  Bars: the
double-precision ones of the other parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu

_SIX = np.array([[0.05 * i + 0.1, 0.13 * i, 0.11 * i + 0.02] for i in range(6)])
_EIGHT = np.array([[0.1 * i, 0.37 * i % 1.0, (0.07 + 0.121 * i) % 1.0] for i in range(8)])


def _cell(n, bands, atoms=None, edge=6.0, **kw):
    c = W.cell_tiny(atoms="pair", n=(n, n, n), a=(edge, edge * 1.1, edge * 0.95), n_bands=bands)
    if atoms is not None:
        c = c.replace(atom_frac=np.asarray(atoms, dtype=np.float64))
    return c.replace(**kw) if kw else c


PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
CASES = [
    # (cell, subgrid, field, stencil half-width, steps)
    (_cell(8, 4), (2, 1, 1), W.Kick(k0=0.01), 4, 3),                       # 8 orbitals: the first that take it
    (_cell(8, 7), (1, 1, 1), W.Kick(k0=0.01), 4, 2),                       # 7 orbitals: the sequence of launches
    (_cell(8, 3, _SIX), (2, 2, 1), PULSE, 4, 3),                           # 6 z groups, two passes
    (_cell(8, 2, _EIGHT, proj_half=2.5), (2, 2, 1), W.Kick(k0=0.01), 6, 2),  # 8 groups, narrow boxes, wide stencil
    (_cell(16, 3, _SIX, 10.0), (3, 1, 1), W.Kick(k0=0.01), 3, 2),
    (_cell(16, 2, [[0.0, 0.1, 0.0], [0.3, 0.2, 0.5], [0.6, 0.7, 0.5]], 10.0), (1, 2, 2), PULSE, 4, 2),
    (W.cell_tiny(atoms="none", n=(16, 16, 16), a=(10.0, 9.0, 11.0), n_bands=4), (2, 1, 1), PULSE, 1, 2),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("propagator", ["taylor4", "etrs"])
def test_step64_vs_oracle(case, propagator):
    cell, mp, field, nd, steps = CASES[case]
    from oracle import dynamics, kpoints
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, steps, field, seed=80 + case)
    P, g = gpu_run(cell, [s], precision="fp64", fd_nd=nd, propagator=propagator)
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], steps, dynamics.field_samples(field, s["dt"], steps),
                           ops=dynamics.Operators(cell, nd), keep_state=False, propagator=propagator)
    compare(g[0], o, FP64_J_TOL, FP64_RHO_TOL)
