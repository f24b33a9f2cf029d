"""Small grids in double precision with more orbitals than take clusters of CTAs: a band per CTA, for
the cases that other tests run with few orbitals (odd axes, up to 8 z groups, narrow boxes, no
atoms, other stencil widths, both propagators), against the oracle, and a restart mid-run bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu

_EIGHT = np.array([[0.1 * i, 0.37 * i % 1.0, (0.07 + 0.121 * i) % 1.0] for i in range(8)])
PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
KICK = W.Kick(k0=0.01, direction=(0.0, 0.6, 0.8))


def _cell(n, bands, atoms="offgrid", **kw):
    c = W.cell_tiny(atoms=atoms if isinstance(atoms, str) else "pair", n=n, a=tuple(0.72 * v for v in n), n_bands=bands)
    return c.replace(**kw) if isinstance(atoms, str) else c.replace(atom_frac=atoms, **kw)


CASES = [
    (lambda: _cell((5, 6, 7), 4), (5, 4, 1), KICK, 4),
    (lambda: _cell((9, 17, 10), 4, _EIGHT, proj_half=3.5), (1, 20, 1), KICK, 4),
    (lambda: _cell((8, 8, 8), 4, _EIGHT), (5, 2, 2), PULSE, 4),
    (lambda: _cell((8, 8, 8), 3, "none"), (3, 3, 3), KICK, 2),
    (lambda: _cell((7, 13, 11), 2, "pair"), (13, 3, 1), PULSE, 6),
    (lambda: _cell((7, 3, 6), 4, "pair"), (5, 4, 1), PULSE, 1),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("propagator", ["taylor4", "etrs"])
def test_band_per_cta_vs_oracle(case, propagator):
    from oracle import dynamics, kpoints
    make, mp, field, nd = CASES[case]
    cell = make()
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 2, field, seed=400 + case)
    P, g = gpu_run(cell, [s], precision="fp64", fd_nd=nd, propagator=propagator)
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 2, dynamics.field_samples(field, s["dt"], 2),
                           ops=dynamics.Operators(cell, nd), keep_state=False, propagator=propagator)
    compare(g[0], o, FP64_J_TOL, FP64_RHO_TOL)


@pytest.mark.parametrize("case", [0, 2, 4])
def test_band_per_cta_restart_bitwise(case):
    make, mp, field, nd = CASES[case]
    cell = make()
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 4, field, seed=410 + case)
    P1, _ = gpu_run(cell, [s], precision="fp64", fd_nd=nd, steps=2)
    mid, step = P1.get_state(0)
    P1.propagate(2)
    P2, _ = gpu_run(cell, [s], precision="fp64", fd_nd=nd, steps=0)
    P2.load_state(0, mid, step)
    P2.propagate(2)
    np.testing.assert_array_equal(P1.get_state(0)[0], P2.get_state(0)[0])
    np.testing.assert_array_equal(P1.density(0), P2.density(0))
    np.testing.assert_array_equal(P1.current(0)[0][3:], P2.current(0)[0][3:])
    P1.close()
    P2.close()
