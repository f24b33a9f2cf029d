"""The whole-step kernel of small grids against the oracle: the smallest and odd
axes, one point above the stencil's width, 8^3 (its Fourier form) with and without
atoms, up to 8 z groups with and without a jump of the minimum image, narrow
boxes, other stencil widths, a field that changes every step, both propagators,
and a grid too large for it; and a restart mid-run bit for bit.  Bars: those of the other parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import (FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run,
                        random_subsim)

pytestmark = pytest.mark.gpu

_EIGHT = np.array([[0.1 * i, 0.37 * i % 1.0, (0.07 + 0.121 * i) % 1.0] for i in range(8)])
PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
KICK = W.Kick(k0=0.01, direction=(0.0, 0.6, 0.8))


def _cell(n, bands, atoms="offgrid", **kw):
    if isinstance(atoms, str):
        c = W.cell_tiny(atoms=atoms, n=n, a=tuple(0.72 * v for v in n), n_bands=bands)
    else:
        c = W.cell_tiny(atoms="pair", n=n, a=tuple(0.72 * v for v in n), n_bands=bands).replace(atom_frac=atoms)
    return c.replace(**kw) if kw else c


CASES = [
    (_cell((5, 6, 7), 4), (2, 1, 1), KICK, 4),
    (_cell((18, 8, 9), 3), (3, 1, 1), PULSE, 4),
    (_cell((9, 17, 10), 4, _EIGHT, proj_half=3.5), (1, 2, 1), KICK, 4),
    (_cell((8, 8, 8), 4, _EIGHT), (2, 1, 2), PULSE, 4),
    (_cell((8, 8, 8), 3, "none"), (2, 2, 1), KICK, 2),
    (_cell((7, 13, 11), 2, "pair"), (2, 2, 1), PULSE, 6),
    (_cell((20, 20, 21), 2, "one"), (2, 2, 1), KICK, 4),     # the sequence of launches in double precision
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("propagator", ["taylor4", "etrs"])
def test_step_any_vs_oracle(case, precision, propagator):
    from oracle import dynamics, kpoints
    cell, mp, field, nd = CASES[case]
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 3, field, seed=200 + case)
    P, g = gpu_run(cell, [s], precision=precision, fd_nd=nd, propagator=propagator)
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 3, dynamics.field_samples(field, s["dt"], 3),
                           ops=dynamics.Operators(cell, nd), keep_state=False, propagator=propagator)
    if precision == "fp64":
        compare(g[0], o, FP64_J_TOL, FP64_RHO_TOL)
    else:
        compare(g[0], o, FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)


@pytest.mark.parametrize("case", [0, 1, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_step_any_restart_bitwise(case, precision):
    cell, mp, field, nd = CASES[case]
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 4, field, seed=230 + case)
    P1, _ = gpu_run(cell, [s], precision=precision, fd_nd=nd, steps=2)
    mid, step = P1.get_state(0)
    P1.propagate(2)
    P2, _ = gpu_run(cell, [s], precision=precision, fd_nd=nd, steps=0)
    P2.load_state(0, mid, step)
    P2.propagate(2)
    np.testing.assert_array_equal(P1.get_state(0)[0], P2.get_state(0)[0])
    np.testing.assert_array_equal(P1.density(0), P2.density(0))
    np.testing.assert_array_equal(P1.current(0)[0][3:], P2.current(0)[0][3:])
    P1.close()
    P2.close()


@pytest.mark.parametrize("n,bands", [((13, 15, 12), 3), ((18, 18, 16), 2), ((16, 16, 8), 3)])
def test_step_any_wide_vs_oracle(n, bands):
    """Single-precision cells of which fewer than four fit an SM (CTAs of 512 threads)."""
    from oracle import dynamics, kpoints
    cell = _cell(n, bands)
    s = random_subsim(cell, (2, 2, 1), (0.25, 0.5, 0.125), 0.04, 3, PULSE, seed=230 + n[0])
    P, g = gpu_run(cell, [s], precision="fp32")
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 3, dynamics.field_samples(PULSE, s["dt"], 3),
                           ops=dynamics.Operators(cell), keep_state=False)
    compare(g[0], o, FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
