"""Double precision on 16^3 grids on both sides of the rule between the one-launch step (and
solver's filter) and the sequence of launches: which of them runs, and its results against
the oracle.  The one-launch side has six and two z groups, no projectors, narrow and
wide stencils and a field that changes every step.  Bars: those of the other parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu

_SIX = np.array([[0.05 * i + 0.1, 0.13 * i, 0.11 * i + 0.02] for i in range(6)])
_EIGHT = np.array([[0.1 * i, 0.37 * i % 1.0, (0.07 + 0.121 * i) % 1.0] for i in range(8)])
_THREE = np.array([[0.0, 0.1, 0.0], [0.3, 0.2, 0.5], [0.6, 0.7, 0.5]])
PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
KICK = W.Kick(k0=0.01)


def _cell(bands, atoms=None, **kw):
    c = W.cell_tiny(atoms="pair" if atoms is not None else "none", n=(16, 16, 16), a=(10.0, 11.0, 9.5), n_bands=bands)
    if atoms is not None:
        c = c.replace(atom_frac=atoms)
    return c.replace(**kw) if kw else c


# cell, subgrid, field, stencil half-width, launches of a Taylor step (6: one launch; 14, 9 without projectors)
CASES = [
    (lambda: _cell(12, _SIX), (1, 1, 1), KICK, 3, 6),
    (lambda: _cell(16, _THREE), (1, 1, 1), PULSE, 4, 6),
    (lambda: _cell(13, _EIGHT, proj_half=5.5), (2, 2, 1), PULSE, 6, 6),
    (lambda: _cell(16), (2, 2, 2), PULSE, 1, 6),
    (lambda: W.cell_a(n_bands=6), (2, 2, 2), KICK, 4, 6),
    (lambda: W.cell_a(n_bands=4), (2, 2, 2), KICK, 4, 14),
    (lambda: _cell(1, _THREE), (4, 2, 1), PULSE, 4, 14),
    (lambda: _cell(4, _EIGHT), (2, 1, 1), KICK, 4, 14),
    (lambda: _cell(8), (1, 1, 1), KICK, 4, 9),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("propagator", ["taylor4", "etrs"])
def test_step_and_route(case, propagator):
    from oracle import dynamics, kpoints
    make, mp, field, nd, per_step = CASES[case]
    cell = make()
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 2, field, seed=330 + case)
    P, g = gpu_run(cell, [s], precision="fp64", fd_nd=nd, propagator=propagator, steps=1, graphs=False)
    before = P.launches()
    P.propagate(1)
    if propagator == "taylor4":
        assert P.launches() - before == per_step
    J, j0 = P.current(0)
    out = dict(J=J, J0m=j0, rho=P.density(0), norms=P.norms(0))
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 2, dynamics.field_samples(field, s["dt"], 2),
                           ops=dynamics.Operators(cell, nd), keep_state=False, propagator=propagator)
    compare(out, o, FP64_J_TOL, FP64_RHO_TOL)


def test_restart_bitwise():
    cell = _cell(16, _THREE)
    s = random_subsim(cell, (1, 1, 1), (0.25, 0.5, 0.125), 0.04, 4, KICK, seed=340)
    P1, _ = gpu_run(cell, [s], precision="fp64", steps=2)
    mid, step = P1.get_state(0)
    P1.propagate(2)
    P2, _ = gpu_run(cell, [s], precision="fp64", steps=0)
    P2.load_state(0, mid, step)
    P2.propagate(2)
    np.testing.assert_array_equal(P1.get_state(0)[0], P2.get_state(0)[0])
    np.testing.assert_array_equal(P1.current(0)[0][3:], P2.current(0)[0][3:])
    P1.close()
    P2.close()


# 5 bands, or no projectors: the sequence of launches; 7: one launch (gaps above the last band)
@pytest.mark.parametrize("bands,atoms,shift", [(5, "pair", (0.25, 0.5, 0.125)), (7, "pair", (0.0, 0.0, 0.0)),
                                               (7, "none", (0.0, 0.0, 0.0))])
def test_ground_state_vs_oracle(bands, atoms, shift):
    from oracle import kpoints, scf
    from oracle.cell import Grid
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints
    cell = W.cell_tiny(n=(16, 16, 16), a=(6.0, 6.0, 6.0), n_bands=bands, atoms=atoms)
    gs = scf.ground_state(cell, kpoints.kpoints_cartesian(cell.a, (1, 1, 1), shift), seed=3, tol=1e-9)
    P = Propagator("fp64")
    sid = P.add_subsim(P.add_cell_spec(cell), shifted_kpoints(cell.a, (1, 1, 1), shift), 0.08, 1)
    P.load_ground_state(sid, W.random_orbitals(1, bands, cell.n, Grid(cell).dv, seed=61))
    _, err = P.ground_state(max_iter=150, tol=1e-9)
    rho = P.density(sid)
    P.close()
    assert err <= 1e-9
    assert np.max(np.abs(rho - gs["rho"])) <= 1e-7 * np.max(gs["rho"])
