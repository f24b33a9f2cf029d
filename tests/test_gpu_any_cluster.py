"""Small grids in double precision whose bands are shared by clusters of four or two CTAs:
the orbital counts at the edges of the rule, rows that the CTAs do not divide (and fewer
rows than CTAs), no atoms, against the oracle; and a restart mid-run bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu

PULSE = W.Pulse(e0=0.05, omega0=0.4, t_pulse=2.0, direction=(0.3, 0.5, 0.8))
# grid, atoms, bands, subgrid, stencil half-width
CASES = [
    ((8, 8, 8), "pair", 19, (2, 2, 1), 4),      # 76 orbitals: the last with a cluster
    ((8, 8, 8), "pair", 11, (7, 1, 1), 4),      # 77: the first without
    ((8, 8, 8), "none", 3, (1, 3, 1), 4),
    ((9, 11, 10), "offgrid", 19, (1, 2, 1), 4),   # 38: four CTAs
    ((9, 10, 11), "offgrid", 13, (1, 1, 3), 4),   # 39: two
    ((9, 7, 8), "offgrid", 7, (11, 1, 1), 3),     # 77: one
    ((7, 3, 6), "pair", 4, (2, 1, 1), 1),
]


def _cell(i):
    n, atoms, bands, mp, nd = CASES[i]
    return W.cell_tiny(atoms=atoms, n=n, a=tuple(0.72 * v for v in n), n_bands=bands), mp, nd


@pytest.mark.parametrize("case", range(len(CASES)))
def test_cluster_vs_oracle(case):
    from oracle import dynamics, kpoints
    cell, mp, nd = _cell(case)
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 2, PULSE, seed=260 + case)
    P, g = gpu_run(cell, [s], precision="fp64", fd_nd=nd)
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 2, dynamics.field_samples(PULSE, s["dt"], 2),
                           ops=dynamics.Operators(cell, nd), keep_state=False)
    compare(g[0], o, FP64_J_TOL, FP64_RHO_TOL)


@pytest.mark.parametrize("case", [0, 3, 4])
def test_cluster_repeats_bitwise(case):
    """Two runs of the same inputs agree bit for bit (a lost barrier would show as a difference)."""
    cell, mp, nd = _cell(case)
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 20, W.Kick(k0=0.01), seed=270 + case)
    out = []
    for _ in range(3):
        P, g = gpu_run(cell, [s], precision="fp64", fd_nd=nd)
        out.append((g[0]["J"].copy(), P.get_state(0)[0].copy()))
        P.close()
    for J, psi in out[1:]:
        assert np.array_equal(J, out[0][0]) and np.array_equal(psi, out[0][1])


@pytest.mark.parametrize("n", [8, 10])
def test_ground_state_cluster_equals_single(n):
    """The solver's filter with a band per cluster (16 orbitals) and with a band per CTA (the
    same sub-simulation six times): the converged densities agree to the solver's tolerance."""
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints
    from oracle.cell import Grid
    cell = W.cell_a_coarse(n=n)
    start = W.random_orbitals(1, cell.n_bands, cell.n, Grid(cell).dv, seed=23)
    rho = []
    for copies in (1, 6):
        P = Propagator("fp64")
        cid = P.add_cell_spec(cell)
        sids = [P.add_subsim(cid, shifted_kpoints(cell.a, (1, 1, 1), (0.25, 0.5, 0.125)), 0.08, 1) for _ in range(copies)]
        for sid in sids:
            P.load_ground_state(sid, start)
        _, err = P.ground_state(max_iter=120, tol=1e-10)
        assert err <= 1e-10
        rho.append(P.density(sids[-1]))
        P.close()
    assert np.max(np.abs(rho[0] - rho[1])) <= 1e-8 * np.max(rho[1])


@pytest.mark.parametrize("case", [0, 3, 4])
@pytest.mark.parametrize("field", [PULSE, W.Kick(k0=0.01)])
def test_cluster_restart_bitwise(case, field):
    cell, mp, nd = _cell(case)
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 4, field, seed=280 + case)
    P1, _ = gpu_run(cell, [s], precision="fp64", fd_nd=nd, steps=2)
    mid, step = P1.get_state(0)
    P1.propagate(2)
    P2, _ = gpu_run(cell, [s], precision="fp64", fd_nd=nd, steps=0)
    P2.load_state(0, mid, step)
    P2.propagate(2)
    assert np.array_equal(P1.get_state(0)[0], P2.get_state(0)[0])
    assert np.array_equal(P1.density(0), P2.density(0))
    assert np.array_equal(P1.current(0)[0][3:], P2.current(0)[0][3:])
    P1.close()
    P2.close()
