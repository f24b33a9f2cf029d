"""Ground states of one band: the Rayleigh matrix is a multiple of the identity, and the
shifted matrix of the power iteration must not vanish.  The solver converges and its
density is the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from oracle import kpoints, scf
from oracle.cell import Grid

pytestmark = pytest.mark.gpu

# cell, k shift: with projectors on both double-precision filters' grids, and free electrons
CASES = [(dict(n=(8, 8, 8), a=(6.0, 6.0, 6.0), n_bands=1, atoms="pair"), (0.25, 0.5, 0.125)),
         (dict(n=(16, 16, 16), a=(8.0, 8.0, 8.0), n_bands=1, atoms="pair"), (0.0, 0.0, 0.0)),
         (dict(n=(9, 10, 8), a=(6.0, 6.0, 6.0), n_bands=1, atoms="none"), (0.0, 0.0, 0.0))]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_ground_state_of_one_band(case):
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints
    spec, shift = CASES[case]
    cell = W.cell_tiny(**spec)
    g = Grid(cell)
    gs = scf.ground_state(cell, kpoints.kpoints_cartesian(cell.a, (1, 1, 1), shift), seed=3, tol=1e-9)
    P = Propagator("fp64")
    sid = P.add_subsim(P.add_cell_spec(cell), shifted_kpoints(cell.a, (1, 1, 1), shift), 0.08, 1)
    P.load_ground_state(sid, W.random_orbitals(1, cell.n_bands, cell.n, g.dv, seed=51 + case))
    _, err = P.ground_state(max_iter=150, tol=1e-9, degree=96)
    rho = P.density(sid)
    P.close()
    assert err <= 1e-9
    assert np.max(np.abs(rho - gs["rho"])) <= 1e-7 * np.max(gs["rho"])
