"""Band norms whose point tiles are shared by a warp's lanes: few bands on grids of many tiles, on
both sides of the rule, units of a warp and units of a whole CTA, against the oracle; and the
finalize of such a run is a small kernel beside the observation that reads the orbitals."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, oracle_run, random_subsim

pytestmark = pytest.mark.gpu

# grid, bands, subgrid
CASES = [((20, 18, 19), 1, (1, 1, 1)), ((20, 18, 19), 33, (1, 1, 1)), ((13, 14, 13), 1, (13, 10, 1)),
         ((13, 14, 13), 2, (13, 10, 1)), ((32, 32, 33), 3, (1, 2, 1))]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_norms_vs_oracle(case):
    n, bands, mp = CASES[case]
    cell = W.cell_tiny(atoms="none", n=n, a=tuple(0.7 * v for v in n), n_bands=bands)
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.04, 1, W.Kick(k0=0.01), seed=370 + case)
    P, g = gpu_run(cell, [s], precision="fp64")
    P.close()
    compare(g[0], oracle_run(cell, s), FP64_J_TOL, FP64_RHO_TOL)


def test_finalize_is_small_beside_the_observation():
    """64^3, 8 bands: 2048 tiles per band (observation 121 us; the finalize 16 us, and 145 us with a
    thread per band)."""
    cell = W.cell_tiny(atoms="none", n=(64, 64, 64), a=(40.0, 40.0, 40.0), n_bands=8)
    rng = np.random.default_rng(7)
    psi = rng.standard_normal((1, 8, 64, 64, 64)) + 1j * rng.standard_normal((1, 8, 64, 64, 64))
    s = dict(mp=(1, 1, 1), shift=(0.0, 0.0, 0.0), psi=psi * 1e-3, dt=0.01, n_steps=12, field=W.Kick(k0=0.01))
    P, _ = gpu_run(cell, [s], precision="fp64", steps=2, graphs=False)
    P.set_profiling(True)
    P.propagate(2)
    a = P.timings()
    P.propagate(8)
    b = P.timings()
    P.close()
    assert b["finalize"] - a["finalize"] < b["observe"] - a["observe"]
