"""Single-precision observation on grids of 16 planes, whose z-march kernel sums four neighbours a
side, with wider and narrower stencils, against the oracle with the same stencil."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, compare, gpu_run, random_subsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(12, 10, 16), (16, 16, 16)])
@pytest.mark.parametrize("nd", [2, 4, 5, 6])
def test_observation_of_16_planes(n, nd):
    from oracle import dynamics, kpoints
    cell = W.cell_tiny(atoms="pair", n=n, a=tuple(0.72 * v for v in n), n_bands=3)
    field = W.Kick(k0=0.01, direction=(0.0, 0.6, 0.8))
    s = random_subsim(cell, (2, 1, 1), (0.25, 0.5, 0.125), 0.04, 2, field, seed=320 + nd)
    P, g = gpu_run(cell, [s], precision="fp32", fd_nd=nd)
    P.close()
    k = kpoints.kpoints_cartesian(cell.a, s["mp"], s["shift"])
    # (the oracle's propagation of both the step and the current takes the stencil of its operators)
    o = dynamics.propagate(cell, k, s["psi"], s["dt"], 2, dynamics.field_samples(field, s["dt"], 2),
                           ops=dynamics.Operators(cell, nd), keep_state=False)
    compare(g[0], o, FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
