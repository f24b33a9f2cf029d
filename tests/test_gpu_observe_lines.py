"""Observation of 32^3 single-precision cells by whole lines against the oracle: a field
along each axis alone and along none, one band and bands that the groups do not divide."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, compare, gpu_run, oracle_run, random_subsim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bands,direction", [(1, (1.0, 0.0, 0.0)), (5, (0.0, 1.0, 0.0)), (9, (0.6, 0.0, 0.8))])
def test_observe_lines_vs_oracle(bands, direction):
    cell = W.cell_tiny(atoms="offgrid", n=(32, 32, 32), a=(20.0, 21.0, 22.0), n_bands=bands)
    s = random_subsim(cell, (1, 2, 1), (0.25, 0.5, 0.125), 0.05, 1, W.Kick(k0=0.01, direction=direction), seed=350 + bands)
    P, g = gpu_run(cell, [s], precision="fp32")
    P.close()
    compare(g[0], oracle_run(cell, s), FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
