"""The observation's band groups against the oracle: bands that the groups do not
divide, one and many units, every observation kernel, and the finalize's ways of
sharing a unit (a warp, a whole CTA, more units than tiles).  Bars of the other
parity tests of each precision."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import (FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run,
                        oracle_run, random_subsim)

pytestmark = pytest.mark.gpu


def _pair(n, bands, a):
    return W.cell_tiny(atoms="pair", n=n, a=a, n_bands=bands)


CASES = [
    # (precision, cell, subgrid): fused 16^3 form, slab form, point-parallel form
    ("fp32", W.cell_a(n_bands=7), (1, 1, 1)),
    ("fp32", W.cell_a(n_bands=5), (2, 2, 1)),
    ("fp32", W.cell_a(n_bands=1), (2, 1, 1)),
    ("fp32", _pair((32, 16, 16), 5, (20.0, 10.0, 10.5)), (1, 2, 1)),
    ("fp32", _pair((10, 9, 11), 37, (7.0, 6.3, 7.7)), (1, 1, 1)),
    ("fp64", _pair((8, 8, 8), 33, (6.0, 6.0, 6.0)), (1, 1, 1)),
    ("fp64", _pair((8, 8, 8), 3, (6.0, 6.0, 6.0)), (4, 4, 2)),
    ("fp32", _pair((8, 8, 8), 2, (6.0, 6.0, 6.0)), (7, 7, 7)),     # 343 units over the tiles' warps
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_band_groups_vs_oracle(case):
    precision, cell, mp = CASES[case]
    s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.05, 1, W.Kick(k0=0.01), seed=160 + case)
    P, g = gpu_run(cell, [s], precision=precision)
    P.close()
    if precision == "fp64":
        compare(g[0], oracle_run(cell, s), FP64_J_TOL, FP64_RHO_TOL)
    else:
        compare(g[0], oracle_run(cell, s), FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
