"""v_Hxc plane by plane against the oracle on grids whose axes take each of its
line transforms (2^n in two parts, plain sums, mixed), odd and even y axes, one
and several sub-simulations, just below and above the size from which grids that
are no power of two take it.  The density and current of a self-consistent step
depend on v_Hxc; bars of the double-precision parity tests."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, oracle_run, random_subsim

pytestmark = pytest.mark.gpu

GRIDS = [((13, 12, 15), 1), ((16, 11, 12), 1), ((32, 8, 9), 1), ((9, 32, 8), 1), ((8, 8, 32), 1), ((10, 12, 14), 2),
         ((10, 12, 17), 1), ((10, 12, 18), 1), ((16, 8, 16), 2), ((7, 30, 11), 1)]


@pytest.mark.parametrize("case", range(len(GRIDS)))
def test_vhxc_planes_vs_oracle(case):
    n, n_sub = GRIDS[case]
    cell = W.cell_tiny(atoms="offgrid", n=n, a=tuple(0.7 * v for v in n), n_bands=2)
    subs = [random_subsim(cell, (1, 1, 1), (0.25 + 0.2 * j, 0.5, 0.1), 0.04, 2, W.Kick(k0=0.01), seed=120 + case, tag=j)
            for j in range(n_sub)]
    P, g = gpu_run(cell, subs, precision="fp64")
    P.close()
    for s, r in zip(subs, g):
        compare(r, oracle_run(cell, s), FP64_J_TOL, FP64_RHO_TOL)
