"""v_Hxc on both sides of the rule between its frequency planes (2 launches) and the launches
over all points (9): flat, long and cubic grids that are no power of two, one and
several sub-simulations; which way runs, and the self-consistent step against the oracle.
Bars of the double-precision parity tests."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import FP64_J_TOL, FP64_RHO_TOL, compare, gpu_run, oracle_run, random_subsim

pytestmark = pytest.mark.gpu

# grid, sub-simulations, launches of v_Hxc
CASES = [((30, 10, 30), 1, 9), ((30, 10, 30), 8, 2), ((70, 9, 8), 1, 9), ((8, 70, 9), 1, 2), ((64, 16, 64), 1, 9),
         ((24, 24, 24), 1, 2), ((36, 36, 36), 1, 9)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_vhxc_route(case):
    n, n_sub, launches = CASES[case]
    cell = W.cell_tiny(atoms="none", n=n, a=tuple(0.7 * v for v in n), n_bands=1)
    subs = [random_subsim(cell, (1, 1, 1), (0.25 + 0.05 * j, 0.5, 0.1), 0.04, 2, W.Kick(k0=0.01), seed=350 + case, tag=j)
            for j in range(n_sub)]
    P, _ = gpu_run(cell, subs, precision="fp64", steps=1, graphs=False)
    before = P.launches()
    P.propagate(1)
    # field, four stages, observation and finalize besides (or the whole step in one launch)
    assert P.launches() - before in (launches + 7, launches + 4)
    for sid in {0, n_sub - 1}:
        J, j0 = P.current(sid)
        compare(dict(J=J, J0m=j0, rho=P.density(sid), norms=P.norms(sid)), oracle_run(cell, subs[sid]), FP64_J_TOL,
                FP64_RHO_TOL)
    P.close()
