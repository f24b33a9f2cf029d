"""A cell with an odd number of orbital values before cells whose kernels copy in bulk
(16-byte starts): each sub-simulation of one context against the oracle."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import (FP32_J_TOL, FP32_NORM_TOL, FP32_RHO_TOL, FP64_J_TOL, FP64_RHO_TOL, compare, oracle_run,
                        random_subsim)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_odd_cell_first(precision):
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints

    def pair(n, bands):
        return W.cell_tiny(atoms="pair", n=n, a=tuple(0.72 * v for v in n), n_bands=bands)

    P = Propagator(precision)
    runs = []
    for i, (cell, mp) in enumerate([(pair((7, 9, 11), 3), (1, 1, 1)), (W.cell_a(n_bands=3), (1, 1, 1)),
                                    (pair((5, 7, 9), 1), (1, 1, 3)), (pair((32, 16, 16), 2), (1, 1, 1))]):
        s = random_subsim(cell, mp, (0.25, 0.5, 0.125), 0.05, 2, W.Kick(k0=0.01), seed=330 + i)
        cid = P.add_cell_spec(cell)
        runs.append((P.add_subsim(cid, shifted_kpoints(cell.a, s["mp"], s["shift"]), s["dt"], 2), cell, s))
    for sid, _, s in runs:
        P.load_ground_state(sid, s["psi"])
        P.set_kick(sid, s["field"].k0, s["field"].direction)
    P.propagate(2)
    for sid, cell, s in runs:
        J, j0 = P.current(sid)
        g = dict(J=J, J0m=j0, rho=P.density(sid), norms=P.norms(sid))
        if precision == "fp64":
            compare(g, oracle_run(cell, s), FP64_J_TOL, FP64_RHO_TOL)
        else:
            compare(g, oracle_run(cell, s), FP32_J_TOL, FP32_RHO_TOL, FP32_NORM_TOL)
    P.close()
