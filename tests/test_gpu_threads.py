"""Two contexts on two host threads whose cells take the same kernels with different amounts
of shared memory (small grids and v_Hxc planes above 48 KB): neither may find its launch
refused by what the other one set, and each gets the bits of its run alone."""
from __future__ import annotations

import threading

import numpy as np
import pytest

import workloads as W
from gpu_common import random_subsim

pytestmark = pytest.mark.gpu

# (precision, atoms, smaller grid, larger grid, bands)
PAIRS = [("fp32", "offgrid", (16, 16, 8), (18, 18, 16), 8), ("fp64", "offgrid", (11, 11, 11), (15, 13, 15), 8),
         ("fp32", "none", (40, 8, 40), (60, 8, 60), 1)]
STEPS, CALLS = 60, 12


def _run(precision, cell, s, out, start=None):
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints
    try:
        P = Propagator(precision)
        P.set_graphs(False)
        sid = P.add_subsim(P.add_cell_spec(cell), shifted_kpoints(cell.a, s["mp"], s["shift"]), s["dt"], STEPS * CALLS)
        P.load_ground_state(sid, s["psi"])
        P.set_kick(sid, 0.01, (1.0, 0.0, 0.0))
        if start is not None:
            start.wait(60)
        for _ in range(CALLS):
            P.propagate(STEPS)
        out.append((P.current(sid)[0], P.density(sid)))
        P.close()
    except Exception as e:   # noqa: BLE001 (carried to the test's own thread)
        out.append(e)


@pytest.mark.parametrize("case", range(len(PAIRS)))
def test_contexts_on_two_threads(case):
    precision, atoms, small, large, bands = PAIRS[case]
    cells = [W.cell_tiny(atoms=atoms, n=n, a=tuple(0.72 * v for v in n), n_bands=bands) for n in (small, large)]
    subs = [random_subsim(c, (1, 1, 1), (0.25, 0.5, 0.125), 0.01, 1, None, seed=300 + case, tag=i)
            for i, c in enumerate(cells)]
    alone, both = [[], []], [[], []]
    for i in range(2):
        _run(precision, cells[i], subs[i], alone[i])
    start = threading.Barrier(2)
    threads = [threading.Thread(target=_run, args=(precision, cells[i], subs[i], both[i], start)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        for r in (alone[i][0], both[i][0]):
            assert not isinstance(r, Exception), r
        for a, b in zip(alone[i][0], both[i][0]):
            assert np.array_equal(a, b)
