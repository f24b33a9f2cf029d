"""Single precision over long runs, against the library's own double precision on the same inputs:
errors that are the same every step (a rounded Taylor coefficient, the rounding of the kinetic
symbol and of the transforms' twiddles, sums that a tensor core cuts off) add up, where rounding noise
averages out.  Bars: 1.5 times what the star-stencil, FP32-contraction kernels that these whole-step
kernels replaced measured on these inputs on GB300 (1.5: the spread between inputs)."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _plane_waves(n, a, count, seed, reach):
    """Orthonormal combinations of the lowest plane waves (as smooth as ground-state orbitals)."""
    g = sorted(((i, j, k) for i in range(-reach, reach + 1) for j in range(-reach, reach + 1)
                for k in range(-reach, reach + 1)), key=lambda v: (v[0] ** 2 + v[1] ** 2 + v[2] ** 2, v))[: 2 * count]
    rng = np.random.default_rng(seed)
    c = np.eye(2 * count, count) + 0.15 * (rng.standard_normal((2 * count, count)) +
                                           1j * rng.standard_normal((2 * count, count)))
    c, _ = np.linalg.qr(c)
    z, y, x = (np.arange(m) / m for m in n[::-1])
    w = np.array([np.exp(2j * np.pi * (v[0] * x[None, None, :] + v[1] * y[None, :, None] + v[2] * z[:, None, None]))
                  for v in g]) / np.sqrt(a[0] * a[1] * a[2])
    return (c.T @ w.reshape(len(g), -1)).reshape((1, count) + n[::-1])


def _run(precision, cell, mp, psi, dt, steps):
    from paper_2112_00920_gb300 import Propagator, shifted_kpoints
    P = Propagator(precision)
    k = shifted_kpoints(cell.a, mp, (0.25, 0.5, 0.125))
    sid = P.add_subsim(P.add_cell_spec(cell), k, dt, max(steps, 1))
    P.load_ground_state(sid, np.repeat(psi, k.shape[0], axis=0))
    P.set_kick(sid, 0.005, (1.0, 0.0, 0.0))
    P.propagate(steps)
    out = dict(J=P.current(sid)[0], J0=P.current(sid)[1], rho=P.density(sid), norms=P.norms(sid))
    P.close()
    return out


def _far(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


CELLS = {
    "8": (lambda: W.cell_a_coarse(n=8), (2, 2, 2), 0.05, 1500),
    "16": (lambda: W.cell_a(), (2, 2, 2), 0.08, 300),
    "32": (lambda: W.cell_b(n_bands=16), (1, 1, 1), 0.08, 150),
    "10x12x14": (lambda: W.cell_tiny(atoms="offgrid", n=(10, 12, 14), a=(7.5, 9.0, 10.5), n_bands=8), (2, 2, 1), 0.05, 1000),
}


def test_strong_projectors():
    """J(0-) of one band of G = 0 over strong s projectors (32^3): nearly all of it their sums, 1.9e-7 off in
    FP32 products; 9.0e-7 with every product added to one tensor-core accumulator."""
    cell = W.cell_b(n_bands=1).replace(e_kb_s=60.0, e_kb_p=0.0)
    psi = np.full((1, 1) + cell.n[::-1], 1.0 / np.sqrt(cell.a[0] * cell.a[1] * cell.a[2]), dtype=np.complex128)
    a, b = (_run(p, cell, (1, 1, 1), psi, 0.01, 0) for p in ("fp32", "fp64"))
    far = _far(a["J0"], b["J0"])
    print("J(0-) off by", far)
    assert far <= 1.5 * 1.9e-7


# norms of the replaced kernels; with dt^2 / 2 rounded 9.4e-8 at 32^3 and 3.1e-7 at 10 x 12 x 14
@pytest.mark.parametrize("name,replaced", [("8", 6.5e-7), ("16", 1.72e-7), ("32", 2.96e-8), ("10x12x14", 1.81e-7)])
def test_norms(name, replaced):
    make, mp, dt, steps = CELLS[name]
    cell = make()
    psi = _plane_waves(cell.n, cell.a, cell.n_bands, 11, 3)
    a, b = (_run(p, cell, mp, psi, dt, steps) for p in ("fp32", "fp64"))
    far = float(np.max(np.abs(a["norms"] - b["norms"])))
    print(name, "norms off by", far)
    assert far <= 1.5 * replaced


# density of the replaced kernels; with the symbol's plain sums and the twiddles' gain left in 6.8e-7 and 3.8e-7
@pytest.mark.parametrize("name,replaced", [("8", 2.76e-7), ("16", 1.47e-7)])
def test_density(name, replaced):
    make, mp, dt, steps = CELLS[name]
    cell = make()
    psi = _plane_waves(cell.n, cell.a, cell.n_bands, 11, 3)
    a, b = (_run(p, cell, mp, psi, dt, steps) for p in ("fp32", "fp64"))
    far = _far(a["rho"], b["rho"])
    print(name, "density off by", far)
    assert far <= 1.5 * replaced
