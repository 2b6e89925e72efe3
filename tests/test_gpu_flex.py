"""Sweeps on tiles of few lines: lines over 514 points, grids with few 32-line
tiles, partial tiles and segments, weak and strong coupling, axial traps and
the Strang splitting, every precision, against the oracle.

FP64 and double-float: rel-L2 <= 1e-12; FP32: 2e-5 in imaginary time, 1e-4 in
real time (as the other parity tests, which run longer).
"""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    from paper_1709_04423_gb300 import gpe
    gpe.load()
    assert torch.cuda.is_available()
    return gpe


def rel_l2(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def tol(prec, imag):
    return 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)


# long x, long y, both; a tile of one line short and over; few lines; 3d with a long axis
LONG = [(515, 40), (40, 515), (700, 601), (1030, 33), (21, 2050), (4100, 5), (530, 7, 6), (9, 6, 530)]
SHORT = [(257, 201), (512, 34), (33, 512), (66, 67), (400, 5), (3, 300), (20, 17, 33)]


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("r", [2e-3, 1.0])     # dt / (4 dx^2): carries that die within a segment, and that cross some
@pytest.mark.parametrize("n", LONG + SHORT)
def test_few_lines_and_long_lines(G, n, r, prec, imag):
    if prec == "df64" and max(n) > 514:
        pytest.skip("the double-float form takes at most 514 points per axis")
    dim, n = len(n), list(n)
    nkl = [1.0, 1.3, 1.6][:dim]
    dx = [14.0 / max(v, 14) for v in n]
    dt = min(4 * r * min(dx) ** 2, 5e-3)
    steps = 12
    phi0 = I.gaussian_state(dim, n, dx, nkl, seed=sum(n), noise=1e-2)
    V = None
    if n[0] % 2:
        V = O.potential(O.Grid(dim, n, dx, dt, nkl, 8.0)) + I.gaussian_bumps(dim, n, dx, seed=5)[0]
    gr = O.Grid(dim, n, dx, dt, nkl, 8.0, V=V)
    p = G.Propagator(dim, n, dx, dt, nkl, 8.0, precision=prec)
    if V is not None:
        p.set_potential(V)
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(steps)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    assert rel_l2(got, O.run(gr, phi0, imag, steps)) <= tol(prec, imag)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("n", [(96, 130), (400, 45), (50, 514)])
def test_axial_strang(G, n, prec, imag):
    n, dx, nkl, dt = list(n), [6.0 / n[0], 12.0 / n[1]], [1.0, 1.7], 5e-4
    rho, z = O.axisym_coords(n[0], dx[0]), O.coords(n[1], dx[1])
    phi0 = np.exp(-0.5 * (rho[None, :] ** 2 + 1.7 * (z[:, None] - 0.2) ** 2)).astype(complex)
    gr = O.Grid(2, n, dx, dt, nkl, 30.0, geom=2, split=1)
    p = G.Propagator(2, n, dx, dt, nkl, 30.0, precision=prec, axisym=True)
    p.set_splitting("strang")
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(40)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    assert rel_l2(got, O.run(gr, phi0, imag, 40)) <= tol(prec, imag)


def test_many_norm_sums_of_long_lines(G):
    """A grid whose last sweep leaves more sums than the next step adds up itself (they are folded first)."""
    n, dx, nkl, dt = [130, 130, 520], [0.1, 0.1, 0.03], [1.0, 1.2, 1.4], 2e-4
    phi0 = I.gaussian_state(3, n, dx, nkl, seed=8, noise=1e-3)
    p = G.Propagator(3, n, dx, dt, nkl, 10.0, precision="f32")
    p.set_state(phi0)
    p.step_imag(4)
    got = p.get_state(device=False).astype(np.complex128)
    norm = p.observables()["norm"]
    p.close()
    assert abs(norm - 1.0) <= 1e-6
    assert rel_l2(got, O.run(O.Grid(3, n, dx, dt, nkl, 10.0), phi0, True, 4)) <= 2e-5
