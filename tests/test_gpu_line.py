"""Every step of a 1d grid in one launch: edges of threads, warps, blocks and
clusters, weak and strong coupling (carries that die within a thread, and
carries that cross several warps), every precision, against the oracle.

FP64 and double-float: rel-L2 <= 1e-12 (as the other parity tests after 1000
steps); FP32: 2e-5 in imaginary time, 1e-4 in real time (likewise).
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


# interior points M = n - 2 on both sides of one warp, one block of S points per thread, a cluster of 2, 4, 8, 16
SIZES = [3, 4, 34, 35, 66, 67, 130, 258, 259, 514, 515, 1026, 1027, 2050, 2051, 6146, 6147, 9000]
# |alpha| ~ 1e-3 and ~0.5 in either precision's reach (dt / (4 dx^2) = 1e-3, 2)
COUPLING = [1e-3, 2.0]


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("r", COUPLING)
@pytest.mark.parametrize("n", SIZES)
def test_line_sizes(G, n, r, prec, imag):
    if prec == "df64" and n > 514:
        pytest.skip("the double-float form takes at most 514 points per axis")
    dx = 16.0 / max(n, 8)
    dt = min(4 * r * dx * dx, 2e-2)
    steps = 5 if n > 2000 else 20
    phi0 = I.gaussian_state(1, [n], [dx], [1.1], seed=n, noise=1e-2)
    if not imag:
        phi0 = phi0 * np.exp(0.7j * O.coords(n, dx))
    gr = O.Grid(1, [n], [dx], dt, [1.1], 9.0)
    p = G.Propagator(1, [n], [dx], dt, [1.1], 9.0, precision=prec)
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(steps)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    tol = 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)
    assert rel_l2(got, O.run(gr, phi0, imag, steps)) <= tol


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("geom", [0, 1, 2])
def test_line_strang_potential_and_traps(G, geom, prec, imag):
    n, dx, dt = 300, 0.04, 1e-3
    nkl, g = [1.3], 20.0
    x = np.arange(n) * dx
    phi0 = (np.exp(-0.5 * (x - 3.0) ** 2) * x * (1 + 0.1j)).astype(complex)
    V = 0.5 * x * x + np.sin(x)
    kw = {1: {"spherical": True}, 2: {"axisym": True}}.get(geom, {})
    gr = O.Grid(1, [n], [dx], dt, nkl, g, V=V, geom=geom, split=1)
    p = G.Propagator(1, [n], [dx], dt, nkl, g, precision=prec, **kw)
    p.set_potential(V)
    p.set_splitting("strang")
    p.set_state(phi0)
    for k in (1, 2, 33):   # the run's opening and closing halves, alone and around whole steps
        (p.step_imag if imag else p.step_real)(k)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    tol = 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)
    assert rel_l2(got, O.run(gr, phi0, imag, 36)) <= tol
