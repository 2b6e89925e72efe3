"""The renormalisation of FP32 states on lines of more than 514 points: their
squares and Simpson weights are summed in FP64 whatever their size, so states
whose squared moduli leave the FP32 range (2e-23 squared underflows, the sum of
squares of 5e18 overflows) come out normalised, as the oracle's do.

rel-L2 <= 2e-5 (the FP32 imaginary-time tolerance of the other parity tests).
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


# a 1d line in one block and over a cluster; a long last axis, a long first and last, a short last axis
# beside a long one; 3d
SIZES = [(515,), (9000,), (40, 600), (530, 540), (21, 700, 9), (9, 6, 530)]


@pytest.mark.parametrize("amp,g", [(2e-23, 8.0), (5e18, 0.0)])
@pytest.mark.parametrize("n", SIZES)
def test_states_whose_squares_leave_the_fp32_range(G, n, amp, g):
    dim, n = len(n), list(n)
    nkl = [1.0, 1.3, 1.6][:dim]
    dx = [14.0 / max(v, 14) for v in n]
    dt = min(0.5 * min(dx) ** 2, 5e-3)
    phi0 = (amp * I.gaussian_state(dim, n, dx, nkl, seed=sum(n), noise=1e-2)).astype(np.complex64)
    p = G.Propagator(dim, n, dx, dt, nkl, g, precision="f32")
    p.set_state(phi0)
    p.step_imag(6)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(dim, n, dx, dt, nkl, g), phi0.astype(np.complex128), True, 6)
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("amp", [2e-23])
def test_radial_line(G, amp):
    n, dx, dt = 700, 0.02, 2e-4
    r = np.arange(n) * dx
    phi0 = (amp * r * np.exp(-0.5 * r * r)).astype(np.complex64)
    p = G.Propagator(1, [n], [dx], dt, [1.1], 8.0, precision="f32", spherical=True)
    p.set_state(phi0)
    p.step_imag(6)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(1, [n], [dx], dt, [1.1], 8.0, geom=1), phi0.astype(np.complex128), True, 6)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
