"""Lines too long for the segmented kernels, around the lengths where the kernel
that takes them changes: tiles of few lines with a thread per component (FP64,
up to 4098 points on few lines), with a thread per segment (up to 8194), and a
thread per line beyond that.  Against the oracle: FP64 rel-L2 <= 1e-12, FP32
2e-5 in imaginary time, 1e-4 in real time, as the other parity tests.
"""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("r", [2e-3, 1.0])     # dt / (4 dx^2): carries that die within a segment, and that cross some
@pytest.mark.parametrize("n", [(4098, 5), (4099, 5), (4, 5000), (8194, 3), (8195, 3), (6, 8195), (9000, 130)])
def test_longest_lines(n, r, prec, imag):
    from paper_1709_04423_gb300 import gpe
    n, nkl = list(n), [1.0, 1.3]
    dx = [14.0 / max(v, 14) for v in n]
    dt = min(4 * r * min(dx) ** 2, 5e-3)
    phi0 = I.gaussian_state(2, n, dx, nkl, seed=sum(n), noise=1e-2)
    p = gpe.Propagator(2, n, dx, dt, nkl, 8.0, precision=prec)
    long = 0 if n[0] > n[1] else 1
    assert p.sweep_kernels(imag)[long] == ("narrow" if n[long] <= 8194 else "thread")
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(5)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(2, n, dx, dt, nkl, 8.0), phi0, imag, 5)
    tol = 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


def run_line(n, prec, imag, steps=4):
    from paper_1709_04423_gb300 import gpe
    dx, nkl = 16.0 / n, [1.1]
    dt = 2.0 * dx * dx      # dt / (4 dx^2) = 0.5
    phi0 = I.gaussian_state(1, [n], [dx], nkl, seed=n, noise=1e-2)
    p = gpe.Propagator(1, [n], [dx], dt, nkl, 9.0, precision=prec)
    kernel = p.sweep_kernels(imag)[0]
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(steps)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(1, [n], [dx], dt, nkl, 9.0), phi0, imag, steps)
    tol = 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    return kernel


# a cluster of 16 blocks: 128 threads each first, then 416 and the largest, 512, then too long for it
@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_longest_1d_lines(prec, imag):
    for n in (6200, 26600, 32770):
        assert run_line(n, prec, imag) == "line"
    assert run_line(32771, prec, imag) == "thread"
