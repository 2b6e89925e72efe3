"""The sub-step N and the renormalisation factor of 1d lines, alone: on a grid
whose spacing is so large that the Crank-Nicolson solve changes nothing
(dt / (4 dx^2) = 1e-21 or less), one step multiplies every point by exp(-i th) or
exp(-th) and, in imaginary time, by 1/sqrt(norm).  th = dt V at g = 0, so V puts
the angles on both sides of every limit between two series (1/32, 1/4) and far
beyond; the size of the state puts the norm anywhere.  Against extended precision
(long double).

Tolerances, relative to the point, u = 2^-53 (FP64) or 2^-24 (FP32); dt is a power
of two, so the angle is exact.
Real time: the coefficients cos th - 1 = -2 sin^2(th/2) and sin th = 2 sin(th/2)
cos(th/2) carry 9 u each at most (the library's sincos 2 ulp, twice, and the
product), are below 2 and 1 and shrink with the angle; the sum adds 4 u:
(4 + 28 min(|th|, 1)) u.  Imaginary time: exp (2 ulp at most) and the product 6 u, the
factor 10 u (the sum over 40 points 10 u, halved by the root; weights, root and
product 4 u), and the norm of points that are 6 u off: 22 u.  Double-float: chains
of 8 (N) and 10 more (the factor) operations of at most 4 2^-48 each.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, DX, DT = 40, 1e9, 2.0 ** -10
E = np.longdouble(2.0)


def angles():
    a = []
    for lim in (2.0 ** -5, 2.0 ** -2, 2.0 ** -3):
        a += [lim * (1 - 2.0 ** -40), lim, lim * (1 + 2.0 ** -40), 0.97 * lim, 1.03 * lim, 0.5 * lim]
    a += [1e-300, 1e-20, 1e-9, 1e-3, 0.6, 1.0, 1.5707963, 2.5, 3.1415926, 6.0, 11.0]
    a += [-v for v in a[:6]]
    return np.array((a + [0.01] * N)[: N - 2])


def one_step(prec, imag, V, psi):
    from paper_1709_04423_gb300 import gpe
    p = gpe.Propagator(1, [N], [DX], DT, [0.0], 0.0, precision=prec)
    assert p.sweep_kernels(imag) == ["line"]
    p.set_potential(V)
    p.set_state(psi)
    (p.step_imag if imag else p.step_real)(1)
    out = p.get_state(device=False)
    p.close()
    return out[1:-1].astype(np.clongdouble)


def simpson():
    w = np.zeros(N, dtype=np.longdouble)
    m = N if N % 2 else N - 1
    w[1:m - 1:2], w[2:m - 1:2], w[0], w[m - 1] = 4, 2, 1, 1
    return w * np.longdouble(DX) / 3


def state(prec, size):
    rng = np.random.default_rng(5)
    psi = size * (rng.uniform(0.5, 1.5, N) * np.exp(1j * rng.uniform(0, 6, N)))
    psi[0] = psi[-1] = 0
    return psi.astype(np.complex64 if prec == "f32" else np.complex128)


def tolerance(prec, th, imag):
    if prec == "df64":
        return (72 if imag else 32) * E ** -48 * np.ones_like(th)
    u = E ** (-53 if prec == "f64" else -24)
    return 22 * u * np.ones_like(th) if imag else (4 + 28 * np.minimum(np.abs(th), 1)) * u


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
def test_substep_over_its_ranges(prec, imag):
    th = angles()
    V = np.zeros(N)
    V[1:-1] = th / DT
    if prec == "f32":       # the potential the FP32 form holds
        V = V.astype(np.float32).astype(np.float64)
    t = np.longdouble(DT) * V[1:-1].astype(np.longdouble)
    psi = state(prec, 1.0)
    x = psi[1:-1].astype(np.clongdouble)
    ref = x * np.exp(-t) if imag else x * (np.cos(t) - 1j * np.sin(t))
    if imag:
        ref = ref / np.sqrt(np.sum(simpson()[1:-1] * np.abs(ref) ** 2))
    got = one_step(prec, imag, V, psi)
    err = np.abs(got - ref) / np.abs(ref)
    assert np.all(err <= tolerance(prec, t, imag)), (float(err.max()), int(err.argmax()))


# inside and outside the range where the FP64 factor starts from an FP32 estimate (norms 1e-30 to 1e30)
@pytest.mark.parametrize("size", [1e-140, 1e-60, 1e-25, 4e-21, 4.6e-21, 5e-21, 6e-21, 1e-9, 1.0, 1e3, 4e9, 4.6e9, 5e9,
                                  6e9, 1e25, 1e140])
@pytest.mark.parametrize("prec", ["f64", "df64", "f32"])
def test_renormalisation_over_its_range(prec, size):
    if prec != "f64" and not 1e-9 <= size <= 1e10:
        pytest.skip("squares and their low words leave the FP32 range")
    psi = state(prec, size)
    x = psi[1:-1].astype(np.clongdouble)
    ref = x / np.sqrt(np.sum(simpson()[1:-1] * np.abs(x) ** 2))
    got = one_step(prec, True, np.zeros(N), psi)
    err = np.abs(got - ref) / np.abs(ref)
    tol = 72 * E ** -48 if prec == "df64" else 10 * E ** (-53 if prec == "f64" else -24)
    assert np.all(err <= tol), float(err.max())
