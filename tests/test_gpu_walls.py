"""A potential that is infinite or undefined at the end points of a line, where
the state is held at zero: no step reads it there, in any precision.  Against
the oracle with a finite value at the ends (which it does not read either);
tolerances of the other 1d tests."""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wall", [np.inf, np.nan])
@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("n", [40, 300])
def test_walls_at_the_end_points(n, prec, imag, wall):
    from paper_1709_04423_gb300 import gpe
    dx, dt, nkl, g = 12.0 / n, 1e-3, [1.0], 6.0
    V = O.potential(O.Grid(1, [n], [dx], dt, nkl, g)) + np.sin(O.coords(n, dx))
    phi0 = I.gaussian_state(1, [n], [dx], nkl, seed=n, noise=1e-2)
    Vw = V.copy()
    Vw[0] = Vw[-1] = wall
    p = gpe.Propagator(1, [n], [dx], dt, nkl, g, precision=prec)
    p.set_potential(Vw)
    p.set_state(phi0)
    (p.step_imag if imag else p.step_real)(20)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(1, [n], [dx], dt, nkl, g, V=V), phi0, imag, 20)
    tol = 1e-12 if prec != "f32" else (2e-5 if imag else 1e-4)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
