"""A last sweep on tiles of few lines that leaves more norm sums than every block
of the next step should add up (4096): they are folded into one first, by a
launch of its own.  The launch count shows that the fold ran, in eager steps
and in replayed blocks; the state is held to the oracle (rel-L2 <= 2e-5, the
FP32 imaginary-time tolerance), the FP64 one to 1e-12."""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# a long y axis makes the z sweep general: 83200 lines of 20 points, 16 per tile
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,folded", [([160, 520, 20], True), ([124, 520, 20], False)])
def test_folded_norm_sums(n, folded, prec):
    from paper_1709_04423_gb300 import gpe
    dx, nkl, dt = [0.1, 0.03, 0.4], [1.0, 1.2, 1.4], 2e-4
    phi0 = I.gaussian_state(3, n, dx, nkl, seed=8, noise=1e-3)
    p = gpe.Propagator(3, n, dx, dt, nkl, 10.0, precision=prec)
    assert p.sweep_kernels(True)[1:] == ["narrow", "narrow"]
    p.set_state(phi0)
    for steps in (4, 40):     # eager steps; captured blocks of 16 among them
        before = gpe.gp_kernel_launches()
        p.step_imag(steps)
        assert gpe.gp_kernel_launches() - before == steps * (4 if folded else 3) + 1   # + the last factor
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(3, n, dx, dt, nkl, 10.0), phi0, True, 44)
    assert np.linalg.norm(got - ref) <= (2e-5 if prec == "f32" else 1e-12) * np.linalg.norm(ref)
