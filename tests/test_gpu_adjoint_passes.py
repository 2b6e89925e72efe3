"""The reverse step's two forms -- the x sweep that also applies the adjoint of N
(32-line tiles) and the separate pass (other x sweeps) -- and the last segment's
states kept from the forward run: a second backward pass, after the first has
overwritten them, must give the same gradients.  FP64 against the CPU adjoint at
the bounds of the other adjoint tests; partial tiles, lines over one 32-point
chunk, one segment, one step per segment.
"""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1709_04423_gb300 import gpe
    gpe.load()
    return gpe


@pytest.mark.parametrize("user_potential", [True, False])
@pytest.mark.parametrize("n,tile,K", [
    ([33, 20], 1, 4), ([70, 33], 1, 1), ([18, 35, 9], 1, 9), ([18, 35, 9], 1, 100),
    ([400, 12], 0, 4),      # FP64 lines whose 32-line tile does not fit
    ([40, 21], 0, 4),
])
def test_reverse_forms_and_repeated_backward(G, n, tile, K, user_potential):
    import torch
    dim, n = len(n), list(n)
    dx, nkl, dt, g, steps = [8.0 / v for v in n], [1.0, 1.2, 1.4][:dim], 2e-3, 6.0, 9
    gr = O.Grid(dim, n, dx, dt, nkl, g)
    if user_potential:
        gr = gr.with_(V=O.potential(gr) + I.gaussian_bumps(dim, n, dx, seed=3, count=4)[0])
    phi0 = I.gaussian_state(dim, n, dx, nkl, seed=11, noise=1e-2)
    target = I.gaussian_state(dim, n, dx, nkl, shift=(0.4, 0.0, 0.0))
    p = G.Propagator(dim, n, dx, dt, nkl, g, precision="f64")
    if user_potential:
        p.set_potential(gr.V)
    s = p.shapes()
    if not tile and n[0] <= 333:
        G.gp_set_shapes(p.h, 0, 2, s["seg_c"], s["flags"])
    p.set_state(phi0)
    G.gp_adjoint_forward(p.h, steps, K)
    dvol = float(np.prod(dx))
    c = np.sum(np.conj(target) * p.get_state(device=False)) * dvol
    lam = torch.tensor(2 * c * target * dvol, device="cuda")
    got = []
    for _ in range(2):
        dV = torch.empty(gr.shape, dtype=torch.float64, device="cuda")
        lam0 = torch.empty_like(lam)
        dg = G.gp_adjoint_backward(p.h, lam.data_ptr(), 1, dV.data_ptr(), 1, lam0.data_ptr())
        got.append((dV.cpu().numpy(), dg, lam0.cpu().numpy()))
    p.close()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1] and np.array_equal(got[0][2], got[1][2])
    J, _, dVr, dgr = O.adjoint_real(gr, phi0, target, steps)
    assert abs(c) ** 2 == pytest.approx(J, rel=1e-12)
    assert np.max(np.abs(got[0][0] - dVr)) <= 1e-10 * np.max(np.abs(dVr))
    assert got[0][1] == pytest.approx(dgr, rel=1e-10)
