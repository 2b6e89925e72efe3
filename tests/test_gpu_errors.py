"""What a sweep that could not do its work leaves behind: an error at the next
synchronising call, and no state that could be taken for a result.  The grid
takes the TMA sweeps by default, so a caller meets them without asking."""
import numpy as np
import pytest

import oracle as O
from tolerances import mu_tol_f32
from paper_1709_04423_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N, DX, NKL = [160, 144, 150], [0.09, 0.1, 0.1], [1.0, 1.4, 1.8]


@pytest.fixture(scope="module")
def G():
    import torch
    from paper_1709_04423_gb300 import gpe
    gpe.load()
    assert torch.cuda.is_available()
    return gpe


@pytest.fixture(scope="module")
def phi0():
    return I.gaussian_state(3, N, DX, NKL, seed=91, noise=1e-3).astype(np.complex64)


def default_handle(G, phi0, monkeypatch):
    monkeypatch.setenv("GPE_WAIT_LIMIT_MS", "20")
    p = G.Propagator(3, N, DX, 1e-3, NKL, 10.0, precision="f32")
    assert p.shapes()["flags"] & G.GP_SHAPE_TMA_X and p.shapes()["flags"] & G.GP_SHAPE_TMA_YZ
    p.set_state(phi0)
    return p


def recovers(G, p, phi0):
    p.set_state(phi0)
    p.step_imag(2)
    got = p.get_state(device=False).astype(np.complex128)
    ref = O.run(O.Grid(3, N, DX, 1e-3, NKL, 10.0), phi0.astype(np.complex128), True, 2)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


READS = {
    "state": lambda G, p: p.get_state(device=False),
    "series": lambda G, p: p.step_series(True, 2, 1, device=False),
    "density": lambda G, p: p.reduced_density((0,), device=False),
    "times": lambda G, p: p.time_sweeps(True, 1),
}


@pytest.mark.parametrize("read", READS)
def test_a_wait_that_ran_out_is_reported_by_every_host_read(G, phi0, monkeypatch, read):
    p = default_handle(G, phi0, monkeypatch)
    G.gp_test_stall_transfers(p.h, 16)
    p.step_imag(2)
    with pytest.raises(G.GPError) as e:
        READS[read](G, p)
    assert e.value.code == G.GP_ERR_TIMEOUT
    G.gp_test_stall_transfers(p.h, 0)
    recovers(G, p, phi0)      # the flag was cleared
    p.close()


def test_a_wait_that_ran_out_leaves_no_results_on_the_device(G, phi0, monkeypatch):
    """A read to device memory returns before the steps have run and cannot report them: it holds NaN."""
    import torch
    p = default_handle(G, phi0, monkeypatch)
    G.gp_test_stall_transfers(p.h, 16)
    p.step_real(2)
    out = torch.view_as_real(p.get_state(device=True))
    assert bool(torch.isnan(out).all())
    assert bool(torch.isnan(p.reduced_density((0, 1))).all())
    assert bool(torch.isnan(p.step_series(False, 2, 1)).all())
    with pytest.raises(G.GPError) as e:     # the error is still there for the next synchronising call
        p.observables()
    assert e.value.code == G.GP_ERR_TIMEOUT
    G.gp_test_stall_transfers(p.h, 0)
    recovers(G, p, phi0)
    assert bool(torch.isfinite(torch.view_as_real(p.get_state(device=True))).all())
    p.close()


CALLS = {
    "step_imag": lambda G, p: p.step_imag(2),
    "step_real": lambda G, p: p.step_real(40),      # (a captured block of steps among them)
    "time_sweeps": lambda G, p: p.time_sweeps(True, 1),
    "time_sweeps_graph": lambda G, p: p.time_sweeps_graph(False, 2),
    "adjoint": lambda G, p: G.gp_adjoint_forward(p.h, 3, 2),
    "series": lambda G, p: p.step_series(True, 2, 1),
}


@pytest.mark.parametrize("call", CALLS)
def test_a_refused_tensor_map_is_an_error(G, phi0, monkeypatch, call):
    p = default_handle(G, phi0, monkeypatch)
    G.gp_test_refuse_maps(p.h, 1)
    with pytest.raises(G.GPError) as e:
        CALLS[call](G, p)
    assert e.value.code == G.GP_ERR_CUDA and "tensor map" in str(e.value)
    G.gp_test_refuse_maps(p.h, 0)
    recovers(G, p, phi0)
    p.close()


def test_a_wait_that_ran_out_while_tuning_is_the_tuners_error(G, phi0, monkeypatch):
    """The state is put back, so a read after it finds it and no error."""
    p = default_handle(G, phi0, monkeypatch)
    shapes = p.shapes()
    G.gp_test_stall_transfers(p.h, 16)
    with pytest.raises(G.GPError) as e:
        G.gp_autotune(p.h, False, 1)
    assert e.value.code == G.GP_ERR_TIMEOUT and "gp_autotune" in str(e.value)
    G.gp_test_stall_transfers(p.h, 0)
    assert p.shapes() == shapes
    assert np.array_equal(p.get_state(device=False), phi0)
    assert np.array_equal(p.get_state(device=True).cpu().numpy(), phi0)
    p.close()
