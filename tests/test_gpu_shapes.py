"""gp_set_shapes decides which kernels run, also on the grids whose default is
tiles of few lines (or, in 1d, a whole run in one launch), and gp_get_shapes and
gp_autotune speak of the kernels that run.  Every shape against the oracle
(FP64 and double-float rel-L2 <= 1e-12, FP32 2e-5 imaginary, 1e-4 real time),
and the 32-line shapes under the index checks of the checking build."""
import numpy as np
import pytest

import oracle as O
from paper_1709_04423_gb300 import inputs as I
from test_gpu_bounds import lib, run, status  # noqa: F401  (lib: the checking build, a fixture)

pytestmark = pytest.mark.gpu

TOL = {("f64", True): 1e-12, ("f64", False): 1e-12, ("df64", True): 1e-12, ("df64", False): 1e-12,
       ("f32", True): 2e-5, ("f32", False): 1e-4}
NARROW = 64 | 128
# grid, (tile_x, seg_x, seg_c, flags), the kernels they name (None: the default shapes)
CASES = [
    ((257, 201), None, None),
    ((257, 201), (1, 16, 16, 1), ["tile", "column"]),
    ((257, 201), (1, 32, 16, 0), ["tile", "column"]),
    ((257, 201), (0, 8, 32, 0), ["warp", "column"]),
    ((257, 201), (1, 16, 32, NARROW), ["narrow", "narrow"]),
    ((40, 33, 24), (1, 4, 4, 1), ["tile", "column", "column"]),
    ((40, 33, 24), (0, 2, 8, 0), ["warp", "column", "column"]),
    ((40, 33, 24), (1, 8, 4, 64), ["narrow", "column", "column"]),
    ((300,), None, ["line"]),
    ((300,), (0, 16, 0, 0), ["warp"]),
    ((300,), (0, 16, 0, 64), ["line"]),
]


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("n,shapes,kernels", CASES)
def test_the_shapes_that_were_set_run(n, shapes, kernels, prec, imag):
    from paper_1709_04423_gb300 import gpe as G
    n, dim = list(n), len(n)
    nkl, dx, dt, steps = [1.0, 1.4, 1.8][:dim], [12.0 / v for v in n], 5e-4, 40
    phi0 = I.gaussian_state(dim, n, dx, nkl, seed=71, noise=1e-3)
    p = G.Propagator(dim, n, dx, dt, nkl, 12.0, precision=prec)
    if shapes is not None:
        G.gp_set_shapes(p.h, *shapes)
        s = p.shapes()
        assert (s["tile_x"], s["seg_x"], s["seg_c"], s["flags"]) == shapes
    if kernels is not None:
        assert p.sweep_kernels(imag) == kernels
    else:
        assert p.sweep_kernels(imag)[0] == "narrow" and p.shapes()["flags"] & G.GP_SHAPE_NARROW_X
    p.set_state(phi0)
    before = G.gp_kernel_launches()
    (p.step_imag if imag else p.step_real)(steps)
    if dim == 1:
        assert G.gp_kernel_launches() - before == (1 if kernels == ["line"] else steps + (1 if imag else 0))
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(dim, n, dx, dt, nkl, 12.0), phi0, imag, steps)
    assert np.linalg.norm(got - ref) <= TOL[prec, imag] * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("n", [(300,), (257, 201), (400, 45), (40, 33, 24), (700,), (600, 40)])
def test_the_tuner_times_and_reports_what_runs(n, prec):
    from paper_1709_04423_gb300 import gpe as G
    if prec == "df64" and max(n) > 514:
        pytest.skip("the double-float form takes at most 514 points per axis")
    n, dim = list(n), len(n)
    nkl, dx, dt = [1.0, 1.4, 1.8][:dim], [12.0 / v for v in n], 1e-4
    phi0 = I.gaussian_state(dim, n, dx, nkl, seed=72, noise=1e-3)
    p = G.Propagator(dim, n, dx, dt, nkl, 12.0, precision=prec)
    p.set_state(phi0)
    ms = G.gp_autotune(p.h, True, 4, timings=True)
    s, kernels = p.shapes(), p.sweep_kernels(True)
    if s["seg_x"]:
        assert 0 < ms[0] < 1e3
        assert (kernels[0] in ("narrow", "line")) == bool(s["flags"] & G.GP_SHAPE_NARROW_X)
    if dim > 1 and s["seg_c"]:
        assert 0 < ms[1] < 1e3
        assert ("narrow" in kernels[1:]) == bool(s["flags"] & G.GP_SHAPE_NARROW_YZ)
    if dim == 1:
        before = G.gp_kernel_launches()
        assert p.time_sweeps(True, 16)[0] > 0 and p.time_sweeps_graph(True, 16)[0] > 0
        if kernels == ["line"]:
            assert G.gp_kernel_launches() - before == 2
        p.set_state(phi0)
    G.gp_set_shapes(p.h, *s.values())      # what a cache file would hold
    assert p.shapes() == s and p.sweep_kernels(True) == kernels
    p.set_state(phi0)
    p.step_imag(20)
    got = p.get_state(device=False).astype(np.complex128)
    p.close()
    ref = O.run(O.Grid(dim, n, dx, dt, nkl, 12.0), phi0, True, 20)
    assert np.linalg.norm(got - ref) <= TOL[prec, True] * np.linalg.norm(ref)


def test_a_real_state_keeps_the_complex_shapes():
    from paper_1709_04423_gb300 import gpe as G
    n, dx, nkl = [64, 40], [0.2, 0.3], [1.0, 1.2]
    p = G.Propagator(2, n, dx, 1e-3, nkl, 5.0, precision="f64")
    kernels = p.sweep_kernels(True)
    assert kernels == ["narrow", "narrow"]
    p.set_state(I.gaussian_state(2, n, dx, nkl).real.astype(complex))
    p.set_real_state(True)
    assert p.sweep_kernels(True) == ["tile", "column"]
    p.autotune(True, nsteps=2, cache=False)
    p.set_real_state(False)
    assert p.sweep_kernels(True) == kernels
    p.close()


def test_each_geometry_is_tuned_for_itself(tmp_path, monkeypatch):
    """A Cartesian grid's tuned shapes (here the pipelined x sweep) are not those of an axial trap of the same size."""
    from paper_1709_04423_gb300 import gpe as G
    monkeypatch.setenv("GPE_TUNE_CACHE", str(tmp_path / "shapes.json"))
    n, kw = [96, 4096 // 8], {"precision": "f64"}
    c = G.Propagator(2, n, [0.1, 0.1], 1e-4, [1.0, 1.0], 5.0, **kw)
    c.set_state(I.gaussian_state(2, n, [0.1, 0.1], [1.0, 1.0]))
    c.autotune(True, nsteps=2)
    import json
    table = json.load(open(tmp_path / "shapes.json"))
    key, = table
    table[key] = dict(tile_x=1, seg_x=8, seg_c=32, flags=G.GP_SHAPE_PIPE_X)   # as the tuner may pick it
    json.dump(table, open(tmp_path / "shapes.json", "w"))
    assert c.autotune(True)["flags"] & G.GP_SHAPE_PIPE_X
    a = G.Propagator(2, n, [0.1, 0.1], 1e-4, [1.0, 1.0], 5.0, axisym=True, **kw)
    a.set_state(np.ones((n[1], n[0]), dtype=complex))
    assert not a.autotune(True, nsteps=2)["flags"] & G.GP_SHAPE_PIPE_X
    assert len(json.load(open(tmp_path / "shapes.json"))) == 2
    c.close()
    a.close()


# imaginary time from 97 points on: FP32 rows with a pending factor arrive by cp.async
@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("prec", ["f64", "f32", "df64"])
@pytest.mark.parametrize("n,shapes", [((130, 37), (1, 16, 4, 1)), ((100, 9, 7), (1, 8, 4, 0)), ((257, 34), (1, 32, 8, 0)),
                                      ((130, 37), (0, 4, 4, 1)), ((17, 5), (1, 4, 4, 1)), ((130,), (0, 4, 0, 0))])
def test_explicit_shapes_pass_the_checks(lib, n, shapes, prec, imag):  # noqa: F811
    run(lib, len(n), list(n), [12.0 / v for v in n], prec, imag, 40, shapes=shapes)
    rc, code, msg = status(lib)
    assert rc == 0 and code == 0, (code, msg)
