"""The tile shapes that small domains are not given by themselves, so that the
kernels of the large ones (marched x1 tiles and tall x2 tiles in binary32, the
marched x2 sweep in binary64) meet every border rule, limiter, form and degenerate
size as well.  Against the oracle, with the bars of tests/test_gpu_parity.py for
the same cases."""
import functools

import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl

from helpers import Case, gpu_config, gpu_domain, pert_rel_linf, pressure_errors, run_gpu, run_oracle
from test_gpu_parity import TOL32, TOL64, _cases

pytestmark = pytest.mark.gpu

P, E, R, T, H = (fvna.BC_PERIODIC, fvna.BC_EXTRAP, fvna.BC_REFLECT, fvna.BC_TAYLOR,
                 fvna.BC_HIFU)
SHAPES32 = [(16, 10), (32, 18), (64, 42), (60, 26)]
SHAPES64 = [(32, 9), (64, 64)]
PARITY = {name: (case, steps) for name, case, steps in _cases()}


def _driven_cases():
    n = 60
    taylor = wl.taylor_initial(n, n, 0.1, 1e-4, x0=-3.0, y0=-3.0, angle=np.pi / 8)
    smooth = wl.random_smooth(96, 96, 1e-3, seed=57)
    mixed = dict(beta=3.5, delta=2e-3, dx=1.0 / 24, taylor_ratio=1e-4, y0=0.0)
    return {
        "taylor": (Case(n, n, taylor, bc=(T,) * 4, beta=3.5, delta=3.5e-4, dx=0.1, x0=-3.0, y0=-3.0,
                        taylor_ratio=1e-4, taylor_angle=np.pi / 8), 40),
        "taylor_x_reflect": (Case(96, 96, smooth, bc=(T, T, R, E), **mixed), 100),
        "reflect_taylor_low": (Case(96, 96, smooth, bc=(R, E, T, E), **mixed), 100),
        "hifu": (Case(90, 50, wl.ambient(90, 50), bc=(H, E, R, E), beta=4.8, delta=2.974e-4, dx=0.1,
                      amp=4.217e-4, focal=5.0, aperture=3.0, envelope=1, t0=-4.0), 80),
        # undriven rows on both sides of the driven ones
        "hifu_off_axis": (Case(90, 50, wl.ambient(90, 50), bc=(H, R, E, E), beta=4.8, delta=2.974e-4,
                               dx=0.1, amp=4.217e-4, focal=5.0, aperture=3.0, envelope=1, t0=-4.0,
                               y0=-1.5), 80),
        "axisymmetric": (Case(64, 40, wl.centred_gaussian(64, 40, 2e-3, 5.0), bc=(E, E, R, E),
                              geometry=1, delta=2e-3, dx=1.0 / 16), 30),
        "axisymmetric_rough": (Case(70, 101, wl.random_cells(70, 101, 1e-3, seed=58),
                                    bc=(P, P, R, R), geometry=1, delta=1e-3), 20),
    }


DRIVEN = _driven_cases()


@functools.lru_cache(maxsize=None)
def _oracle(name):
    return run_oracle(*{**PARITY, **DRIVEN}[name])


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1311_3004_gb300 import build
    build.build()


@pytest.mark.parametrize("tile_x,tile_y", SHAPES64)
@pytest.mark.parametrize("name", list(PARITY))
def test_parity_fp64(name, tile_x, tile_y):
    case, steps = PARITY[name]
    qo, so = _oracle(name)
    qg, sg = run_gpu(case, steps, tile_x=tile_x, tile_y=tile_y)
    assert sg["rc"] == 0 and sg["steps"] == so["step"] == steps and sg["t"] == so["t"]
    assert pert_rel_linf(qg, qo) <= TOL64


@pytest.mark.parametrize("tile_x,tile_y", SHAPES32)
@pytest.mark.parametrize("name", list(PARITY))
def test_parity_fp32(name, tile_x, tile_y):
    case, steps = PARITY[name]
    qo, so = _oracle(name)
    qg, sg = run_gpu(case, steps, precision=fvna.FP32_PERT, tile_x=tile_x, tile_y=tile_y)
    assert sg["rc"] == 0 and sg["steps"] == so["step"] == steps
    assert pert_rel_linf(qg, qo) <= TOL32


@pytest.mark.parametrize("tile_x,tile_y", [(0, 0)] + SHAPES64)
@pytest.mark.parametrize("name", list(DRIVEN))
def test_driven_fp64(name, tile_x, tile_y):
    case, steps = DRIVEN[name]
    qo, so = _oracle(name)
    qg, sg = run_gpu(case, steps, tile_x=tile_x, tile_y=tile_y)
    assert so["status"] == 0 and sg["rc"] == 0
    if name.startswith("axisymmetric"):          # no analytic values: the same bits
        assert pert_rel_linf(qg, qo) <= TOL64
    else:
        assert pert_rel_linf(qg, qo) <= 5e-11 and np.max(np.abs(qg - qo)) <= 1e-14


@pytest.mark.parametrize("tile_x,tile_y", [(0, 0)] + SHAPES32)
@pytest.mark.parametrize("name", list(DRIVEN))
def test_driven_fp32(name, tile_x, tile_y):
    case, steps = DRIVEN[name]
    qo, so = _oracle(name)
    qg, sg = run_gpu(case, steps, precision=fvna.FP32_PERT, tile_x=tile_x, tile_y=tile_y)
    assert so["status"] == 0 and sg["rc"] == 0
    peak, l2 = pressure_errors(qg[0] - 1.0, qo[0] - 1.0)
    assert peak <= 1e-5 and l2 <= 1e-5, (peak, l2)


@pytest.mark.parametrize("precision,shapes", [(fvna.FP64, SHAPES64), (fvna.FP32_PERT, SHAPES32)])
def test_budgets(precision, shapes):
    """The sum of the state changes by minus the outflow (the bars of
    tests/test_gpu_budget.py: 1e-11 and 2e-5 of the largest change)."""
    n, m = 120, 90
    q0 = wl.gaussian_pulse(n, m, 2e-3, 6.0, seed=3)
    q0[1] += 0.3 * (q0[0] - 1.0)
    c = Case(n, m, q0, bc=(E, E, E, E), delta=2e-3, dx=1.0 / 24)
    for tile_x, tile_y in shapes:
        s = fvna.Solver(gpu_config(c, precision, tile_x=tile_x, tile_y=tile_y), [gpu_domain(c)],
                        [q0])
        b0 = (np.array([np.sum(q0[0] - 1.0), np.sum(q0[1]), np.sum(q0[2])])
              if precision == fvna.FP64 else s.budget(0))
        s.set_budgets(True)
        s.run(max_steps=400)
        change, out = s.budget(0) - b0, s.outflow(0)
        s.close()
        scale = np.max(np.abs(change))
        assert scale > 1e-4
        tol = 1e-11 if precision == fvna.FP64 else 2e-5
        assert np.max(np.abs(change + out)) <= tol * scale, (tile_x, tile_y, change, -out)
