"""Binary64 states that only the general form takes (a nonlinearity or a flow
beyond the others' bounds) against the oracle, bit for bit: zero waves beside
nonzero ones, faces that are subsonic and faces that are not in one warp, both x2
kernels, two and three dimensions."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl
from helpers import Case, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

P, E, R = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1311_3004_gb300 import build
    build.build()


def _state(name, n, m):
    q = wl.random_smooth(n, m, 2e-3, seed=7)
    q[:, m // 3:m // 2] = np.array([1.0, 0.0, 0.0])[:, None, None]   # a band at rest: zero waves
    if name == "slow flow":
        q[1:] += 0.1 * q[0]
    elif name == "mixed flow":           # subsonic (up to 1/sqrt(2)) beside not subsonic
        q[1] += q[0] * _flow(n)
    return q


def _flow(n):
    return 0.7 + 0.04 * np.cos(2.0 * np.pi * np.arange(n) / n)


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("tile_x,tile_y", [(0, 0), (64, 9)])
@pytest.mark.parametrize("name,beta", [("strong nonlinearity", 6.3), ("slow flow", 3.5),
                                       ("mixed flow", 3.5)])
def test_2d(name, beta, tile_x, tile_y, limiter):
    n, m = 95, 61
    c = Case(n, m, _state(name, n, m), bc=(P, P, R, E), beta=beta, delta=1e-3, nu_w=0.4,
             limiter=limiter)
    qo, so = run_oracle(c, 8)
    qg, sg = run_gpu(c, 8, tile_x=tile_x, tile_y=tile_y)
    assert so["status"] == 0 and sg["rc"] == 0
    assert np.array_equal(qg, qo)
    assert sg["dt"] == so["dt"] and sg["smax"] == so["smax"]


@pytest.mark.parametrize("axis", [0, 1, 2, 3])
def test_3d(axis):
    import oracle
    nx, ny, nz = 33, 30, 29
    q0 = wl.random_smooth3(nx, ny, nz, 2e-3, seed=axis)
    q0[:, 8:12] = np.array([1.0, 0.0, 0.0, 0.0])[:, None, None, None]
    if axis:
        q0[axis] += q0[0] * _flow(nx)
    cfg = dict(beta=3.5 if axis else 6.3, delta=1e-3, dx=1 / 24, nu_w=0.4)
    s = fvna.Solver3(fvna.make_config(precision=fvna.FP64, **cfg),
                     fvna.make_domain3(nx, ny, nz, (P,) * 6), q0)
    st = s.run(max_steps=5)
    q = s.q()
    s.close()
    qo, so = oracle.run3(oracle.Params3(nx=nx, ny=ny, nz=nz, bc=(P,) * 6, **cfg), q0, 5)
    assert st["steps"] == 5 and so["status"] == 0
    assert np.array_equal(q, qo)


def test_time_of_the_general_form():
    """A step wholly in the general form takes no more than 2.2 times one in the
    fast form at 2048 x 2048 (2.08 measured, scatter a percent; 3.99 ms against
    1.81, with one form in the kernels, is 2.2; plain operations and a 0/0 in
    every warp took 2.48)."""
    n = 2048
    q = wl.ambient(n, n)
    q[0] += 1e-3 * np.cos(0.05 * np.arange(n))[:, None] * np.cos(0.05 * np.arange(n))
    q[1:] += 1e-4 * (q[0] - 1.0)
    ms = []
    for beta in (3.5, 6.3):
        cfg = fvna.make_config(precision=fvna.FP64, beta=beta, delta=1e-4, dx=1 / 40,
                               dt_fixed=0.005)
        s = fvna.Solver(cfg, [fvna.make_domain(n, n)], [q])
        s.step_timed()
        ms.append(min(sum(s.step_timed()[:2]) for _ in range(5)))
        s.close()
    assert ms[1] <= 2.2 * ms[0], ms
