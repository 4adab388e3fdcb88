"""Binary32 3D fields whose sound speed leaves the series of the subsonic form:
in some rows of a tile's march only (against the oracle, within the 1e-5 of
tests/test_gpu_3d.py), and everywhere, where a step may cost 1.5 times a usual one
(1.32 measured at 200^3; tiles marched to their end first took 1.65, general
lines alone 1.54)."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl
from test_gpu_3d import _rel, _run

pytestmark = pytest.mark.gpu

P, E, R = 0, 1, 2


@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("at", [0, 3, 6, 7, 8, 30, 44])
def test_strong_rows(axis, at):
    """Rows `at`..at+3 along x3 (axis 1) or x2 (axis 2) beyond the series, one tile a line."""
    nx, ny, nz = 67, 48, 48
    q0 = wl.random_smooth3(nx, ny, nz, 2e-3, seed=at)
    rows = [slice(None)] * 4
    rows[0], rows[axis], rows[3] = 0, slice(at, at + 4), slice(20, 40)
    q0[tuple(rows)] += 0.03
    q, st, qo, so = _run(nx, ny, nz, q0, (P, P, R, E, E, R), 4, precision=fvna.FP32_PERT, tile_y=64,
                         dt_fixed=0.01)
    assert st["rc"] == fvna.OK and so["status"] == 0
    assert _rel(q, qo) <= 1e-5


def test_time_of_strong_fields():
    n = 200
    w = np.cos(0.05 * np.arange(n) + 0.3)
    w = w[:, None, None] * w[:, None] * w
    ms = []
    for amp in (1e-3, 0.02):
        q = wl.ambient3(n, n, n)
        q[0] += amp * w
        cfg = fvna.make_config(precision=fvna.FP32_PERT, beta=3.5, delta=1e-4, dx=1 / 40,
                               dt_fixed=0.005)
        s = fvna.Solver3(cfg, fvna.make_domain3(n, n, n), q)
        s.step_timed()
        ms.append(min(sum(s.step_timed()) for _ in range(9)))
        s.close()
    assert ms[1] <= 1.5 * ms[0], ms
