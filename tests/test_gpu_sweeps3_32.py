"""Binary32 3D sweeps on pairs of lines against the 3D oracle (within 1e-5 of
the perturbation, the bar of tests/test_gpu_3d.py): the edges of the 60-cell
segments, of the 64-column tiles and of odd row counts, tiles of every height
class, and data for which the subsonic form with the series does not hold (a
flow beyond it along each axis, large amplitudes) next to data for which it does."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl
from test_gpu_3d import _rel, _run

pytestmark = pytest.mark.gpu

P, E, R = 0, 1, 2


@pytest.mark.parametrize("shape", [(59, 3, 5), (60, 5, 3), (61, 7, 9), (63, 4, 4), (64, 64, 3),
                                   (65, 5, 70), (1, 1, 1), (2, 33, 7), (125, 9, 11)])
@pytest.mark.parametrize("tile", [0, 4, 64])
def test_edges(shape, tile):
    nx, ny, nz = shape
    q0 = wl.random_smooth3(nx, ny, nz, 3e-3, seed=nx + 7 * nz)
    bc = (E,) * 6 if min(shape) < 3 else (P, P, R, E, E, R)
    q, st, qo, so = _run(nx, ny, nz, q0, bc, 5, precision=fvna.FP32_PERT, tile_y=tile)
    assert st["rc"] == fvna.OK and so["status"] == 0
    assert _rel(q, qo) <= 1e-5
    assert abs(st["smax"] - so["smax"]) <= 1e-6 * so["smax"]


@pytest.mark.parametrize("axis", [1, 2, 3])
@pytest.mark.parametrize("flow", [0.0, 0.75])
@pytest.mark.parametrize("limiter", [0, 2])
def test_beyond_the_subsonic_form(axis, flow, limiter):
    nx, ny, nz = 67, 21, 19
    q0 = wl.random_smooth3(nx, ny, nz, 3e-3, seed=axis)
    q0[axis] += flow
    q0[0, 4:9, 3:8, 10:20] += 0.03      # c^2 - 1 beyond the series there
    q, st, qo, so = _run(nx, ny, nz, q0, (P, P, P, P, P, P), 5, precision=fvna.FP32_PERT,
                         limiter=limiter, dt_fixed=0.01)
    assert st["rc"] == fvna.OK and so["status"] == 0
    assert _rel(q, qo) <= 1e-5
