"""Detaching a correction that was never attached changes nothing: the steps
after fvna_set_correction(ctx, NULL) are those of a context that never made
the call, in both splittings and precisions (a Strang step ends after its
second x1 sweep, not in the x2 sweep)."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, E, R = fvna.BC_PERIODIC, fvna.BC_EXTRAP, fvna.BC_REFLECT


@pytest.mark.parametrize("splitting", [fvna.SPLIT_GODUNOV, fvna.SPLIT_STRANG])
@pytest.mark.parametrize("precision", [fvna.FP64, fvna.FP32_PERT])
def test_detach_without_a_network(precision, splitting):
    nx, ny = 97, 66
    q0 = wl.random_smooth(nx, ny, 2e-3, seed=21)
    cfg = fvna.make_config(precision=precision, beta=3.5, delta=2e-3, dx=1.0 / 32, nu_w=0.9,
                           splitting=splitting, steps_per_graph=4)
    dom = fvna.make_domain(nx, ny, bc=(P, P, E, R))
    got = []
    for detach in (False, True):
        s = fvna.Solver(cfg, [dom], [q0])
        if detach:
            s.set_correction(None, 1.0, 1.0)
        n0 = s.launch_count()
        st = s.run(max_steps=8)
        s.step_timed()
        got.append((s.q(0), st["t"], st["nu_mean"], s.stats(0)["t"], s.launch_count() - n0))
        s.close()
    assert np.array_equal(got[0][0], got[1][0])
    assert got[0][1:] == got[1][1:]
