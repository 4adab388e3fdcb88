"""The binary32 3D sweeps take lines in pairs; a cell that is not a number in
one line of a pair leaves the other line as it is without it: the line next to
it holds data beyond the series form, which has to be seen all the same."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import fvna
from paper_1311_3004_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("substep", [1, 2, 4])
@pytest.mark.parametrize("first", [0, 1])
def test_the_other_line_of_the_pair(substep, first):
    """first: which line of the pair holds the number that is none."""
    n = 20
    # (x1, x2) position of the two lines; x1 lines pair by rows, the others by columns
    bad, good = ((10, 8 + first), (10, 9 - first)) if substep == 1 else \
                ((8 + first, 10), (9 - first, 10))
    q0 = wl.ambient3(n, n, n)
    q0[0, 10, good[1], good[0]] += 0.06        # c^2 - 1 = 0.15 at its faces
    got = []
    for nan in (False, True):
        q = q0.copy()
        if nan:
            q[{1: 1, 2: 2, 4: 3}[substep], 10, bad[1], bad[0]] = np.nan   # normal momentum
        cfg = fvna.make_config(precision=fvna.FP32_PERT, beta=3.5, dx=0.1, dt_fixed=0.03)
        s = fvna.Solver3(cfg, fvna.make_domain3(n, n, n, substeps=substep), q)
        st = s.run(max_steps=1, check=False)
        got.append(s.q())
        s.close()
        assert st["steps"] == 1
        assert st["rc"] == (fvna.ERR_NAN if nan else fvna.OK)
    a, b = got
    line = (slice(None), 10, good[1], slice(None)) if substep == 1 else \
           (slice(None), 10, slice(None), good[0]) if substep == 2 else \
           (slice(None), slice(None), good[1], good[0])
    assert np.max(np.abs(a[line] - q0[line])) > 1e-3
    assert np.array_equal(a[line], b[line])
