"""Binary64 sweeps against the oracle, bit for bit, where their forms meet: the
edges of the x1 segments and x2 tiles, and states inside, across and outside
the bounds of the fast form (momenta down to subnormals, amplitudes that leave
it, faces that are not subsonic, limiter ratios of nearly orthogonal waves)."""
import numpy as np
import pytest

from paper_1311_3004_gb300 import workloads as wl
from helpers import Case, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

P, E, R = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1311_3004_gb300 import build
    import oracle
    build.build()
    oracle.build()


@pytest.mark.parametrize("nx,ny", [(1, 1), (27, 3), (28, 7), (29, 29), (30, 1), (31, 33), (59, 5),
                                   (60, 16), (61, 2), (62, 17), (124, 9), (3, 200), (700, 3)])
@pytest.mark.parametrize("tile_x,tile_y", [(0, 0), (64, 9)])
def test_edges(nx, ny, tile_x, tile_y):
    bc = (E, E, E, E) if min(nx, ny) < 3 else (P, P, R, E)
    c = Case(nx, ny, wl.random_smooth(nx, ny, 2e-3, seed=nx + ny), bc=bc, delta=2e-3)
    qo, so = run_oracle(c, 6)
    qg, sg = run_gpu(c, 6, tile_x=tile_x, tile_y=tile_y)
    assert np.array_equal(qg, qo)
    assert sg["dt"] == so["dt"] and sg["smax"] == so["smax"]


def _states():
    n, m = 61, 40
    rng = np.random.default_rng(3)
    smooth = wl.random_smooth(n, m, 1e-3, seed=5)
    out = {}
    # momenta spread over the exponent range, down to subnormals and zeros
    q = smooth.copy()
    q[1:] = rng.choice([-1, 1], size=q[1:].shape) * 2.0 ** rng.uniform(-1074, -5, size=q[1:].shape)
    q[1:][rng.random(q[1:].shape) < 0.2] = 0.0
    out["scattered"] = q
    # each of the fast form's ranges by itself: down to 2^-400, and from there to the subnormals
    for name, lo, hi in (("small", -399, -5), ("smaller", -1070, -402)):
        q = smooth.copy()
        q[1:] = rng.choice([-1, 1], size=q[1:].shape) * 2.0 ** rng.uniform(lo, hi,
                                                                           size=q[1:].shape)
        q[1:][rng.random(q[1:].shape) < 0.1] = 0.0
        out[name] = q
        q = q.copy()
        q[0] = 1.0
        out[name + " at rest"] = q
    # a pulse at rest: exact zeros around it, then a numerical precursor that decays without end
    q = wl.centred_gaussian(n, m, 1e-3, 2.0)
    out["precursor"] = q
    # some rows inside the bounds, some outside
    q = smooth.copy()
    q[0, 10:14] += 0.08
    q[2, 25] = 0.07
    out["mixed"] = q
    q = wl.random_cells(n, m, 0.08, seed=9)   # larger ones leave the hyperbolic region
    out["large"] = q
    q = smooth.copy()
    q[1] += 0.75
    out["not subsonic"] = q
    # transverse momentum alone: normal waves zero, transverse ones not
    q = wl.ambient(n, m)
    q[2] = 1e-3 * rng.uniform(-1, 1, size=(m, n))
    out["shear"] = q
    q = smooth.copy()
    q[2] *= 1e-40
    out["thin transverse"] = q
    return out


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("name", list(_states()))
def test_states(name, limiter):
    q = _states()[name]
    _, m, n = q.shape
    c = Case(n, m, q, bc=(P, P, E, R), delta=1e-3, nu_w=0.4, limiter=limiter)
    steps = 60 if name == "precursor" else 8
    qo, so = run_oracle(c, steps)
    qg, sg = run_gpu(c, steps)
    assert so["status"] == 0 and sg["rc"] == 0
    assert np.array_equal(qg, qo)


@pytest.mark.parametrize("shape", [(28, 29, 57), (56, 27, 3), (1, 5, 30), (61, 2, 28)])
@pytest.mark.parametrize("amp,thin", [(1e-3, 1.0), (1e-3, 1e-60), (0.08, 1.0)])
def test_3d_edges(shape, amp, thin):
    """Edges of the 28-cell segments along each axis, momenta below the fast
    form's bounds, amplitudes beyond them."""
    from test_gpu_3d import _run
    nx, ny, nz = shape
    q0 = wl.random_smooth3(nx, ny, nz, amp, seed=nx + nz)
    q0[2] *= thin
    q0[3, :, ny // 2:] = 0.0
    q, st, qo, so = _run(nx, ny, nz, q0, (E, E, E, E, E, E) if 1 in shape or 2 in shape else
                         (P, P, R, E, E, R), 5)
    assert st["rc"] == 0 and so["status"] == 0
    assert np.array_equal(q, qo)
