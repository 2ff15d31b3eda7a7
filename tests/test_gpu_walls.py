"""Every meeting of wall types at a corner, and cells that touch two facing walls.

The wall form of a sweep takes its sources and signs from a table indexed by the
walls a cell touches (csrc/wall_table.cuh).  Each arrangement of wall types below
puts different pairs at the corners; together they cover all nine ordered pairs of
a side wall and a top/bottom wall.  The narrow grids have a coarsest level one
cell wide or high.  FP64 against the FP64 oracle at the product's 1e-12 (relative
L-infinity), fixed V-cycles, with and without the history of the fullway
bounce-back (several sweeps per level).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2409_11382_gb300 import biot, workloads as W  # noqa: E402

S, D, N = W.SYMMETRY, W.DIRICHLET, W.NEUMANN
# (bottom, right, top, left) displacement types, one DIRICHLET side at least
WALLS = [(D, S, N, S), (D, N, N, D), (S, D, S, N), (N, S, D, D), (D, D, D, N), (N, N, S, D), (D, D, S, S)]
GRIDS = [(24, 20, 3), (8, 4, 3), (4, 8, 3)]
TOL64 = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_11382_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


def problem(walls, nx, ny, levels, seed=1):
    rng = np.random.default_rng(seed)
    sides = []
    for i, t in enumerate(walls):
        n = nx if i in (W.BOTTOM, W.TOP) else ny
        side = dict(eta_type=t, p_type={S: S, D: N, N: D}[t])
        if t == D:
            side["eta_profile"] = 0.01 * rng.normal(size=(2, 2 * n + 1))
        elif t == N:
            side["eta_profile"] = rng.normal(size=(2, 2 * n + 1))
            side["p_profile"] = 0.1 * rng.normal(size=2 * n + 1)
        sides.append(side)
    params = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=0.8, mu=0.6, alpha=0.9, c0=0.5, kappa=0.3, dt=0.02, r=0.5,
                  levels=levels, K=3, gamma=0.75, tol=1e-10, ne_max=50, ne_fixed=3, precision=W.FP64)
    return params, sides


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("walls", WALLS)
def test_wall_corners_match_oracle(walls, grid):
    params, sides = problem(walls, *grid)
    with biot.Solver(params, sides) as s:
        assert s.step(3) == biot.OK
        got = dict(eta=s.read_u()[0], p=s.read_p()[0], sigma=s.read_stress())
    o = O.Oracle(params, sides)
    assert o.step(3) == 0
    ref = dict(eta=o.read_u()[0], p=o.read_p()[0], sigma=o.read_stress())
    o.close()
    for k in ref:
        assert np.abs(got[k] - ref[k]).max() <= TOL64 * np.abs(ref[k]).max(), k
