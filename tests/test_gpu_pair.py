"""The packed two-cells-per-lane sweep of large FP32 levels (csrc/sweep_pair.cuh) at
the edges of its range.

With a fixed number of V-cycles a large FP32 level runs the packed sweep; in
tolerance mode, which keeps the ghost moments, it runs the general strips.  With an
unreachable tolerance and the same V-cycle cap both make the same iterates, and every
form of a sweep rounds alike, so the two agree bitwise.  Covered: a last strip of 60,
56 and 4 columns, row counts that end a strip early, the smallest level it takes and
one just below, every wall type, periodic sides, a body force and a source, a row
length it refuses (not a multiple of four), and an FP64 level below a packed one.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2409_11382_gb300 import biot, workloads as W  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_11382_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


def sides_of(kind, nx, ny):
    load = W.step_load(nx)
    if kind != "mixed":
        return W.top_load_sides(nx, load, W.PERIODIC if kind == "periodic" else W.SYMMETRY)
    wall = 0.01 * np.sin(np.linspace(0.0, 3.0, 2 * ny + 1))
    top = np.stack([0.2 * load, -load])
    return [dict(eta_type=W.DIRICHLET, p_type=W.NEUMANN),
            dict(eta_type=W.NEUMANN, p_type=W.DIRICHLET, p_profile=wall),
            dict(eta_type=W.NEUMANN, p_type=W.DIRICHLET, eta_profile=top),
            dict(eta_type=W.DIRICHLET, p_type=W.NEUMANN, eta_profile=np.stack([wall, wall]))]


CASES = [(64, 1032, 3, "roller", 0), (68, 1000, 3, "mixed", 0), (120, 552, 2, "periodic", 0), (1024, 64, 3, "mixed", 0),
         (256, 256, 4, "roller", 0), (252, 260, 2, "periodic", 0), (248, 264, 3, "mixed", 0), (254, 264, 2, "mixed", 0),
         (512, 516, 3, "mixed", 0), (512, 512, 2, "roller", biot.OPT_COARSEST_STORAGE), (640, 520, 3, "mixed", 1 << 30)]


@pytest.mark.parametrize("nx, ny, levels, walls, options", CASES)
def test_packed_sweep_equals_general_strips(nx, ny, levels, walls, options):
    sources = options == 1 << 30
    params = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=1.0, mu=1.0, alpha=0.9, c0=0.3, kappa=0.1, dt=0.002, r=0.5,
                  levels=levels, K=3, gamma=0.75, tol=1e-30, ne_max=2, ne_fixed=2, precision=W.FP32,
                  options=0 if sources else options)
    out = []
    for fixed in (2, 0):
        with biot.Solver(dict(params, ne_fixed=fixed), sides_of(walls, nx, ny)) as s:
            if sources:
                rng = np.random.default_rng(4)
                s.set_sources(rng.normal(size=(2, ny, nx)), rng.normal(size=(ny, nx)))
            s.step(3)
            out.append((s.read_u()[0], s.read_p()[0], s.read_stress(), s.stats()["total_cycles"]))
    assert out[0][3] == out[1][3] == 8
    for a, b in zip(out[0][:3], out[1][:3]):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
