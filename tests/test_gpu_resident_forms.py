"""The cluster launch of the small levels (csrc/sweep_resident.cuh) against one launch
per sweep, bitwise.

The solve at t = 0 runs one launch per sweep; with BIOT_OPT_SEGMENTS it takes the
cluster launch for every coarse level without double-float first moments: all of them
in FP64, and in FP32 with BIOT_OPT_COARSE_LO_OFF.  Nothing else differs between the two
solves, so they pin the cluster launch, levels of one CTA and of one cell included, to
the separate sweeps.  Covered: FP32 levels over an FP64 or an FP32 coarsest level and
FP64 ones; roller, periodic, displacement and traction walls at the sides; V, W and F
cycles and the full-multigrid start; fixed counts and tolerance mode (ghost moments); the
largest level of each precision (64^2 in FP32, 2048 cells in FP64) and a 66 x 64 one.
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
    return [dict(eta_type=W.DIRICHLET, p_type=W.NEUMANN),
            dict(eta_type=W.NEUMANN, p_type=W.DIRICHLET, eta_profile=np.stack([wall, -wall]), p_profile=wall),
            dict(eta_type=W.NEUMANN, p_type=W.DIRICHLET, eta_profile=np.stack([0.2 * load, -load])),
            dict(eta_type=W.DIRICHLET, p_type=W.NEUMANN, eta_profile=np.stack([wall, wall]))]


def solve(params, sides):
    with biot.Solver(params, sides) as s:
        out = (s.read_u()[0], s.read_p()[0], s.read_stress())  # the solve at t = 0
        st = s.stats()
        return out, st["total_cycles"], st["kernel_launches"]


GRIDS = [(16, 16, 5), (32, 32, 4), (64, 64, 5), (128, 128, 6), (128, 64, 4), (24, 20, 3), (4, 96, 3), (96, 4, 3), (132, 128, 3)]
FORMS = [dict(precision=W.FP32, options=biot.OPT_COARSE_LO_OFF),
         dict(precision=W.FP32, options=biot.OPT_COARSE_LO_OFF | biot.OPT_COARSEST_STORAGE),
         dict(precision=W.FP64, options=0)]
CYCLES = [dict(), dict(cycle=biot.CYCLE_W), dict(cycle=biot.CYCLE_F), dict(fmg=1),
          dict(ne_fixed=0, ne_max=4, tol=1e-30), dict(ne_fixed=0, ne_max=3, tol=1e-30, cycle=biot.CYCLE_F)]


@pytest.mark.parametrize("walls", ["roller", "periodic", "mixed"])
@pytest.mark.parametrize("form", range(len(FORMS)))
@pytest.mark.parametrize("cycle", range(len(CYCLES)))
def test_cluster_launch_equals_separate_sweeps(cycle, form, walls):
    for nx, ny, levels in GRIDS:
        params = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=0.8, mu=0.6, alpha=0.9, c0=0.5, kappa=0.3, dt=0.02, r=0.5,
                      levels=levels, K=3, gamma=0.75, tol=1e-10, ne_max=50, ne_fixed=3)
        params.update(FORMS[form])
        params.update(CYCLES[cycle])
        sides = sides_of(walls, nx, ny)
        sep, ne_sep, l_sep = solve(params, sides)
        res, ne_res, l_res = solve(dict(params, options=params["options"] | biot.OPT_SEGMENTS), sides)
        assert ne_sep == ne_res and l_res < l_sep, (nx, ny)
        for a, b in zip(sep, res):
            assert np.abs(a).max() > 0 and np.array_equal(a, b), (nx, ny)
