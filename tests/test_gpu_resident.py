"""The coarse-grid correction of the small levels as one cluster launch
(csrc/sweep_resident.cuh) at the edges of its range: level shapes that divide
unevenly among the cluster's blocks, levels one cell wide or high, periodic sides,
the largest levels it takes and the first it leaves to separate launches.

FP64 against the FP64 oracle at the product's 1e-12 (relative L-infinity).  FP32: a
batch takes the cluster launch from another level down than a single instance, and
every form of a sweep rounds alike, so the two agree bitwise.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2409_11382_gb300 import biot, workloads as W  # noqa: E402

TOL64 = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_11382_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)


def problem(nx, ny, levels, precision, periodic=False, **kw):
    p = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=1.0, mu=1.0, alpha=0.9, c0=0.3, kappa=0.1, dt=0.01, r=0.5,
             levels=levels, K=3, gamma=0.75, tol=1e-10, ne_max=60, ne_fixed=2, precision=precision, **kw)
    load = 1.0 + np.sin(np.linspace(0.0, 3.0, 2 * nx + 1))
    return p, W.top_load_sides(nx, load, W.PERIODIC if periodic else W.SYMMETRY)


def read(s):
    return dict(eta=s.read_u()[0], p=s.read_p()[0], sigma=s.read_stress())


# coarse shapes 22 x 18 / 11 x 9 (uneven slabs), 2 x 40 / 1 x 20 and 40 x 2 / 20 x 1
# (thin), 32^2 and 40 x 52 (the FP64 bound, above it), one-cell coarsest
FP64 = [(44, 36, 3, False, {}), (4, 80, 3, True, {}), (80, 4, 3, False, {}), (64, 64, 4, True, {}), (80, 104, 4, False, {}),
        (16, 16, 5, False, {}), (44, 36, 3, False, dict(cycle=biot.CYCLE_W)), (48, 32, 4, True, dict(cycle=biot.CYCLE_F)),
        (44, 36, 3, False, dict(ne_fixed=0, tol=1e-9))]


@pytest.mark.parametrize("case", range(len(FP64)))
def test_fp64_matches_oracle(case):
    nx, ny, levels, periodic, kw = FP64[case]
    params, sides = problem(nx, ny, levels, W.FP64, periodic)
    params.update(kw)
    with biot.Solver(params, sides) as s:
        s.step(3)
        got, ne = read(s), s.stats()["total_cycles"]
    o = O.Oracle(params, sides)
    o.step(3)
    ref = dict(eta=o.read_u()[0], p=o.read_p()[0], sigma=o.read_stress())
    assert ne == o.stats()["total_cycles"]
    o.close()
    for k in ref:
        assert np.abs(got[k] - ref[k]).max() <= TOL64 * np.abs(ref[k]).max(), k


# 64^2 and 56 x 72 coarse levels (the FP32 bound and just inside), 66 x 64 (above), thin
FP32 = [(128, 128, 5, False), (112, 144, 5, True), (132, 128, 3, False), (4, 256, 3, True), (256, 4, 3, False), (88, 56, 4, False)]


@pytest.mark.parametrize("options", [0, biot.OPT_COARSEST_STORAGE, biot.OPT_SEGMENTS])
def test_fp32_batch_equals_single(options):
    probs = [problem(nx, ny, levels, W.FP32, per, options=options) for nx, ny, levels, per in FP32]
    with biot.Batch(probs) as b:
        b.step(3)
        got = [read(b[i]) for i in range(len(probs))]
    for (p, sides), g in zip(probs, got):
        with biot.Solver(p, sides) as s:
            s.step(3)
            ref = read(s)
        for k in ref:
            assert np.array_equal(g[k], ref[k]), (p["nx"], p["ny"], k)
