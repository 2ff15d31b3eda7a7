"""FP64 levels from 128^2 cells on take 16 x 8 tiles, smaller ones 8 x 2: the first
size with the large tiles, the last without, and ragged ones, against the FP64 oracle
at the product's 1e-12 (relative L-infinity)."""
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


@pytest.mark.parametrize("nx, ny, levels, side", [(128, 128, 4, W.SYMMETRY), (128, 126, 2, W.SYMMETRY),
                                                  (140, 132, 3, W.PERIODIC), (18, 1012, 2, W.SYMMETRY)])
def test_fp64_tiles_match_oracle(nx, ny, levels, side):
    params = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=1.0, mu=1.0, alpha=0.9, c0=0.3, kappa=0.1, dt=0.002, r=0.5,
                  levels=levels, K=3, gamma=0.75, tol=1e-10, ne_max=50, ne_fixed=2, precision=W.FP64)
    sides = W.top_load_sides(nx, W.step_load(nx), side)
    with biot.Solver(params, sides) as s:
        assert s.step(2) == biot.OK
        got = dict(eta=s.read_u()[0], p=s.read_p()[0], sigma=s.read_stress())
    o = O.Oracle(params, sides)
    assert o.step(2) == 0
    ref = dict(eta=o.read_u()[0], p=o.read_p()[0], sigma=o.read_stress())
    o.close()
    for k in ref:
        assert np.abs(got[k] - ref[k]).max() <= TOL64 * np.abs(ref[k]).max(), k
