"""biot_autotune on levels that run as packed strips: the heights it returns are the
launch's, and no height changes a bit of the result, on ragged levels too."""
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


# several packed levels; a ragged one; rows that end a strip early; above an FP64 level
@pytest.mark.parametrize("nx, ny, levels", [(1024, 1024, 4), (640, 520, 3), (68, 1000, 3), (1024, 132, 3), (512, 512, 2)])
def test_tuned_packed_heights_keep_results(nx, ny, levels):
    params = dict(nx=nx, ny=ny, lx=1.0, ly=ny / nx, lam=1.0, mu=1.0, alpha=0.9, c0=0.3, kappa=0.1, dt=0.002, r=0.5,
                  levels=levels, K=3, gamma=0.75, tol=1e-30, ne_max=2, ne_fixed=2, precision=W.FP32)
    sides = W.top_load_sides(nx, W.step_load(nx))
    out = []
    for tune in (False, True):
        with biot.Solver(params, sides) as s:
            if tune:
                shapes = s.autotune()
                assert set(shapes) >= {f"L{levels - 1}_smooth", f"L{levels - 1}_restrict"}
                assert all(r >= 4 and r % 2 == 0 and ms > 0 for r, ms in shapes.values()), shapes
            s.step(2)
            out.append((s.read_u()[0], s.read_p()[0], s.read_stress()))
    for a, b in zip(*out):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
