"""A not-a-number in c through one step with a uniform velocity along one axis.
In FP32 it is an interfacial donor on rows that are not whole 16-byte lanes and
reaches the cell downstream; on whole lanes it is an empty one and stays in its
cell.  In double a positive NaN is a full donor: the flux is the velocity's, and
the cell downstream takes the volume u dt."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("nx", [32, 33, 7])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_nan_donor(precision, nx, axis):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07463_gb300 import build, vof

    build.build()
    shape = (6, 5, nx)
    dt_ = torch.float64 if precision == 0 else torch.float32
    c = torch.zeros((1,) + shape, dtype=dt_, device=DEV)
    u = torch.zeros((3,) + shape, dtype=dt_, device=DEV)
    u[axis] = 1.0
    at = [2, 2, nx - 1 if axis == 0 else 3]  # along x across the periodic end
    c[(0, *at)] = float("nan")
    ctx = vof.Context(vof.make_config(nx, 5, 6, precision=precision), c, u)
    if precision == 2:
        ctx.vof_set_mlp(vof.mlp_weights_empty(DEV), 1e-3)
    ctx.vof_step(0.25, 1)
    got = c[0].cpu().numpy()
    ctx.close()
    down = list(at)
    down[2 - axis] = (down[2 - axis] + 1) % shape[2 - axis]
    want = np.zeros(shape)
    want[tuple(at)] = np.nan
    want[tuple(down)] = 0.25 if precision == 0 else (np.nan if nx % 4 else 0.0)
    assert np.array_equal(got, want, equal_nan=True)
