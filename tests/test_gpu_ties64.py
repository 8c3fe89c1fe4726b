"""FP64 normals of whole fields near the ties of the Mixed-Youngs-Centred rule
and beside values that are not finite: vof_normals against the oracle (the
stencils of tests/test_plic64_normals.py through the GPU code; the tolerance is
derived there)."""
import numpy as np
import pytest

import oracle as O
from paper_2407_07463_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def vof():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07463_gb300 import build, vof

    build.build()
    vof.lib()
    return vof


def field(kind, shape, rng):
    if kind == "residues":
        return (rng.choice([0.0, 0.0, 0.0, 1.0, 0.5], shape) +
                rng.choice([0.0, 0.0, 0.0, 1e-17, -1e-17, 3e-18, 1e-16], shape))
    if kind == "layers":  # aligned with the grid: every candidate's sums cancel exactly
        return np.broadcast_to(rng.choice([0.0, 0.3, 1.0], (shape[0], 1, 1)), shape).copy()
    c = synth.sphere_cell_fractions(shape, np.array([[6.2, 7.1, 5.4]]), 3.7)
    at = tuple(rng.integers(n, size=6) for n in shape)
    c[at] = rng.choice([np.nan, np.inf, -np.inf], 6)
    return c


@pytest.mark.parametrize("kind", ["residues", "layers", "not finite"])
def test_normals_near_ties(vof, kind):
    shape = (11, 14, 12)
    c = field(kind, shape, np.random.default_rng(3))
    ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0]), torch.from_numpy(c[None].copy()).to(DEV),
                      torch.zeros((3,) + shape, dtype=torch.float64, device=DEV))
    got = ctx.vof_normals(0).cpu().numpy()
    ctx.close()
    pad = np.pad(c, 1, mode="wrap")
    for k, j, i in zip(*np.nonzero((c > 0) & (c < 1))):
        st = pad[k:k + 3, j:j + 3, i:i + 3].ravel()
        with np.errstate(all="ignore"):
            want, slope = O.myc(st), np.abs(O.youngs(st)).max()
            largest = np.abs(np.delete(st, 13)).max()
            tol = 1e-14 + (2.0 ** -39 * largest / slope if slope > 0 and np.isfinite(largest) else 0.0)
        assert np.array_equal(np.isnan(got[k, j, i]), np.isnan(want)), (k, j, i)
        assert np.nan_to_num(np.abs(got[k, j, i] - want)).max() <= min(tol, 1e-6), (k, j, i)
