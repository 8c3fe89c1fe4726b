"""Curvature on grids for which csrc/curvature.cu takes tiles of different
lengths (256 to 8192 cells, whole and partial last tiles), and on a field whose
cells are nearly all interfacial, so that a tile's list is full.  Against the
oracle at the gates of the other curvature tests: the same NaN pattern, 1e-11."""
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


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("shape", [(16, 16, 16), (31, 29, 33), (40, 52, 64), (60, 72, 96), (110, 90, 131), (150, 184, 190)])
def test_sizes(vof, shape, full):
    rng = np.random.default_rng(5)
    if full:  # a smooth field between 0 and 1 in every cell
        z, y, x = np.meshgrid(*(np.arange(n) / n for n in shape), indexing="ij")
        wave = np.sin(2 * np.pi * (2 * x + y) + 0.3) * np.sin(2 * np.pi * (y - z) + 0.7)
        c = 0.5 + 0.49 * wave
    else:
        c = synth.sphere_cell_fractions(shape, rng.random((2, 3)) * np.array(shape[::-1]), 0.2 * min(shape))
        c = np.clip(c, 0.0, 1.0)
    ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0], h=0.5), torch.from_numpy(c[None].copy()).to(DEV),
                      torch.zeros((3,) + shape, dtype=torch.float64, device=DEV))
    got = ctx.vof_curvature(0).cpu().numpy()
    ctx.close()
    want = O.curvature(c, 0.5)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.nanmax(np.abs(got - want), initial=0.0) <= 1e-11
