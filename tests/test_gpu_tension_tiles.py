"""Curvature and surface tension where the tiled kernels (csrc/curvature.cu)
have edges: partial tiles, rows that are not whole 16-byte lanes, unaligned
buffers, axes shorter than the seven cells of a column, several fields.
Against the oracle at the gates of the other curvature tests: the same NaN
pattern, 1e-11 in double; on these small grids every selection is far from a
tie in double."""
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


@pytest.mark.parametrize("shape,K", [((24, 20, 28), 1), ((30, 26, 33), 3), ((17, 40, 36), 2), ((9, 9, 5), 2),
                                     ((5, 12, 14), 1)])
@pytest.mark.parametrize("shift", [False, True])
def test_tension(vof, shape, K, shift):
    rng = np.random.default_rng(7)
    r = 0.42 * min(shape)
    c = np.stack([np.clip(synth.sphere_cell_fractions(shape, rng.random((1, 3)) * np.array(shape[::-1]), r), 0, 1)
                  for _ in range(K)])
    buf = torch.empty(c.size + 1, dtype=torch.float64, device=DEV)
    c_d = buf[int(shift):int(shift) + c.size].view(c.shape)
    c_d.copy_(torch.from_numpy(c))
    ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=K, h=0.5), c_d,
                      torch.zeros((3,) + shape, dtype=torch.float64, device=DEV))
    kap = np.stack([O.curvature(c[k], 0.5) for k in range(K)])
    for k in range(K):
        got = ctx.vof_curvature(k).cpu().numpy()
        assert np.array_equal(np.isnan(got), np.isnan(kap[k]))
        assert np.nanmax(np.abs(got - kap[k]), initial=0.0) <= 1e-11
    out = torch.empty(3 * c[0].size + 1, dtype=torch.float64, device=DEV)[int(shift):][:3 * c[0].size].view((3,) + shape)
    f = ctx.vof_surface_tension(0.7, out=out).cpu().numpy()
    want = O.surface_tension(c, kap, 0.7, 0.5)
    assert np.abs(f - want).max() <= 1e-11
    ctx.close()
