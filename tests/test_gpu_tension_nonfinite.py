"""The surface-tension source beside values of c that are not finite: a face
without a curvature adds gamma * 0 * (c - c'), which is not a number there, so
that a field that has blown up shows in the force.  Against the oracle's source of
vof_curvature's curvatures: the same NaN and infinite faces, the others within
what a curvature loses by differencing sums of seven cells (two second and a
mixed difference over h^2: 16 ulps of 7 times 0.7 / h^2 = 314 ulps, 7e-14 in
double, 4e-5 in FP32)."""
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


def context(vof, c, precision, h):
    dt_ = torch.float64 if precision == 0 else torch.float32
    shape = c.shape[1:]
    return vof.Context(vof.make_config(shape[2], shape[1], shape[0], k_capacity=len(c), k_active=len(c), h=h,
                                       precision=precision), torch.from_numpy(c).to(DEV, dt_).contiguous(),
                       torch.zeros((3,) + shape, dtype=dt_, device=DEV))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("nx", [32, 31])
@pytest.mark.parametrize("precision", [0, 1])
def test_source_beside_a_value_that_is_not_finite(vof, precision, nx, value):
    shape, h = (18, 20, nx), 0.5
    c = np.stack([synth.sphere_cell_fractions(shape, np.array([p]), 4.6) for p in ((8.3, 9.1, 7.7), (20.2, 11.4, 9.5))])
    c = c.astype(np.float32).astype(np.float64)
    for f, k, j, i in ((0, 0, 0, 0), (0, 5, 19, nx - 1), (1, 17, 10, 16), (1, 9, 11, 20)):  # ends, beside and inside a drop
        c[f, k, j, i] = value
    ctx = context(vof, c, precision, h)
    kap = np.stack([ctx.vof_curvature(q).cpu().numpy().astype(np.float64) for q in range(2)])
    with np.errstate(all="ignore"):
        want = O.surface_tension(c, kap, 0.7, h)
    got = ctx.vof_surface_tension(0.7).cpu().numpy().astype(np.float64)
    ctx.close()
    # infinite faces (a curvature times an infinite difference) have their sign
    assert np.isnan(want).any()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isinf(got), np.isinf(want)) and np.array_equal(got[np.isinf(got)], want[np.isinf(want)])
    ok = np.isfinite(want)
    assert np.abs(got[ok] - want[ok]).max() <= (7e-14 if precision == 0 else 4e-5)


def test_source_with_a_coefficient_beyond_fp32(vof):
    c = synth.sphere_cell_fractions((12, 12, 32), np.array([[8.3, 6.1, 5.7]]), 3.6)[None]
    ctx = context(vof, c, 1, 1.0)
    assert torch.isnan(ctx.vof_surface_tension(1e300)[:, 0, 0, 20]).all()  # inf * 0, as on every other face
    ctx.close()
