"""FP64 plane geometry (csrc/plic64.cuh) where its pieces meet: tiny and equal
normal components, fractions at the breaks of the volume, residues, and scales
far from one.

Tolerance: a volume is a quotient of sums of about ten rounded terms, none
cancelling by more than a factor of three, so a few 1e-16 on either side;
1e-14 as for the volumes of the other tests."""
import numpy as np
import pytest

import oracle as O

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


def breaks(a, b, c):
    """Volumes at the breaks of the lower half (x = a, b, min(c, a + b), S/2)."""
    S = a + b + c
    return [O.plic_volume([a, b, c], min(x, S / 2)) for x in (a, b, min(c, a + b), a + b, S / 2)]


NORMALS = [(0.2, 0.3, 0.5), (1 / 3, 1 / 3, 1 / 3), (0.25, 0.25, 0.5), (0.1, 0.45, 0.45), (1e-9, 0.4, 0.6),
           (1e-17, 0.5, 0.5), (1e-12, 1e-9, 1.0), (1e-25, 1e-24, 1.0), (1e-40, 1e-35, 1.0), (0.0, 0.3, 0.7),
           (0.0, 1e-20, 1.0), (0.0, 0.0, 1.0), (1e-300, 0.5, 0.5)]


@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e120])
@pytest.mark.parametrize("n", NORMALS)
def test_plane_constant_and_volume(vof, n, scale):
    cs = [v for q in breaks(*n) for v in (q * (1 - 1e-12), q, q * (1 + 1e-12), q - 1e-9, q + 1e-9)]
    cs += [0.5, 1e-3, 1e-8, 1e-16, 1e-40, 1 - 1e-3, 1 - 1e-8, 1 - 2e-16, np.nextafter(0.5, 1), 0.37, 0.81]
    cs = np.array([v for q in cs for v in (q, 1 - q) if 0 < v < 1])
    signs = np.array([[1, 1, 1], [-1, 1, 1], [1, -1, -1], [-1, -1, -1]])
    perms = np.array([[0, 1, 2], [2, 0, 1], [1, 2, 0]])
    m = np.concatenate([(np.array(n)[p] * s)[None].repeat(len(cs), 0) for p in perms for s in signs])
    c = np.tile(cs, len(perms) * len(signs))
    al = vof.vof_plic_alpha(torch.from_numpy(m * scale).to(DEV), torch.from_numpy(c).to(DEV))
    v = vof.vof_plic_volume(torch.from_numpy(m * scale).to(DEV), al).cpu().numpy()
    al = al.cpu().numpy() / scale
    assert np.isfinite(al).all() and np.isfinite(v).all()
    assert np.abs(v - c).max() <= 1e-14
    vo = np.array([O.plic_volume(m[t], al[t]) for t in range(len(c))])
    assert np.abs(vo - c).max() <= 1e-14



def pattern(kind, rng, shape=(7, 9, 11)):
    k, j, i = np.meshgrid(*[np.arange(s) for s in shape], indexing="ij")
    if kind == "diagonal":  # equal quotients of two or three axes
        c = np.clip((i + j + k - 13) * 0.25 + 0.5, 0.0, 1.0)
    elif kind == "axis":
        c = np.clip((k - 3) * 0.75 + 0.5, 0.0, 1.0)
    elif kind == "sixteenths":
        c = rng.integers(0, 17, shape) / 16.0
    elif kind == "mixed":
        c = np.where(rng.random(shape) < 0.3, 0.0, np.where(rng.random(shape) < 0.5, 1.0, rng.random(shape)))
    elif kind == "flat":  # differences far below the values
        c = 0.5 + 1e-6 * rng.standard_normal(shape)
    elif kind == "spread":  # sixteen decades
        c = 10.0 ** (-16.0 * rng.random(shape))
    elif kind == "rounding":  # whole numbers of 2^-56 among zeros, norms of 1 to a few units in the last place
        c = np.where(rng.random(shape) < 0.5, 0.0, rng.integers(1, 200, shape) * 2.0 ** -56)
    else:  # residues about the least norm at which the rule takes Youngs' normal
        c = 10.0 ** (-29.0 - 3.0 * rng.random(shape))
    return np.ascontiguousarray(c, dtype=np.float64)


# Tolerance: a sum of the rule has at most nine terms of weight up to 2 and
# 16 values' weight in all, so its rounding is below 8 * 16 * 2^-53 = 1.5e-14
# of the largest value; a component of the normal is off by that over the
# largest component (0.3 or more of the values in all but the flat field, whose
# differences are 1e-6 of them).  A centred-column normal has a component 1.
@pytest.mark.parametrize("kind, tol", [("diagonal", 1e-13), ("axis", 1e-13), ("sixteenths", 1e-13),
                                       ("mixed", 1e-13), ("flat", 1e-7), ("spread", 1e-13),
                                       ("residue", 1e-13), ("rounding", 1e-13)])
def test_normal_direction(vof, kind, tol):
    c = pattern(kind, np.random.default_rng(5))
    cfg = vof.make_config(c.shape[2], c.shape[1], c.shape[0])
    f = torch.from_numpy(c[None]).to(DEV)
    u = torch.zeros((3,) + c.shape, dtype=torch.float64, device=DEV)
    ctx = vof.Context(cfg, f, u)
    m = ctx.vof_normals(0).cpu().numpy()
    ctx.close()
    o = O.normals(c)
    assert np.isfinite(m).all()
    assert np.abs(m - o).max() <= tol
