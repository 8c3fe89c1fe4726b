"""The sweep passes' maps of non-zero words (csrc/boxes.cuh): fields that
change completely between calls (stale sweep buffers), whole-word and ragged
rows, one to sixteen fields, rows shorter than a word, buffers that are not
16-byte aligned.  Against the FP64 oracle: 1e-12 per cell in double, 1e-5 in
mixed precision (the gates of the other step tests), and the occupancy that
Step 1 sees."""
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


def field_set(shape, K, seed):
    """K fields: a sphere each, some empty, one full, one of residues only."""
    rng = np.random.default_rng(seed)
    c = np.zeros((K,) + shape)
    for k in range(K):
        kind = (k + seed) % 4
        if kind == 1 and K > 2:
            continue
        r = min(3.3, 0.45 * min(shape))
        cen = rng.random((1, 3)) * np.array([shape[2], shape[1], shape[0]])
        c[k] = synth.sphere_cell_fractions(shape, cen, r)
        if kind == 2 and K > 3:
            c[k] = 1.0
    return c


def unaligned(t):
    """A copy of t one element past a 16-byte boundary."""
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=DEV)
    out = flat[1:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("shape,K", [((6, 5, 32), 1), ((9, 8, 64), 16), ((7, 6, 100), 3), ((6, 7, 33), 4),
                                     ((5, 6, 31), 2), ((4, 5, 4), 2), ((5, 4, 3), 1), ((3, 4, 130), 5)])
@pytest.mark.parametrize("precision,shift", [(0, False), (1, False), (1, True)])
def test_fields_replaced_between_calls(vof, shape, K, precision, shift):
    dt_ = torch.float64 if precision == 0 else torch.float32
    tol = 1e-12 if precision == 0 else 1e-5
    u = synth.solenoidal_velocity(shape, 4, 0.5, 0.6, 3)
    u[0] -= 0.4
    dt = synth.dt_for_cfl(u, 0.4)
    u_d = torch.from_numpy(u).to(DEV, dt_).contiguous()
    c_d = torch.zeros((K,) + shape, dtype=dt_, device=DEV)
    if shift:
        u_d, c_d = unaligned(u_d), unaligned(c_d)
    cfg = vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=K, precision=precision, recolour=0)
    ctx = vof.Context(cfg, c_d, u_d)
    u64 = u_d.cpu().numpy().astype(np.float64)
    step = 0
    for call in range(3):
        c = field_set(shape, K, 10 * call + 1)
        c_d.copy_(torch.from_numpy(c).to(DEV, dt_))
        n = 1 + call % 2
        ctx.vof_step(dt, n)
        want, _ = O.advect(c_d.new_tensor(c).cpu().numpy().astype(np.float64), u64, dt, 1.0, n, first_step=step)
        step += n
        got = c_d.cpu().numpy().astype(np.float64)
        assert np.abs(got - want).max() <= tol
    ctx.close()


def test_recolour_after_replaced_fields(vof):
    """Steps 1-4 inside a call see the occupancy of the fields as replaced:
    the moves equal those of a fresh context."""
    shape, K = (40, 40, 64), 3
    cen = synth.rsa_centres(shape, 4.0, 14, 5)
    rng = np.random.default_rng(2)
    a = synth.coloured_fields(shape, cen, 4.0, rng.integers(0, 2, 14), K)
    b = synth.coloured_fields(shape, cen, 4.0, rng.integers(0, 2, 14), K)
    u = synth.solenoidal_velocity(shape, 4, 0.3, 0.5, 4)
    dt = synth.dt_for_cfl(u, 0.3)
    out = []
    for first in (a, b):
        c_d = torch.from_numpy(first.copy()).to(DEV)
        ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=K, recolour=1), c_d,
                          torch.from_numpy(u).to(DEV))
        if first is a:  # three steps of other fields first: the same rotation comes again
            ctx.vof_step(dt, 3)
            c_d.copy_(torch.from_numpy(b))
        rep = ctx.vof_step(dt, 3)
        out.append((c_d.cpu().numpy(), rep["n_moved"]))
        ctx.close()
    assert out[0][1] == out[1][1] and out[0][1] > 0
    assert np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("band", [0.0, 1e-3, 0.4999])
@pytest.mark.parametrize("shape,K", [((3, 4, 5), 1), ((9, 8, 64), 3)])
def test_refined_faces(vof, shape, K, band):
    """The faces queued for the FP64 step of the mixed path: none, a few, nearly
    all, with less than one block of faces and with a part-filled last block."""
    u = synth.solenoidal_velocity(shape, 4, 0.5, 0.6, 3)
    dt = synth.dt_for_cfl(u, 0.4)
    c_d = torch.from_numpy(field_set(shape, K, 2)).to(DEV, torch.float32).contiguous()
    u_d = torch.from_numpy(u).to(DEV, torch.float32).contiguous()
    want, _ = O.advect(c_d.cpu().numpy().astype(np.float64), u_d.cpu().numpy().astype(np.float64), dt, 1.0, 1)
    cfg = vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=K, precision=1, recolour=0,
                          alpha_fp64_band=band)
    ctx = vof.Context(cfg, c_d, u_d)
    ctx.vof_step(dt, 1)
    assert np.abs(c_d.cpu().numpy() - want).max() <= 1e-5
    ctx.close()


@pytest.mark.parametrize("nx", [32, 33, 64, 70])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_words_entered_along_x(vof, nx, sign):
    """Interfacial cells at the ends of words, carried along x into words that
    hold nothing (also across the wrap, into a last word of one and six cells)."""
    shape, K = (4, 4, nx), 3
    c = np.zeros((K,) + shape)
    rng = np.random.default_rng(nx)
    for k, i in enumerate((0, 31, nx - 1)):
        c[k, 1:3, 1:3, i] = 0.3 + 0.6 * rng.random((2, 2))
    u = np.zeros((3,) + shape)
    u[0], u[1], u[2] = sign, 0.31, -0.23
    c_d = torch.from_numpy(c).to(DEV)
    ctx = vof.Context(vof.make_config(nx, 4, 4, k_capacity=K, k_active=K, recolour=0), c_d,
                      torch.from_numpy(u).to(DEV))
    ctx.vof_step(0.4, 3)
    want, _ = O.advect(c, u, 0.4, 1.0, 3)
    assert np.abs(c_d.cpu().numpy() - want).max() <= 1e-12
    ctx.close()
