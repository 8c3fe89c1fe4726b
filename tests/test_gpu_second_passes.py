"""Kernels whose blocks take several tiles on large inputs (shared memory used
again from tile to tile).  A periodic field repeated along the axes gives the
repeated result: one tile per block on the small box, many on the large one.

The steps are bit for bit the same (a cell's arithmetic sees its neighbours
only).  The drop sums are FP64 atomics of at most 300 terms per drop, 300 * 2^-53
of a sum of positive terms: 1e-12, for the inertia about a centroid that itself
is so far off 1e-10.  The training gradient is compared with the FP64 backprop at
the gate of its other tests (BF16 operands: 1e-2 per tensor)."""
import numpy as np
import pytest

import oracle as O
from helpers import MLP_SPANS
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


def network(vof, seed):
    rng = np.random.default_rng(seed)
    p = np.zeros(O.MLP_NPARAM)
    p[0:2048].reshape(64, 32)[:, :27] = rng.normal(scale=(2 / 27) ** 0.5, size=(64, 27))
    p[2048:6144] = rng.normal(scale=(2 / 64) ** 0.5, size=4096)
    p[6144:7168].reshape(16, 64)[:3] = rng.normal(scale=(1 / 64) ** 0.5, size=(3, 64))
    p[7168:7296] = rng.normal(scale=0.1, size=128)
    q = torch.from_numpy(p.astype(np.float32))
    q[:7168] = q[:7168].bfloat16().float()
    return q, vof.vof_mlp_params_to_weights(q.to(DEV))


@pytest.mark.parametrize("shape,reps", [((32, 32, 32), (4, 4, 4)), ((30, 32, 31), (4, 4, 3))])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_steps(vof, precision, shape, reps):
    """Every cell interfacial: 50 thousand faces a sweep against some two million
    (a block of the flux kernels takes another tile from 311296 on, one of the
    network's from 77824)."""
    rng = np.random.default_rng(4)
    dt_ = torch.float64 if precision == 0 else torch.float32
    c0 = torch.from_numpy(rng.random((2,) + shape)).to(DEV, dt_)
    u0 = torch.from_numpy(rng.uniform(-1, 1, (3,) + shape)).to(DEV, dt_)
    out = []
    for r in ((1, 1, 1), reps):
        c, u = c0.repeat(1, *r).contiguous(), u0.repeat(1, *r).contiguous()
        nz, ny, nx = c.shape[1:]
        ctx = vof.Context(vof.make_config(nx, ny, nz, k_capacity=2, k_active=2, precision=precision), c, u)
        if precision == 2:
            ctx.vof_set_mlp(network(vof, 1)[1], 0.05)
        ctx.vof_step(0.3, 2)
        ctx.close()
        out.append(c)
    assert torch.equal(out[0].repeat(1, *reps), out[1])


@pytest.mark.parametrize("precision", [0, 1])
def test_drops(vof, precision):
    """512 x 256 x 256 (1.05 million words: tiles of several rounds and blocks of
    several tiles from 0.93 million on) from boxes of 32 cells a side."""
    n, reps = 32, (16, 8, 8)
    dt_ = torch.float64 if precision == 0 else torch.float32
    cen0 = np.array([[6.3, 7.2, 8.4], [20.6, 9.1, 11.7], [13.4, 26.2, 30.8], [29.7, 21.3, 16.2]])
    c0 = sum(synth.sphere_cell_fractions((n, n, n), p[None], r) for p, r in zip(cen0, (3.1, 3.6, 4.0, 2.7)))
    c0 = torch.from_numpy(np.clip(c0, 0, 1)).to(DEV, dt_)
    res = []
    for r in ((1, 1, 1), reps):
        c = c0.repeat(*r)[None].contiguous()
        nz, ny, nx = c.shape[1:]
        ctx = vof.Context(vof.make_config(nx, ny, nz, precision=precision), c,
                          torch.zeros((3, nz, ny, nx), dtype=dt_, device=DEV))
        lab, m = ctx.vof_label(0)
        vol, cen = ctx.vof_drop_table(0, lab, m)
        I, _ = ctx.vof_drop_shape(0, lab, m, cen)
        res.append((m, *(t.cpu().numpy() for t in (vol, cen, I)), ctx.vof_stats(reset=True)))
        ctx.close()
    (m0, vol0, cen0, I0, s0), (m1, vol1, cen1, I1, s1) = res
    assert m0 == 4 and m1 == 4 * 1024 and s1["n_drops"] == m1 and s1["events"] == m1
    want, _ = O.label(c0.cpu().numpy().astype(np.float64), tau=1e-6)
    vo, co = O.drop_table(c0.cpu().numpy().astype(np.float64), want, 4, 1.0)
    np.testing.assert_allclose(vol0, vo, rtol=1e-12)
    d = (cen1 % n)[:, None, :] - cen0[None]
    d -= n * np.round(d / n)
    which = np.abs(d).max(2).argmin(1)
    assert np.array_equal(np.bincount(which), [1024] * 4)
    assert np.abs(d[np.arange(m1), which]).max() <= 1e-10
    np.testing.assert_allclose(vol1, vol0[which], rtol=1e-12)
    np.testing.assert_allclose(I1, I0[which], rtol=1e-10, atol=1e-10 * np.abs(I0).max())
    assert s1["volume"] == pytest.approx(1024 * s0["volume"], rel=1e-12)
    np.testing.assert_array_equal(s1["hist_r"], 1024 * s0["hist_r"])
    np.testing.assert_allclose(s1["R"], s0["R"], rtol=1e-10)
    assert s1["chi_drops"] == m1


@pytest.mark.parametrize("n", [19457, 20000, 40001])
def test_gradient(vof, n):
    """More than one tile of 128 samples per block of a 152-SM device."""
    rng = np.random.default_rng(n)
    st = rng.random((n, 27)).astype(np.float32)
    tgt = rng.normal(size=(n, 3))
    tgt = (tgt / np.linalg.norm(tgt, axis=1, keepdims=True)).astype(np.float32)
    p, w = network(vof, 3)
    g, loss = vof.vof_mlp_grad(w, torch.from_numpy(st).to(DEV), torch.from_numpy(tgt).to(DEV))
    x, t = [], []
    for s, v in zip(st.astype(np.float64), tgt.astype(np.float64)):
        c, sign, perm = O.mlp_canon(s.reshape(3, 3, 3))
        x.append(c)
        t.append([sign[perm[q]] * v[perm[q]] for q in range(3)])
    lo, go = O.mlp_loss_grad(p.numpy().astype(np.float64), np.array(x), np.array(t))
    g = g.cpu().numpy().astype(np.float64)
    assert loss / n == pytest.approx(lo, rel=1e-3)
    for a, b in MLP_SPANS.values():
        assert np.linalg.norm(g[a:b] - go[a:b]) <= 1e-2 * np.linalg.norm(go[a:b])
