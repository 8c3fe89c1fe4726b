"""A context's and a batch's sweep buffers are cleared when they are created
(csrc/boxes.cuh, k_clear_sp): whatever the workspace held (not-a-number bits,
or bits that read as ordinary fractions), the steps match the FP64 oracle with
the gates of the other step tests.  Whole-word, ragged and short rows, fields
that are not active, boxes of different sizes in one batch."""
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


@pytest.fixture(params=[0x3F, 0xFF])
def held(request, monkeypatch):
    """Every workspace (a byte tensor) holds this byte throughout."""
    empty = torch.empty

    def filled(*a, **k):
        t = empty(*a, **k)
        return t.fill_(request.param) if t.dtype == torch.uint8 else t

    monkeypatch.setattr(torch, "empty", filled)


def box(shape, K, active, seed):
    rng = np.random.default_rng(seed)
    c = np.zeros((K,) + shape)
    for k in range(active):
        cen = rng.random((1, 3)) * np.array([shape[2], shape[1], shape[0]])
        c[k] = synth.sphere_cell_fractions(shape, cen, 0.4 * min(shape))
    u = synth.solenoidal_velocity(shape, 4, 0.5, 0.6, seed)
    return c, u, synth.dt_for_cfl(u, 0.4)


@pytest.mark.parametrize("shape,K,active", [((4, 5, 3), 1, 1), ((5, 6, 33), 4, 3), ((6, 7, 64), 16, 16), ((40, 36, 48), 5, 2)])
@pytest.mark.parametrize("precision", [0, 1])
def test_context_on_used_workspace(vof, held, shape, K, active, precision):
    dt_ = torch.float64 if precision == 0 else torch.float32
    c, u, dt = box(shape, K, active, K)
    c_d = torch.from_numpy(c).to(DEV, dt_).contiguous()
    u_d = torch.from_numpy(u).to(DEV, dt_).contiguous()
    ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=active, precision=precision,
                                      recolour=0), c_d, u_d)
    want, _ = O.advect(c_d.cpu().numpy().astype(np.float64)[:active], u_d.cpu().numpy().astype(np.float64), dt, 1.0, 3)
    ctx.vof_step(dt, 3)
    got = c_d.cpu().numpy().astype(np.float64)
    assert np.abs(got[:active] - want).max() <= (1e-12 if precision == 0 else 1e-5)
    assert not got[active:].any()
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_on_used_workspace(vof, held, precision):
    dt_ = torch.float64 if precision == 0 else torch.float32
    data = [box((8, 8, 32), 2, 2, 1), box((5, 6, 36), 3, 1, 2), box((6, 5, 100), 8, 8, 3)]
    active = [2, 1, 8]
    cs = [torch.from_numpy(c).to(DEV, dt_).contiguous() for c, _, _ in data]
    us = [torch.from_numpy(u).to(DEV, dt_).contiguous() for _, u, _ in data]
    want = [O.advect(c.cpu().numpy().astype(np.float64)[:a], u.cpu().numpy().astype(np.float64), dt, 1.0, 3)[0]
            for c, u, a, (_, _, dt) in zip(cs, us, active, data)]
    B = vof.Batch(list(zip(cs, us, [dt for _, _, dt in data])), precision=precision, k_active=active)
    B.step(3)
    B.report()
    for c, w, a in zip(cs, want, active):
        got = c.cpu().numpy().astype(np.float64)
        assert np.abs(got[:a] - w).max() <= (1e-12 if precision == 0 else 1e-5)
        assert not got[a:].any()
    B.close()
