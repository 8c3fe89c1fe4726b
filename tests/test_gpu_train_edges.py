"""Training gradient at the edges of its 128-sample tiles and for a weight blob
that is not 16-byte aligned, against the FP64 backprop of the same BF16
forward (the gate of the other gradient test: 1e-2 relative per tensor; the
back-propagated values are rounded to BF16, 2^-9, at two layers)."""
import numpy as np
import pytest

import oracle as O
from helpers import MLP_SPANS

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


def network(seed):
    rng = np.random.default_rng(seed)
    p = np.zeros(O.MLP_NPARAM)
    p[0:2048].reshape(64, 32)[:, :27] = rng.normal(scale=(2 / 27) ** 0.5, size=(64, 27))
    p[2048:6144] = rng.normal(scale=(2 / 64) ** 0.5, size=4096)
    p[6144:7168].reshape(16, 64)[:3] = rng.normal(scale=(1 / 64) ** 0.5, size=(3, 64))
    p[7168:7296] = rng.normal(scale=0.1, size=128)
    p = p.astype(np.float32)
    q = torch.from_numpy(p)
    q[:7168] = q[:7168].bfloat16().float()
    return q


@pytest.mark.parametrize("n,shift", [(1, 0), (127, 0), (128, 4), (129, 0), (300, 8)])
def test_gradient(vof, n, shift):
    rng = np.random.default_rng(n)
    st = rng.random((n, 27)).astype(np.float32)
    tgt = rng.normal(size=(n, 3))
    tgt = (tgt / np.linalg.norm(tgt, axis=1, keepdims=True)).astype(np.float32)
    p = network(3)
    blob = vof.vof_mlp_params_to_weights(p.to(DEV))
    buf = torch.zeros(blob.numel() + 16, dtype=torch.uint8, device=DEV)
    w = buf[shift:shift + blob.numel()]
    w.copy_(blob)
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
