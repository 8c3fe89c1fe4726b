"""Drop tables by runs and the two-stage nearest-neighbour search (csrc/post.cu)
where they can go wrong, against the FP64 oracle: runs across words and
periodic ends, drops longer than half a period, values the exact integer sums
do not hold, several fields in one chain, rows of any length; tiles of the
pair search, ties, more candidates than a warp's list holds, coordinates
outside the box.

Tolerances: sums of at most a few 1e4 terms of one sign in double, 1e-16 each,
so 1e-12 relative; centroids 1e-11 absolute on boxes of up to 100 cells."""
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


def scene(shape, seed):
    """Spheres, a bar along x longer than half a period, single residue cells."""
    rng = np.random.default_rng(seed)
    n = max(1, int(np.prod(shape) / 3000))
    c = np.clip(synth.sphere_cell_fractions(shape, rng.random((n, 3)) * np.array(shape[::-1]), 3.2), 0, 1)
    c[0, 0, : max(1, (3 * shape[2]) // 4)] = 0.7
    c[0, 0, -1] = 0.4
    free = np.argwhere(c == 0)
    for q in free[rng.choice(len(free), min(6, len(free)), replace=False)]:
        c[tuple(q)] = 10.0 ** rng.uniform(-9, -5)
    return c


@pytest.mark.parametrize("shape", [(12, 10, 64), (9, 11, 100), (14, 12, 37), (8, 9, 32), (6, 5, 20)])
@pytest.mark.parametrize("precision,tau,conn", [(0, 1e-6, 6), (1, 1e-6, 6), (1, 0.0, 26), (0, 0.0, 26)])
def test_drop_tables(vof, shape, precision, tau, conn):
    dt_ = torch.float64 if precision == 0 else torch.float32
    K = 3
    c = np.stack([scene(shape, 5 * k + 1) for k in range(K)])
    c[2] *= 1.3 if precision == 1 else 1.0  # values above one
    c_d = torch.from_numpy(c).to(DEV, dt_).contiguous()
    c = c_d.cpu().numpy().astype(np.float64)
    h = 0.5
    cfg = vof.make_config(shape[2], shape[1], shape[0], k_capacity=K, k_active=K, precision=precision, tag_tau=tau,
                          connectivity=conn, h=h)
    ctx = vof.Context(cfg, c_d, torch.zeros((3,) + shape, dtype=dt_, device=DEV))
    st = ctx.vof_stats(reset=True)
    total, drops = 0.0, 0
    for f in range(K):
        lab, n = ctx.vof_label(f)
        lo, no = O.label(c[f], tau=tau, connectivity=conn)
        assert n == no and np.array_equal(lab.cpu().numpy(), lo)
        vol, cen = ctx.vof_drop_table(f, lab, n)
        vo, co = O.drop_table(c[f], lo, no, h)
        L = np.array(shape[::-1]) * h
        np.testing.assert_allclose(vol.cpu().numpy(), vo, rtol=1e-12)
        d = cen.cpu().numpy() - co
        d -= L * np.round(d / L)
        assert np.abs(d).max() <= 1e-11
        I, _ = ctx.vof_drop_shape(f, lab, n, torch.from_numpy(co).to(DEV))
        Io, _ = O.drop_inertia(c[f], lo, no, co, h)
        assert (np.abs(I.cpu().numpy() - Io) <= 1e-12 * np.abs(Io) + 1e-12 * np.abs(Io).max(1, keepdims=True)).all()
        total += vo.sum()
        drops += no
    assert st["n_drops"] == drops
    assert st["volume"] == pytest.approx(total, rel=1e-12)
    ctx.close()


def lattice(m, a):
    g = (np.arange(m) + 0.5) * a
    return np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)


PAIR_CASES = {
    "two": lambda r: (r.random((2, 3)) * 10, [10.0] * 3, 0.0),
    "tile_edge": lambda r: (r.random((513, 3)) * 30, [30.0] * 3, 0.0),
    "two_tiles": lambda r: (r.random((1025, 3)) * [30, 40, 50], [30.0, 40.0, 50.0], 1e-9),
    "lattice_ties": lambda r: (lattice(6, 4.0), [24.0] * 3, 1e-9),
    "many_candidates": lambda r: (r.random((300, 3)) * 8, [8.0] * 3, 2.0),
    "all_candidates": lambda r: (r.random((90, 3)) * 8, [8.0] * 3, 50.0),
    "outside_box": lambda r: (r.random((200, 3)) * 60 - 20, [30.0] * 3, 0.0),
    "far_from_origin": lambda r: (r.random((200, 3)) * 30 + 1e6, [30.0] * 3, 0.0),
    "close_pairs": lambda r: (np.concatenate([q := r.random((100, 3)) * 30, q + 1e-9 * r.normal(size=(100, 3))]),
                              [30.0] * 3, 0.0),
}


@pytest.mark.parametrize("name", sorted(PAIR_CASES))
def test_nearest_pairs(vof, name):
    cen, box, tie = PAIR_CASES[name](np.random.default_rng(12))
    hr, hrt, mom = vof.vof_pair_stats(torch.from_numpy(np.ascontiguousarray(cen)).to(DEV), box, 200, 0.25, tie_tol=tie)
    ref = O.PairStats(200, 0.25).add(cen, box, tie_tol=tie)
    np.testing.assert_allclose(hr.cpu().numpy(), ref.hist_r, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(hrt.cpu().numpy(), ref.hist_rt, rtol=1e-12, atol=1e-12)
    m = mom.cpu().numpy()
    scale = np.abs(cen).max()
    assert m[12] == ref.E
    np.testing.assert_allclose(m[:3], ref.msum, atol=1e-12 * len(cen) * scale)
    np.testing.assert_allclose(m[3:12], ref.rsum, rtol=1e-12, atol=1e-12 * len(cen) * scale)
