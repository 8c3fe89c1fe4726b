"""vof_drop_table on a grid of nearly 2^31 cells: drops among its last cells take
their own smallest cell as the origin of the minimum image (166 GB on the
device; skipped where less is free).  The centroid of a drop of whole cells is
the mean of their centres, within one rounding per operation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_drops_in_the_last_cells():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07463_gb300 import build, vof

    build.build()
    nx, ny, nz = 128, 128, 130816
    cfg = vof.make_config(nx, ny, nz, precision=vof.VOF_MIXED, stats_rbins=1, stats_tbins=1)
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < vof.vof_workspace_size(cfg) + 5 * 4 * nx * ny * nz + (12 << 30):
        pytest.skip("not enough device memory")
    c = torch.zeros((1, nz, ny, nx), dtype=torch.float32, device=DEV)
    u = torch.zeros((3, nz, ny, nx), dtype=torch.float32, device=DEV)
    labels = torch.zeros((nz, ny, nx), dtype=torch.int32, device=DEV)
    # (x, y, z) of the middle cell of seven; the first lies half a period in x and y from the cells of index
    # 0x7f7f7f7f and INT_MAX - 1 (a root taken from there splits it), the last wraps in y
    centres = [(63, 62, 130700), (62, 62, 130812), (64, 0, 12)]
    for tag, (x, y, z) in enumerate(centres, 1):
        for d in ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)):
            at = (z + d[2], (y + d[1]) % ny, x + d[0])
            c[(0,) + at] = 1.0
            labels[at] = tag
    ctx = vof.Context(cfg, c, u)
    vol, cen = (t.cpu().numpy() for t in ctx.vof_drop_table(0, labels, len(centres)))
    ctx.close()
    del c, u, labels, ctx
    torch.cuda.empty_cache()
    assert np.array_equal(vol, [7.0] * 3)
    assert np.abs(cen - (np.array(centres) + 0.5)).max() <= 1e-10
