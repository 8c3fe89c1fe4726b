"""A new context's statistics accumulators start at zero whatever the workspace
held: the first event of a context over two drops counts two, in whole numbers."""
import numpy as np
import pytest

from paper_2407_07463_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("rbins,tbins", [(1, 1), (7, 3), (31, 33), (1024, 150)])
def test_first_event(monkeypatch, rbins, tbins):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07463_gb300 import build, vof

    build.build()
    empty = torch.empty

    def filled(*a, **k):
        t = empty(*a, **k)
        return t.fill_(0x7F) if t.dtype == torch.uint8 else t

    monkeypatch.setattr(torch, "empty", filled)
    shape = (20, 18, 22)
    c = synth.sphere_cell_fractions(shape, np.array([[5.2, 5.1, 5.3], [15.4, 12.2, 14.6]]), 3.2)
    ctx = vof.Context(vof.make_config(shape[2], shape[1], shape[0], stats_rbins=rbins, stats_tbins=tbins),
                      torch.from_numpy(c[None].copy()).to(DEV),
                      torch.zeros((3,) + shape, dtype=torch.float64, device=DEV))
    r = ctx.vof_stats(reset=False)
    ctx.close()
    assert r["n_drops"] == 2 and r["events"] == 2 and r["chi_drops"] == 2
    assert r["hist_r"].sum() == 2 and r["hist_rt"].sum() == 2
    assert np.abs(r["M"]).max() <= 1e-12  # the two separations are each other's opposites
