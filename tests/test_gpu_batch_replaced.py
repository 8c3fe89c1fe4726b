"""A batch whose fields were replaced between steps, listed afresh by tune(),
advances as a new batch does (after three steps, when the sweeps' order is that
of the first step again): bit for bit."""
import numpy as np
import pytest

from paper_2407_07463_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("precision", [0, 1])
def test_replaced_fields(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07463_gb300 import build, vof

    build.build()
    dt_ = torch.float64 if precision == 0 else torch.float32
    data = []
    for seed, shape in enumerate([(12, 10, 64), (9, 14, 36), (20, 8, 4)]):
        rng = np.random.default_rng(seed)
        c = [synth.sphere_cell_fractions(shape, rng.random((1, 3)) * np.array(shape[::-1]), 0.3 * min(shape))[None]
             for _ in range(2)]
        u = synth.solenoidal_velocity(shape, 4, 0.5, 0.6, seed)
        data.append([torch.from_numpy(q).to(DEV, dt_).contiguous() for q in (*c, u)] + [synth.dt_for_cfl(u, 0.4)])

    def batch(which):
        cs = [d[which].clone() for d in data]
        return cs, vof.Batch([(c, d[2], d[3]) for c, d in zip(cs, data)], precision=precision)

    got, B = batch(0)
    B.step(3)
    for c, d in zip(got, data):
        c.copy_(d[1])
    B.tune()
    B.step(2)
    B.report()
    B.close()
    want, B = batch(1)
    B.step(2)
    B.report()
    B.close()
    for g, w in zip(got, want):
        assert torch.equal(g, w)
