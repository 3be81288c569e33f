"""One launch group codes both fields of a takeshot on every lane of a batch:
the streams, hence the gradients, are those of single shots."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [dict(store_mode="codec", tol=1e-4), dict(store_mode="rate", rate=9)])
@pytest.mark.parametrize("dims,shape", [(2, (33, 41)), (2, (70, 260)), (3, (22, 31, 27))])
def test_lanes_equal_single_shots(dims, shape, mode):
    # fields of one chunk and of many, odd block counts
    import torch
    c = make_case(dims, 4, shape, 4, 30)
    m = C.Model(c.pg)
    m.set_model(torch.from_numpy(c.vel).cuda())
    inner = [(n - 9) * 10.0 for n in shape]
    shots = [C.ShotSpec(src=(20.0, 0.5 * inner[1] if dims == 3 else 0.0, x), rec=c.rec, f0=c.f0, t0=c.t0)
             for x in np.linspace(0.2, 0.8, 3) * inner[-1]]
    dl = [m.forward_shot(s) * 0.9 for s in shots]
    want, phis = np.zeros(shape), []
    for s, d in zip(shots, dl):
        phi, g, _ = m.adjoint_gradient(s, d, 5, grad_kind=C.SLOWNESS2, **mode)
        w = C.stream_words(m.h)
        assert w.size > 0 and w.size % 2 == 0 and (w > 0).all()
        want += g.cpu().numpy().astype(np.float64)
        phis.append(phi)
    phi, got, _ = m.batch_gradient(shots, dl, 5, grad_kind=C.SLOWNESS2, **mode)
    # FP64 sums of three float32 values, compensated against plain: a few ulp
    assert abs(phi - sum(phis)) <= 4e-16 * sum(phis) * 3
    np.testing.assert_allclose(got.cpu().numpy(), want, rtol=0, atol=1e-15 * np.abs(want).max() * 3)
    m.close()
