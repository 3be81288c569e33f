"""Receivers of OT4 steps fed by tensor copies: pass 1, which samples them, has
a z run of its own, so its grid may hold fewer threads than there are
receivers while the step's own tile would hold enough, and the other way
round.  Every receiver is sampled either way, bitwise as by the
vector-blocked passes (the same operations in the same order)."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


def _run(monkeypatch, c, step, lap):
    import torch
    monkeypatch.setenv("CKFWI_TILE_FWD", step)
    monkeypatch.setenv("CKFWI_TILE_ADJ", step)
    if lap:
        monkeypatch.setenv("CKFWI_TILE_OT4_LAP", lap)
    else:
        monkeypatch.delenv("CKFWI_TILE_OT4_LAP", raising=False)
    m = C.Model(c.pg)
    m.set_model(torch.from_numpy(c.vel).cuda())
    d = m.forward_shot(c.shot())
    out = [d.cpu().numpy()]
    for kw in (dict(ckpt_slots=4), dict(ckpt_slots=5, host_slots=2), dict(ckpt_slots=5, store_mode="fp16")):
        phi, g, st = m.adjoint_gradient(c.shot(), d * 0.9, **kw)
        assert st["fwd_ver"] == int(step.split(",")[0])
        out += [np.float64(phi), g.cpu().numpy()]
    m.close()
    return out


# 32 x 18 points a plane: two CTAs, 256 threads a z run; 702 receivers
@pytest.mark.parametrize("step,lap", [(2, 24), (24, 2), (24, 24), (8, 9)])
def test_every_receiver_is_sampled(monkeypatch, step, lap):
    nt = 12
    c = make_case(3, 8, (24, 18, 32), 4, nt, nrec=26, time_order=4)
    assert c.rec.shape[0] == 702
    a = _run(monkeypatch, c, "6,32,16,12,4,0", None)
    b = _run(monkeypatch, c, "10,32,16,%d,4,1" % step, "10,32,16,%d,4,1" % lap)
    assert (np.abs(a[0]).max(axis=0) > 0).all()
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
