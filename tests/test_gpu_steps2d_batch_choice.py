"""2D batches whose forward steps are launches of many and whose reverse steps
are one a launch, and the other way round: equal to one-step launches bit for
bit in every storage; and the form a batch chooses is not slower than one-step
launches, where taking the many-step ones wherever they fit was."""
import time

import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


def _case(shape, so, nt, shots):
    import torch
    g = C.GridSpec(2, shape, 8, 10.0, so, 0.8, nt, 3.0)
    r = np.random.default_rng(3)
    ext = [(s - 2 * g.nbl - 1) * g.h for s in shape]
    rec = np.stack([np.full(30, 20.0), np.zeros(30), r.uniform(0, ext[1], 30)], axis=1)
    sh = [C.ShotSpec(src=(20.0, 0.0, (i + 0.5) / shots * ext[1]), rec=rec, f0=0.02, t0=min(40.0, 0.4 * nt * 0.8))
          for i in range(shots)]
    vel = torch.linspace(1.6, 2.8, shape[0], device="cuda")[:, None].expand(shape).contiguous()
    return g, vel, sh


def _batch(monkeypatch, form, g, vel, sh, dl, slots, **kw):
    if form:
        monkeypatch.setenv("CKFWI_BATCH_VER", form)
    else:
        monkeypatch.delenv("CKFWI_BATCH_VER", raising=False)
    m = C.Model(g)
    m.set_model(vel)
    out = m.batch_gradient(sh, dl, slots, **kw)
    return m, out


@pytest.mark.parametrize("store,kw", [("fp32", {}), ("bf16", dict(use_graph=True)), ("codec", dict(tol=1e-5)),
                                      ("rate", dict(rate=14, use_graph=True))])
@pytest.mark.parametrize("nt,slots", [(1, 1), (40, 6), (70, 40), (24, 24)])
def test_mixed_forms(monkeypatch, store, kw, nt, slots):
    if slots == 1 and store in ("codec", "rate"):
        pytest.skip("compressed storage takes two slots or more")
    g, vel, sh = _case((83, 140), 8, nt, 3)
    m = C.Model(g)
    m.set_model(vel)
    dl = [m.forward_shot(s) * 0.9 for s in sh]
    m.close()
    want = None
    for form in ("1", "9,1", "1,9", "9"):
        m, (phi, grad, st) = _batch(monkeypatch, form, g, vel, sh, dl, slots, store_mode=store, **kw)
        assert [st["fwd_ver"], st["adj_ver"]] == [int(form[0]), int(form[-1])]
        m.close()
        if want is None:
            want = (phi, grad.cpu().numpy())
        assert phi == want[0]
        np.testing.assert_array_equal(want[1], grad.cpu().numpy())


def test_choice_is_no_slower(monkeypatch):
    import torch
    g, vel, sh = _case((600, 1200), 16, 60, 8)
    dl = [torch.zeros((g.nt + 1, 30), device="cuda") for _ in sh]
    best = []
    for form in ("1", None):
        m, (_, grad, _) = _batch(monkeypatch, form, g, vel, sh, dl, 12)
        t = []
        for _ in range(6):
            t0 = time.perf_counter()
            m.batch_gradient(sh, dl, 12, grad_sum=grad)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        best.append(min(t))
        m.close()
    # the same here, both chosen by time; 1.3 with many-step launches wherever they fit
    assert best[1] < 1.12 * best[0]
