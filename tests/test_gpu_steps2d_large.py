"""2D grids large enough that launches of many steps are timed: in several
tiles, and, for recorded gradients, against one step a launch, forward and
reverse apart.  Whatever is chosen equals one-step launches bit for bit and is
not slower than they are."""
import time

import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu

ONE_STEP = "1,128,1,16"


def _case(shape, so, nt):
    g = C.GridSpec(2, shape, 10, 10.0, so, 0.8, nt, 3.0)
    r = np.random.default_rng(4)
    ext = [(s - 2 * g.nbl - 1) * g.h for s in shape]
    rec = np.stack([np.full(64, 20.0), np.zeros(64), r.uniform(0, ext[1], 64)], axis=1)
    return g, C.ShotSpec(src=(20.0, 0.0, 0.5 * ext[1]), rec=rec, f0=0.02, t0=min(40.0, 0.4 * nt * 0.8))


def _model(monkeypatch, g, fwd, adj):
    import torch
    for name, tile in (("CKFWI_TILE_FWD", fwd), ("CKFWI_TILE_ADJ", adj)):
        if tile:
            monkeypatch.setenv(name, tile)
        else:
            monkeypatch.delenv(name, raising=False)
    m = C.Model(g)
    m.set_model(torch.linspace(1.6, 2.8, g.shape[0], device="cuda")[:, None].expand(g.shape).contiguous())
    return m


KINDS = [dict(ckpt_slots=4), dict(ckpt_slots=30), dict(ckpt_slots=9, store_mode="bf16"),
         dict(ckpt_slots=9, store_mode="fp16"), dict(ckpt_slots=9, store_mode="codec", tol=1e-5),
         dict(ckpt_slots=9, store_mode="rate", rate=14), dict(ckpt_slots=6, host_slots=2)]


# 517 x 509: just above the size from which times decide; 97 x 203: below it
@pytest.mark.parametrize("shape,so,nt", [((517, 509), 4, 1), ((517, 509), 16, 30), ((700, 1101), 16, 24), ((97, 203), 8, 40)])
def test_equal_to_one_step_launches(monkeypatch, shape, so, nt):
    g, shot = _case(shape, so, nt)
    want = None
    for fwd, adj in ((ONE_STEP, ONE_STEP), (None, ONE_STEP), (ONE_STEP, None), (None, None)):
        m = _model(monkeypatch, g, fwd, adj)
        d = m.forward_shot(shot)
        res = [d.cpu().numpy()]
        for kw in KINDS:
            kw = dict(kw, ckpt_slots=min(kw["ckpt_slots"], nt))
            if nt == 1 and kw.get("store_mode", "fp32") not in ("fp32", "bf16", "fp16"):
                continue                # compressed storage takes two slots or more
            for graph in (False, True, True):
                phi, grad, _ = m.adjoint_gradient(shot, d * 0.9, use_graph=graph, **kw)
                res += [np.float64(phi), grad.cpu().numpy()]
        m.close()
        if want is None:
            want = res
        for a, b in zip(want, res):
            np.testing.assert_array_equal(a, b)
    assert nt == 1 or np.abs(want[2]).max() > 0


@pytest.mark.parametrize("shape,so", [((800, 1600), 16), ((700, 1100), 16)])
def test_no_slower_than_one_step_launches(monkeypatch, shape, so):
    import torch
    g, shot = _case(shape, so, 130)
    d, grad = torch.zeros((g.nt + 1, shot.nrec), device="cuda"), torch.empty(shape, device="cuda")
    best = []
    for tile in (ONE_STEP, None):
        m = _model(monkeypatch, g, tile, tile)
        for call in (lambda: m.forward_shot(shot, d_sim=d),
                     lambda: m.adjoint_gradient(shot, d, 4, use_graph=True, grad=grad)):
            t = []
            for _ in range(7):
                t0 = time.perf_counter()
                call()
                torch.cuda.synchronize()
                t.append(time.perf_counter() - t0)
            best.append(min(t))
        m.close()
    # by the estimate alone the gradient of 800 x 1600 took 1.23 of the one-step launches' time
    assert best[2] < 1.05 * best[0] and best[3] < 1.07 * best[1], best
