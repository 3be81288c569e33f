"""Many receivers in 2D launches of many steps: more in a tile than its shared
list holds, other receivers in the next call, with and without graphs and in
batches; equal to the one-step kernels bit for bit, and not slower."""
import time

import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu

ONE_STEP = "1,128,1,16"


def _shot(g, n, seed):
    r = np.random.default_rng(seed)
    ext = [(s - 2 * g.nbl - 1) * g.h for s in g.shape]
    rec = np.stack([np.full(n, 20.0), np.zeros(n), r.uniform(0, ext[1], n)], axis=1)
    rec[n // 2:, 0] = r.uniform(0, 60.0, n - n // 2)
    return C.ShotSpec(src=(20.0, 0.0, 0.4 * ext[1]), rec=rec, f0=0.02, t0=20.0)


def _model(monkeypatch, g, one):
    import torch
    for k in ("CKFWI_TILE_FWD", "CKFWI_TILE_ADJ"):
        if one:
            monkeypatch.setenv(k, ONE_STEP)
        else:
            monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("CKFWI_BATCH_VER", "1" if one else "9")
    m = C.Model(g)
    m.set_model(torch.full(g.shape, 2.0, device="cuda"))
    return m


def test_crowded_tiles(monkeypatch):
    g = C.GridSpec(2, (90, 150), 10, 10.0, 8, 0.8, 70, 3.0)
    shots = [_shot(g, n, n) for n in (6000, 40, 9001)]
    out = []
    for one in (True, False):
        m = _model(monkeypatch, g, one)
        res = []
        for s in shots + shots[:1]:
            d = m.forward_shot(s)
            res.append(d.cpu().numpy())
            for graph in (False, True, True):
                phi, grad, st = m.adjoint_gradient(s, d * 0.9, 6, use_graph=graph)
                res += [np.float64(phi), grad.cpu().numpy()]
            assert st["fwd_ver"] == (1 if one else 9)
        phi, grad, st = m.batch_gradient(shots, [m.forward_shot(s) * 0.9 for s in shots], 6)
        assert st["fwd_ver"] == (1 if one else 9)
        out.append(res + [np.float64(phi), grad.cpu().numpy()])
        m.close()
    assert np.abs(out[0][0]).max() > 0
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_many_receivers_on_a_line_are_no_slower(monkeypatch):
    import torch
    g = C.GridSpec(2, (464, 1104), 10, 10.0, 8, 0.8, 300, 3.0)
    r = np.random.default_rng(1)
    n = 20000
    rec = np.stack([np.full(n, 20.0), np.zeros(n), r.uniform(0, 10830.0, n)], axis=1)
    shot = C.ShotSpec(src=(20.0, 0.0, 5000.0), rec=rec, f0=0.02)
    d = torch.empty((g.nt + 1, n), device="cuda")
    best = []
    for one in (True, False):
        m = _model(monkeypatch, g, one)
        t = []
        for _ in range(8):
            t0 = time.perf_counter()
            m.forward_shot(shot, d_sim=d)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        best.append(min(t))
        m.close()
    assert best[1] < best[0]      # 0.5 of it; with every tile looking at every receiver, 2.1
