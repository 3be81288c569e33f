"""2D launches of many steps (Tile.ver 9) against the one-step kernels: the
same operations on every point, so the results are equal bit for bit (no
tolerance).  Grids from a single tile to one with a tile on every SM, last
tiles of one row or column up to full ones, receivers on tile corners, runs
shorter and longer than one launch's steps, every storage, and batches whose
lanes need several groups."""
import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C
from paper_1810_05268_gb300 import synth

pytestmark = pytest.mark.gpu

ONE_STEP = {"CKFWI_TILE_FWD": "1,128,1,16", "CKFWI_TILE_ADJ": "1,128,1,16"}


def _case(shape, so, nt, nbl, nrec, seed=3):
    h, dt = 10.0, 0.8
    vel = synth.grf(shape, 3.0, seed, 1.5, 3.0).astype(np.float32)
    g = C.GridSpec(2, shape, nbl, h, so, dt, nt, 3.0)
    inner = [(n - 2 * nbl - 1) * h for n in shape]
    r = synth.rng(seed + 1)
    # receivers anywhere, some on grid points
    rec = np.stack([r.uniform(0, inner[0], nrec), np.zeros(nrec), r.uniform(0, inner[1], nrec)], axis=1)
    rec[::3] = np.round(rec[::3] / h) * h
    shot = C.ShotSpec(src=(0.3 * inner[0], 0.0, 0.6 * inner[1]), rec=rec, f0=0.024, t0=min(60.0, 0.4 * nt * dt))
    return g, vel, shot


def _model(monkeypatch, g, vel, one_step):
    import torch
    for k, v in ONE_STEP.items():
        if one_step:
            monkeypatch.setenv(k, v)
        else:
            monkeypatch.delenv(k, raising=False)
    m = C.Model(g)
    m.set_model(torch.from_numpy(vel).cuda())
    return m


@pytest.mark.parametrize("so", [2, 4, 8, 16])
@pytest.mark.parametrize("shape,nt,nrec", [((21, 23), 9, 5), ((64, 130), 70, 700), ((97, 203), 131, 40),
                                           ((201, 161), 66, 101)])
def test_many_steps_equal_one_step(monkeypatch, so, shape, nt, nrec):
    import torch
    g, vel, shot = _case(shape, so, nt, 5, nrec)
    out = []
    for one in (True, False):
        m = _model(monkeypatch, g, vel, one)
        d = m.forward_shot(shot)
        dobs = d * 0.9
        res = [d.cpu().numpy()]
        for kw in (dict(ckpt_slots=nt), dict(ckpt_slots=5), dict(ckpt_slots=9, use_graph=True)):
            for _ in range(2 if kw.get("use_graph") else 1):
                phi, grad, st = m.adjoint_gradient(shot, dobs, **kw)
            res += [np.float64(phi), grad.cpu().numpy()]
        assert (st["fwd_ver"], st["adj_ver"]) == ((1, 1) if one else (9, 9))
        out.append(res)
        m.close()
    torch.cuda.synchronize()
    assert np.abs(out[0][0]).max() > 0
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("kw", [dict(store_mode="fp16"), dict(store_mode="bf16"), dict(store_mode="codec", tol=1e-4),
                                dict(store_mode="rate", rate=12), dict(store_mode="fp32", host_slots=4),
                                dict(store_mode="fp16", host_slots=3)])
@pytest.mark.parametrize("slots", [3, 14])
def test_storage_of_many_steps(monkeypatch, kw, slots):
    g, vel, shot = _case((75, 118), 8, 90, 6, 30)
    kw = dict(kw, host_slots=min(kw["host_slots"], slots - 2)) if "host_slots" in kw else kw
    out = []
    for one in (True, False):
        m = _model(monkeypatch, g, vel, one)
        dobs = m.forward_shot(shot) * 0.9
        phi, grad, _ = m.adjoint_gradient(shot, dobs, slots, **kw)
        out.append((phi, grad.cpu().numpy()))
        m.close()
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("store", ["fp32", "bf16", "codec"])
@pytest.mark.parametrize("shape,shots", [((40, 60), 3), ((420, 700), 7)])
def test_batches_of_many_steps(monkeypatch, store, shape, shots):
    g, vel, s0 = _case(shape, 8, 24, 5, 20)
    sh = [C.ShotSpec(src=(s0.src[0], 0.0, x), rec=s0.rec, f0=s0.f0, t0=s0.t0)
          for x in np.linspace(20.0, (shape[1] - 12) * 10.0, shots)]
    out = []
    for bv in ("1", "9"):
        m = _model(monkeypatch, g, vel, bv == "1")
        monkeypatch.setenv("CKFWI_BATCH_VER", bv)
        dl = [m.forward_shot(s) * 0.9 for s in sh]
        phi, grad, st = m.batch_gradient(sh, dl, 6, store_mode=store, tol=1e-4, use_graph=store == "bf16")
        assert st["fwd_ver"] == int(bv)
        out.append((phi, grad.cpu().numpy()))
        m.close()
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
