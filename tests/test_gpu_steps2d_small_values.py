"""2D launches of many steps against the one-step kernels where values get so
small that products round to zero: order 2 on a grid much wider than the wave
has come, so its tail runs out below the smallest numbers.  Compared by their
bytes: the signs of zeros are the same too."""
import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu

ONE_STEP = "1,128,1,16"
MANY = "9,184,1,19,4"


def _medium(shape):
    import torch
    g = torch.Generator().manual_seed(1)
    c = torch.randn((1, 1) + tuple(n // 12 + 2 for n in shape), generator=g).cuda()
    f = torch.nn.functional.interpolate(c, size=tuple(shape), mode="bilinear", align_corners=True)[0, 0]
    return (2.2 + 0.5 * torch.tanh(f)).contiguous()


@pytest.mark.parametrize("so", [2, 4, 8])
@pytest.mark.parametrize("store", ["fp32", "bf16"])
def test_bytes_of_a_tail(monkeypatch, so, store):
    import torch
    shape, nt, nrec = (464, 1104), 200, 40
    g = C.GridSpec(2, shape, 10, 10.0, so, 0.8, nt, 3.0)
    x = np.random.default_rng(0).uniform(0, 10830.0, nrec)
    rec = np.stack([np.full(nrec, 20.0), np.zeros(nrec), x], axis=1)
    shot = C.ShotSpec(src=(20.0, 0.0, 5415.0), rec=rec, f0=0.02, t0=40.0)
    vel, dobs = _medium(shape), torch.zeros((nt + 1, nrec), device="cuda")
    out = []
    for one in (True, False):
        for k in ("CKFWI_TILE_FWD", "CKFWI_TILE_ADJ"):
            monkeypatch.setenv(k, ONE_STEP if one else MANY)
        monkeypatch.setenv("CKFWI_BATCH_VER", "1" if one else "9")
        m = C.Model(g)
        m.set_model(vel)
        res = [m.forward_shot(shot).cpu().numpy()]
        for kw in (dict(ckpt_slots=nt, store_mode="fp32"), dict(ckpt_slots=20, store_mode=store)):
            _, grad, st = m.adjoint_gradient(shot, dobs, **kw)
            res.append(grad.cpu().numpy())
        assert (st["fwd_ver"], st["adj_ver"]) == ((1, 1) if one else (9, 9))
        res.append(m.batch_gradient([shot] * 2, [dobs] * 2, 20, store_mode=store, grad_f32=True)[1].cpu().numpy())
        out.append(res)
        m.close()
    # the tail is in the gradient: zeros beyond it, and the smallest numbers before them
    assert (out[0][1] == 0).any() and (np.abs(out[0][1][out[0][1] != 0]) < 1e-38).any()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32))
