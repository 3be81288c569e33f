"""Waits that run out (CKFWI_TMA_WAIT_LIMIT < 0: they give up at once) in the
2D launches of many steps, the OT4 passes and the batched steps fed by tensor
copies: the call reports TIMEOUT, and the same model's next call, with the
usual bound, gives the values of a model that never timed out, bit for bit.
On a stream of its own, which the default stream does not order."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu

ONE_STEP = "1,128,1,16"


def _shots(c, n):
    x = np.linspace(20.0, (c.pg.shape[-1] - 2 * c.pg.nbl - 3) * 10.0, n)
    return [C.ShotSpec(src=(c.src[0], c.src[1], float(v)), rec=c.rec, f0=c.f0, t0=c.t0) for v in x]


def _calls(m, c, dobs, kind):
    """Results of one call of every kind under test"""
    if kind == "forward":
        return [m.forward_shot(c.shot()).cpu().numpy()]
    if kind == "batch":
        phi, g, _ = m.batch_gradient(_shots(c, 3), [dobs] * 3, 5)
    else:
        phi, g, _ = m.adjoint_gradient(c.shot(), dobs, 5, use_graph=kind == "graph")
    return [np.float64(phi), g.cpu().numpy()]


@pytest.mark.parametrize("dims,tf,ta,kind", [
    (2, None, None, "forward"), (2, None, None, "gradient"), (2, None, None, "graph"), (2, None, None, "batch"),
    (2, None, ONE_STEP, "gradient"), (2, ONE_STEP, None, "gradient"),
    (4, "10,32,16,9,4,1", "6,32,16,9,4,0", "forward"), (4, "10,32,16,9,4,2", "10,32,16,9,4,1", "graph"),
    (4, "6,32,16,9,4,0", "10,32,16,9,4,1", "gradient"), (3, None, None, "batch")])
def test_timeout_then_exact_results(monkeypatch, dims, tf, ta, kind):
    import torch
    nt = 40
    if dims == 2:
        c = make_case(2, 8, (97, 203), 5, nt, seed=3)
    else:
        c = make_case(3, 8, (35, 43, 70), 6, nt, seed=9, time_order=4 if dims == 4 else 2)
        monkeypatch.setenv("CKFWI_BATCH_VER", "8")
    for name, tile in (("CKFWI_TILE_FWD", tf), ("CKFWI_TILE_ADJ", ta)):
        if tile:
            monkeypatch.setenv(name, tile)
    vel = torch.from_numpy(c.vel).cuda()
    dobs = torch.from_numpy(1e-3 * np.random.default_rng(1).standard_normal((nt + 1, len(c.rec))).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        m = C.Model(c.pg)
        m.set_model(vel)
        want = _calls(m, c, dobs, kind)
        m.close()
        m = C.Model(c.pg)
        m.set_model(vel)
        for tuned in (False, True):       # the first call of a model, and one after good ones
            if tuned or kind == "batch":  # (a batch's tiles are timed with the usual bound)
                _calls(m, c, dobs, kind)
            monkeypatch.setenv("CKFWI_TMA_WAIT_LIMIT", "-1")
            with pytest.raises(C.CkfwiError) as e:
                _calls(m, c, dobs, kind)
            assert e.value.status == C.TIMEOUT
            monkeypatch.delenv("CKFWI_TMA_WAIT_LIMIT")
            for _ in range(2):
                for x, y in zip(want, _calls(m, c, dobs, kind)):
                    np.testing.assert_array_equal(x, y)
        m.close()
