"""OT4 passes fed by tensor copies (Tile.ver 10) against the vector-blocked
ones: the same operations in the same order, so the results are equal bit for
bit (no tolerance).  Widths that leave 0, 3 and 26 points in the last 32-point
tile, depths below and above a z run, every storage (host slots and 16-bit
states take the vector-blocked passes within the same gradient)."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


def _run(monkeypatch, tile, c, nt, calls):
    import torch
    monkeypatch.setenv("CKFWI_TILE_FWD", tile)
    monkeypatch.setenv("CKFWI_TILE_ADJ", tile)
    m = C.Model(c.pg)
    m.set_model(torch.from_numpy(c.vel).cuda())
    d = m.forward_shot(c.shot())
    out = [d.cpu().numpy()]
    for kw in calls:
        phi, g, st = m.adjoint_gradient(c.shot(), d * 0.9, **kw)
        assert st["fwd_ver"] == st["adj_ver"] == int(tile.split(",")[0])
        out += [np.float64(phi), g.cpu().numpy()]
    m.close()
    return out


@pytest.mark.parametrize("pf", [1, 2])
@pytest.mark.parametrize("so,shape,zlen", [(2, (20, 18, 32), 20), (4, (23, 33, 35), 5), (8, (41, 29, 58), 12),
                                           (8, (22, 50, 64), 40), (16, (37, 34, 61), 9)])
def test_bitwise_equal(monkeypatch, so, shape, zlen, pf):
    nt = 14
    c = make_case(3, so, shape, 4, nt, time_order=4)
    calls = [dict(ckpt_slots=nt), dict(ckpt_slots=4, use_graph=True), dict(ckpt_slots=5, store_mode="fp16"),
             dict(ckpt_slots=5, store_mode="bf16", host_slots=2), dict(ckpt_slots=6, host_slots=3),
             dict(ckpt_slots=4, store_mode="codec", tol=1e-4)]
    a = _run(monkeypatch, "6,32,16,%d,4,0" % zlen, c, nt, calls)
    b = _run(monkeypatch, "10,32,16,%d,4,%d" % (zlen, pf), c, nt, calls)
    assert np.abs(a[0]).max() > 0
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
