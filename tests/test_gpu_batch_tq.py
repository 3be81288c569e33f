"""Batched steps fed by tensor copies (generation 8) against the vector-blocked
ones: every lane runs the same operations in the same order, so the sums are
equal bit for bit (no tolerance).  Lanes of different sizes (last tiles of 1, 3
and 32 points, depths below a z run), every storage, graph replay."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu

SHAPES = [(24, 20, 33), (30, 33, 35), (22, 49, 64)]
SURVEY, OFFSETS = (40, 60, 70), [(0, 0, 0), (10, 27, 35), (18, 5, 6)]


@pytest.mark.parametrize("so", [2, 4, 8, 16])
@pytest.mark.parametrize("kw", [dict(ckpt_slots=13), dict(ckpt_slots=4, use_graph=True),
                                dict(ckpt_slots=5, store_mode="fp16"),
                                dict(ckpt_slots=5, store_mode="codec", tol=1e-4)])
def test_windows(monkeypatch, so, kw):
    import torch
    cases = [make_case(3, so, s, 3, 13, seed=i) for i, s in enumerate(SHAPES)]
    out = []
    for ver in ("3", "8"):
        monkeypatch.setenv("CKFWI_BATCH_VER", ver)
        models, dl = [], []
        for c in cases:
            m = C.Model(c.pg)
            m.set_model(torch.from_numpy(c.vel).cuda())
            monkeypatch.setenv("CKFWI_TILE_FWD", "3,32,16,8,4")
            monkeypatch.setenv("CKFWI_TILE_ADJ", "3,32,16,8,4")
            dl.append(m.forward_shot(c.shot()) * 0.9)
            models.append(m)
        for _ in range(2):       # the second replays the graph, where there is one
            phi, g, st = C.batch_gradient_models(models, [c.shot() for c in cases], dl, OFFSETS, SURVEY, **kw)
            assert st["fwd_ver"] == st["adj_ver"] == int(ver)
            out.append((phi, g.cpu().numpy()))
        for m in models:
            m.close()
    assert np.abs(out[0][1]).max() > 0
    for phi, g in out[1:]:
        assert phi == out[0][0]
        np.testing.assert_array_equal(g, out[0][1])
