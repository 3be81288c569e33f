"""What the autotuner times for the one-step kernels of 2D grids: runs down to
four rows at every order, and none so long that SMs are left without a CTA
(columns of a 2D grid are few, so such a run takes ten times a good one's
time, in every first call on a large grid)."""
import re

import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("so,ot", [(16, 2), (8, 2), (16, 4)])
def test_runs_of_2d_grids(monkeypatch, capfd, so, ot):
    import numpy as np
    import torch
    shape = (1500, 2900)                # beyond the launches of many steps, either direction
    monkeypatch.setenv("CKFWI_VERBOSE", "1")
    m = C.Model(C.GridSpec(2, shape, 10, 10.0, so, 0.8, 4, 3.0, ot))
    m.set_model(torch.full(shape, 2.0, device="cuda"))
    rec = np.array([[100.0, 0.0, 400.0]])
    capfd.readouterr()
    m.forward_shot(C.ShotSpec(src=(2000.0, 0.0, 3000.0), rec=rec, f0=0.02))
    m.close()
    lines = re.findall(r"autotune (\w+) ver (\d+) tile (\d+)x1 vec \d+ zlen (\d+):", capfd.readouterr().err)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert {p for p, _, _, _ in lines} == {"fwd", "adj"}
    for _, _, bx, z in lines:
        assert -(-shape[1] // int(bx)) * -(-shape[0] // int(z)) >= sms, (bx, z)
    assert min(int(z) for _, _, _, z in lines) == 4
