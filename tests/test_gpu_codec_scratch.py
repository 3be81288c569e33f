"""Codec gradients where memory serves the scratch of one field only
(CKFWI_SCRATCH_BYTES stands for it): results equal those with room for both
fields bit for bit, single and batched, recorded or not, and the scratch is
settled once a model, not in every call."""
import numpy as np
import pytest

from gpu_cases import make_case
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,shape", [(3, (30, 34, 41)), (2, (60, 77))])
def test_one_field_at_a_time(monkeypatch, capfd, dims, shape):
    import torch
    nt = 60
    c = make_case(dims, 8, shape, 5, nt, seed=4)
    vel = torch.from_numpy(c.vel).cuda()
    dobs = torch.from_numpy(1e-3 * np.random.default_rng(2).standard_normal((nt + 1, len(c.rec))).astype(np.float32)).cuda()
    out = []
    for short in (False, True):
        if short:
            monkeypatch.setenv("CKFWI_SCRATCH_BYTES", "0")
            monkeypatch.setenv("CKFWI_VERBOSE", "1")
        m = C.Model(c.pg)
        m.set_model(vel)
        res = []
        for graph in (True, True, False):
            phi, g, _ = m.adjoint_gradient(c.shot(), dobs, 7, store_mode="codec", tol=1e-6, use_graph=graph)
            res += [np.float64(phi), g.cpu().numpy()]
        if short:
            assert capfd.readouterr().err.count("codec scratch for one field") == 1
        for _ in range(2):
            phi, g, _ = m.batch_gradient([c.shot()] * 2, [dobs] * 2, 7, store_mode="codec", tol=1e-6)
            res += [np.float64(phi), g.cpu().numpy()]
        if short:
            # the clone of the second lane
            assert capfd.readouterr().err.count("codec scratch for one field") == 1
        out.append(res)
        m.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
