"""The status of a call that meets several conditions: a pool that overflows
is reported before a non-finite value (a program that grows its pool on
POOL_OVERFLOW and gives up on NONFINITE has to see the former)."""
import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


def _status(m, shot, dobs, **kw):
    with pytest.raises(C.CkfwiError) as e:
        m.adjoint_gradient(shot, dobs, 6, store_mode="codec", tol=1e-4, **kw)
    return e.value.status


@pytest.mark.parametrize("shape", [(40, 60), (36, 40, 44)])
def test_overflow_comes_before_nonfinite(shape):
    import torch
    nt, dims = 200, len(shape)
    g = C.GridSpec(dims, shape, 5, 10.0, 4, 0.8, nt, 3.0)
    m = C.Model(g)
    # far above the velocity the time step is stable for: the field grows past FP32's range
    m.set_model(torch.full(shape, 40.0, device="cuda"))
    mid = 0.4 * (shape[0] - 11) * 10.0
    rec = np.array([[mid, mid if dims == 3 else 0.0, mid]])
    shot = C.ShotSpec(src=tuple(rec[0]), rec=rec, f0=0.024)
    dobs = torch.zeros((nt + 1, 1), device="cuda")
    fields = 2 * 6 * int(np.prod(shape)) * 4
    # non-finite blocks are stored verbatim: no pool of this size is too small for them
    assert _status(m, shot, dobs, pool_bytes=2 * fields) == C.NONFINITE
    for graph in (False, True):
        assert _status(m, shot, dobs, pool_bytes=fields // 40, use_graph=graph) == C.POOL_OVERFLOW
    assert _status(m, shot, dobs, pool_bytes=2 * fields) == C.NONFINITE
    # and a model in the stable range runs
    m.set_model(torch.full(shape, 2.0, device="cuda"))
    phi, grad, _ = m.adjoint_gradient(shot, dobs, 6, store_mode="codec", tol=1e-4, pool_bytes=2 * fields)
    assert np.isfinite(phi) and bool(torch.isfinite(grad).all())
    m.close()
