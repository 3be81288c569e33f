"""Device memory of 2D models: the extra fields of the launches of many steps
only on grids that such launches take, and counted where the width of a batch
is chosen from the free memory."""
import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _field(shape, so):
    """bytes of a padded field"""
    k = so // 2
    return (shape[0] + 2 * k) * ((max(4, (k + 3) // 4 * 4) + shape[1] + k + 31) // 32 * 32) * 4


def test_grid_beyond_the_sms_takes_no_extra_fields():
    import torch
    shape, nt, pool = (1500, 3000), 12, 8 << 20
    f, n = _field(shape, 8), shape[0] * shape[1]
    vel = torch.full(shape, 2.0, device="cuda")
    rec = np.array([[100.0, 0.0, 400.0]])
    shot = C.ShotSpec(src=(2000.0, 0.0, 3000.0), rec=rec, f0=0.02)
    dobs, grad = torch.zeros((nt + 1, 1), device="cuda"), torch.empty(shape, device="cuda")
    for counted in (False, True):           # the first round loads the kernels
        a = _free()
        m = C.Model(C.GridSpec(2, shape, 10, 10.0, 8, 0.8, nt, 3.0))
        m.set_model(vel)
        b = _free()
        _, _, st = m.adjoint_gradient(shot, dobs, 4, store_mode="codec", tol=1e-5, pool_bytes=pool, grad=grad)
        c = _free()
        m.close()
        if counted:
            assert st["fwd_ver"] != 9 and st["adj_ver"] != 9
            # ten fields and the velocity; the pool and two fields' codec scratch
            assert a - b < 10.6 * f + 4 * n
            assert b - c < pool + 2.2 * 4 * C.codec_bound_words(2, shape[0], 1, shape[1]) + 2 * f


def test_batch_stays_within_the_memory_it_is_given(monkeypatch):
    import torch
    # a field just within two 2 MB allocation units, so that none is lost to rounding
    shape, nt, shots, given = (928, 1104), 8, 12, 800 << 20
    vel = torch.full(shape, 2.0, device="cuda")
    rec = np.array([[100.0, 0.0, 400.0]])
    sh = [C.ShotSpec(src=(2000.0, 0.0, 300.0 * (i + 1)), rec=rec, f0=0.02) for i in range(shots)]
    dl = [torch.zeros((nt + 1, 1), device="cuda") for _ in sh]
    kw = dict(store_mode="codec", tol=1e-5, pool_bytes=2 << 20)
    monkeypatch.setenv("CKFWI_FREE_BYTES", str(given))
    monkeypatch.setenv("CKFWI_BATCH_VER", "9")
    for counted in (False, True):
        m = C.Model(C.GridSpec(2, shape, 10, 10.0, 8, 0.8, nt, 3.0))
        m.set_model(vel)
        m.adjoint_gradient(sh[0], dl[0], 4, **kw)
        out = torch.empty(shape, dtype=torch.float64, device="cuda")
        a = _free()
        _, _, st = m.batch_gradient(sh, dl, 4, grad_sum=out, **kw)
        b = _free()
        m.close()
        if counted:
            assert st["fwd_ver"] == st["adj_ver"] == 9
            # not one lane at a time either
            assert 2 * _field(shape, 8) < a - b <= given
