"""Standalone codec calls keep their scratch and words between calls: streams
do not depend on what was called before (other sizes, either mode, calls that
failed), bit for bit."""
import ctypes

import numpy as np
import pytest

from paper_1810_05268_gb300 import ckfwi as C
from paper_1810_05268_gb300._lib import lib

pytestmark = pytest.mark.gpu


def _field(shape, seed):
    import torch
    r = np.random.default_rng(seed)
    return torch.from_numpy(np.cumsum(r.standard_normal(shape), axis=-1).astype(np.float32)).cuda()


def _raw(x, cap):
    """status of a compression into a buffer of `cap` words"""
    import torch
    out = torch.zeros(max(cap, 1), dtype=torch.int32, device="cuda")
    used, flags = ctypes.c_longlong(0), ctypes.c_int(0)
    nz, ny, nx = x.shape
    return lib().ckfwi_codec_compress(ctypes.c_void_p(x.data_ptr()), 3, nz, ny, nx, 1e-3,
                                      ctypes.c_void_p(out.data_ptr()), cap, ctypes.byref(used), ctypes.byref(flags),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))


def test_calls_do_not_depend_on_history():
    import torch
    a, b = _field((21, 34, 47), 1), _field((9, 5, 130), 2)
    nan = a.clone()
    nan[3, 4, 5] = float("nan")

    def streams():
        return [C.codec_compress(a, 1e-2)[0], C.codec_compress(b, 1e-3)[0], C.codec_compress_rate(b, 11)[0],
                C.codec_compress(a, 1e-2)[0]]

    first = streams()
    assert torch.equal(first[0], first[3])
    fields = [C.codec_decompress(first[0], a.shape), C.codec_decompress(first[2], b.shape)]
    assert float((fields[0] - a).abs().max()) <= 1e-2
    # failures in between: a pool that overflows at the table and at the payload, a corrupt stream of
    # either mode, a rate word out of range, a non-finite value
    for cap in (20, first[0].numel() - 1):
        assert _raw(a, cap) == C.POOL_OVERFLOW
    for s, shape, word in ((first[0], a.shape, 5), (first[2], b.shape, 8), (first[2], b.shape, 1)):
        bad = s.clone()
        bad[word] = 77
        with pytest.raises(C.CkfwiError) as e:
            C.codec_decompress(bad, shape)
        assert e.value.status == C.CORRUPT
    assert C.codec_compress(nan, 1e-2)[1] and C.codec_compress_rate(nan, 8)[1]
    again = streams()
    for x, y in zip(first, again):
        assert torch.equal(x, y)
    assert torch.equal(C.codec_decompress(again[0], a.shape), fields[0])
    assert torch.equal(C.codec_decompress(again[2], b.shape), fields[1])
