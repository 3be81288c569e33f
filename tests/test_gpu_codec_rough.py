"""Fixed-accuracy streams of rough fields, whose chunks are long (half the
field's size): bit for bit the oracle's, from one block to more than 1024
chunks, and the copies of a compression keep their loads in flight."""
import time

import numpy as np
import pytest

from oracle import codec as OC
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 4), (64, 66), (463, 777), (4, 4, 4), (5, 17, 33), (33, 64, 129), (131, 133, 135)])
@pytest.mark.parametrize("tol", [1e-2, 1e-5, 1e-7])
def test_streams_of_rough_fields(shape, tol):
    import torch
    x = np.random.default_rng(len(shape)).standard_normal(shape).astype(np.float32)
    ref, _ = OC.compress(x, tol)
    words, _ = C.codec_compress(torch.from_numpy(x).cuda(), tol)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), ref)
    y = C.codec_decompress(words, shape).cpu().numpy()
    assert np.array_equal(y.view(np.uint32), OC.decompress(ref, shape).view(np.uint32))


def _best(f):
    import torch
    t = []
    for _ in range(40):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_long_chunks_are_copied_at_speed():
    import torch
    torch.manual_seed(0)
    x = torch.randn((300, 400, 400), device="cuda").cumsum(-1) * 1e-3
    y = torch.empty_like(x)
    copy = _best(lambda: [y.copy_(x) for _ in range(8)])
    # 0.493 ms against eight copies' 0.47; 0.618 with one load in flight a thread
    assert _best(lambda: C.codec_compress(x, 1e-5)) < 1.18 * copy
