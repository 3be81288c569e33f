"""Fixed-rate streams of one or two blocks, at their exact length: the
shortest ones (one 4 x 4 block at 1 or 2 bits a value, 17 words) are shorter
than the fixed-accuracy mode's table for the same field.  Stream and field
equal the oracle's bit for bit; a stream cut by one word is still refused."""
import numpy as np
import pytest

from oracle import codec as OC
from paper_1810_05268_gb300 import ckfwi as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1), (4, 4), (3, 2), (4, 5), (4, 4, 4), (1, 1, 1), (2, 4, 5)])
@pytest.mark.parametrize("rate", [1, 2, 3, 32])
def test_shortest_streams(shape, rate):
    import torch
    x = np.random.default_rng(rate + len(shape)).standard_normal(shape).astype(np.float32)
    ref, _ = OC.compress_rate(x, rate)
    words, _ = C.codec_compress_rate(torch.from_numpy(x).cuda(), rate)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), ref)
    y = C.codec_decompress(words.clone(), shape).cpu().numpy()
    assert np.array_equal(y.view(np.uint32), OC.decompress(ref, shape).view(np.uint32))
    with pytest.raises(C.CkfwiError) as e:
        C.codec_decompress(words[:-1].clone(), shape)
    assert e.value.status == C.CORRUPT
