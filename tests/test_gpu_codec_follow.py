"""A compressed checkpoint one step after another reads its u^{s-1} from the
stream of the one below.  That stream keeps its room in the pool and its entry
in the statistics; a pool of exactly the peak is enough, one word less is not."""
import numpy as np
import pytest

from gpu_cases import make_case

torch = pytest.importorskip("torch")
C = pytest.importorskip("paper_1810_05268_gb300.ckfwi")

pytestmark = pytest.mark.gpu


def _pairs(nt, slots):
    """Per checkpoint: does it follow the one below by one step, nothing restored between."""
    acts = C.revolve_schedule(nt, slots)[0].tolist()
    return [i >= 2 and acts[i - 1][0] == 0 and acts[i - 1][2] == 1 and acts[i - 2][0] == 1 for i, a in enumerate(acts)
            if a[0] == 1]


@pytest.mark.parametrize("dims,shape", [(3, (21, 26, 37)), (2, (61, 75))])
@pytest.mark.parametrize("mode", [dict(store_mode="codec", tol=1e-4), dict(store_mode="rate", rate=9)])
@pytest.mark.parametrize("slots", [3, 12, 25])
def test_following_checkpoints(dims, shape, mode, slots):
    nt = 26
    case = make_case(dims, 4, shape, 5, nt, seed=5)
    m = C.Model(case.pg)
    m.set_model(torch.from_numpy(case.vel).cuda())
    d = m.forward_shot(case.shot()) * 1.02
    _, g, _ = m.adjoint_gradient(case.shot(), d, ckpt_slots=slots, **mode)
    words = np.asarray(m.stream_words(), dtype=np.int64).reshape(-1, 2)     # u^s, u^{s-1} of each checkpoint
    follows = _pairs(nt, slots)
    assert len(words) == len(follows) and any(follows)
    for k, f in enumerate(follows):
        assert words[k].min() > 0
        assert not f or words[k, 1] == words[k - 1, 0]
    # the pool's peak is the streams' of the slots held at once, and is enough
    held, peak = {}, 0
    takes = iter(words.sum(axis=1))
    for op, _, b in C.revolve_schedule(nt, slots)[0].tolist():
        if op == 1:
            held = {k: w for k, w in held.items() if k < b}
            held[b] = int(next(takes))
            peak = max(peak, 4 * sum(held.values()))
    for graph in (False, True):
        h = m.adjoint_gradient(case.shot(), d, ckpt_slots=slots, pool_bytes=peak, use_graph=graph, **mode)[1]
        assert torch.equal(g, h)
    with pytest.raises(C.CkfwiError):
        m.adjoint_gradient(case.shot(), d, ckpt_slots=slots, pool_bytes=peak - 4, **mode)
    m.close()


@pytest.mark.parametrize("mode", [dict(store_mode="codec", tol=1e-6), dict(store_mode="rate", rate=24)])
def test_batched_lanes(mode):
    nt = 26
    case = make_case(3, 4, (21, 26, 37), 5, nt, seed=6)
    m = C.Model(case.pg)
    m.set_model(torch.from_numpy(case.vel).cuda())
    d = m.forward_shot(case.shot()) * 1.02
    _, one, _ = m.adjoint_gradient(case.shot(), d, ckpt_slots=12, **mode)
    _, two, _ = m.batch_gradient([case.shot()] * 2, [d, d], ckpt_slots=12, **mode)
    assert torch.equal(two, 2.0 * one.double())
    m.close()
