"""FP32 device checkpoints keep u^{s-1} where the step before wrote it (their
own slot, or the slot below's u^s for checkpoints one step apart).  Gradients
over slot counts from one to all but one state, with and without host slots,
single shots and batches, are bitwise the gradient that keeps every state."""
import pytest

from gpu_cases import make_case

torch = pytest.importorskip("torch")
C = pytest.importorskip("paper_1810_05268_gb300.ckfwi")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("time_order", [2, 4])
@pytest.mark.parametrize("nt", [2, 3, 11, 26])
def test_checkpointed_equals_all_states_kept(nt, time_order):
    case = make_case(3, 4, (21, 26, 37), 5, nt, seed=5, time_order=time_order)
    m = C.Model(case.pg)
    m.set_model(torch.from_numpy(case.vel).cuda())
    # data nobody recorded: the misfit is not zero however few the steps
    d = torch.ones_like(m.forward_shot(case.shot()))
    _, ref, _ = m.adjoint_gradient(case.shot(), d, ckpt_slots=nt)
    assert torch.isfinite(ref).all() and (nt < 11 or float(ref.abs().max()) > 0)
    for slots in sorted({1, 2, 3, 4, 7, nt - 1} & set(range(1, nt))):
        for hs in sorted({0, 1, slots // 2, slots - 1} & set(range(slots))):
            kw = dict(ckpt_slots=slots, host_slots=hs)
            for graph in (False, True):
                _, g, _ = m.adjoint_gradient(case.shot(), d, use_graph=graph, **kw)
                assert torch.equal(g, ref), (kw, graph)
    b = m.batch_gradient([case.shot()] * 2, [d, d], ckpt_slots=nt)[1]
    for slots in sorted({2, 4, nt - 1} & set(range(1, nt))):
        g = m.batch_gradient([case.shot()] * 2, [d, d], ckpt_slots=slots)[1]
        assert torch.equal(g, b), slots
    m.close()
