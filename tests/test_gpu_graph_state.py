"""State that a captured refinement shares with its context stays what the next call needs."""
import numpy as np
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402

SCHEDULE = ((3, 4), (0, 1))
K = 6


def test_batch_graph_outlives_a_change_of_path():
    """The batch's graph keeps the loop state of its contexts, also when one of them has changed its path and back."""
    h = synth.graph(3, 3000, 9000)
    part = synth.part_perm(5, h.n, K)
    ctxs = [jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(K)) for _ in range(2)]
    states = [jet.JetState(c, part) for c in ctxs]
    batch = jet.jet_batch_create(ctxs)
    want = jet.jet_batch_refine(batch, SCHEDULE, 3, states)
    refined = [s.part.clone() for s in states]
    for path in (True, False):
        jet.jet_set_graph_path(ctxs[0], path)
        for s in states:
            s.part.copy_(torch.as_tensor(part))
        assert jet.jet_batch_refine(batch, SCHEDULE, 3, states) == want
        assert all(torch.equal(s.part, r) for s, r in zip(states, refined))
    batch.close()
    for c in ctxs:
        c.close()
