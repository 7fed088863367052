"""State that a captured refinement shares with its context stays what the next call needs."""
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


def _candidates(ctx, st):
    n = ctx.hg.n
    out = [torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"),
           torch.zeros(n, dtype=torch.uint8, device="cuda")]
    jet.jet_candidates(ctx, (3, 4), st.part, st.phi, torch.zeros(n, dtype=torch.uint8, device="cuda"), *out)
    return out


@pytest.mark.parametrize("how", ["refine", "batch", "team", "autotune"])
def test_a_second_launch_names_the_phi_of_its_bitmasks(how):
    """A state is refined, another one is counted, the first is refined again by the captured graph: a call on the
    other state finds its own bitmasks."""
    h = synth.uniform(4, 3000, 3300, base=2, geo=(1, 2), size_cap=32)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(K))
    first, other = jet.JetState(ctx, synth.part_perm(1, h.n, K)), jet.JetState(ctx, synth.part_random(2, h.n, K))
    batch = jet.jet_batch_create([ctx])
    if how in ("team", "autotune"):
        jet.jet_batch_set_team(batch, 1, 256)

    def refine():
        first.part.copy_(torch.as_tensor(synth.part_perm(1, h.n, K)))
        if how == "refine":
            jet.jet_refine(ctx, SCHEDULE, 3, first.part, first.phi, first.block_w)
        elif how == "autotune":
            jet.jet_batch_autotune(batch, SCHEDULE, 3, [first], [(1, 256)], sample=1, trial_iterations=2)
        else:
            jet.jet_batch_refine(batch, SCHEDULE, 3, [first])

    refine()
    jet.jet_build_pincounts(ctx, other.part, other.phi, other.block_w)
    refine()
    got = _candidates(ctx, other)
    fresh = jet.jet_ctx_create(ctx.hg, jet.params(K))
    want = _candidates(fresh, jet.JetState(fresh, other.part.clone()))
    member = want[2].bool()
    assert torch.equal(got[2], want[2]) and int(member.sum()) > 0
    for g, w in zip(got[:2], want[:2]):
        assert torch.equal(g[member], w[member])
    batch.close()
    ctx.close()
    fresh.close()
