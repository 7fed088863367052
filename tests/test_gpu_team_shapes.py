"""Multi-block teams of fewer than 1,024 threads: the local selection's room follows the threads.

A team's block selects in shared memory up to 4 records a thread and one block
of the partition per 32 threads: k at and just above the latter bound, record
counts on both sides of the former, for every block size, against jet_refine;
and smaller blocks still share an SM.
"""
import numpy as np
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402

SCHEDULE = ((3, 4), (0, 1))


@pytest.mark.parametrize("ctas,threads", [(2, 128), (4, 160), (2, 256), (8, 256), (4, 512), (2, 768), (2, 1024)])
@pytest.mark.parametrize("over", [0, 1])
def test_selection_at_the_bounds_of_its_room(ctas, threads, over):
    k = min(ctas * (threads // 32) + over, 256)
    n = 4 * threads * ctas * 2  # the drift below overloads about half of the blocks: some rounds fit, some do not
    h = synth.uniform(n + k, n, int(1.1 * n), base=2, geo=(1, 2), size_cap=32, c_max=3, w_max=3)
    rng = np.random.RandomState(k)
    part = synth.part_perm(k, n, k)
    drift = rng.rand(n) < 0.4
    part[drift] = rng.randint(0, max(1, k // 2), int(drift.sum()))
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))
    want = jet.JetState(ctx, part)
    res = jet.jet_refine(ctx, SCHEDULE, 3, want.part, want.phi, want.block_w)
    got = jet.JetState(ctx, part)
    batch = jet.jet_batch_create([ctx])
    for split in (0, 1 << 30):
        jet.jet_batch_set_team(batch, ctas, threads, split)
        got.part.copy_(torch.as_tensor(part))
        assert jet.jet_batch_refine(batch, SCHEDULE, 3, [got])[0] == res
        assert torch.equal(got.part, want.part) and torch.equal(got.phi, want.phi)
        assert torch.equal(got.block_w, want.block_w)
    batch.close()
    ctx.close()


def test_small_blocks_share_an_sm():
    """Two blocks of 512 threads fit an SM's registers: a batch of many small instances takes about half the time in
    teams of 8 x 512 that it takes in teams of 8 x 1,024 (the same time while shared memory let one be resident)."""
    ctxs, parts = [], []
    for i in range(160):
        h = synth.uniform(i, 1500, 1650, base=2, geo=(1, 2), size_cap=32)
        ctxs.append(jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(8)))
        parts.append(torch.as_tensor(synth.part_perm(i, h.n, 8)).cuda())
    states = [jet.JetState(c, p.clone()) for c, p in zip(ctxs, parts)]
    batch = jet.jet_batch_create(ctxs)

    def fastest(threads):
        jet.jet_batch_set_team(batch, 8, threads)
        times = []
        for _ in range(4):
            for s, p in zip(states, parts):
                s.part.copy_(p)
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            jet.jet_batch_refine(batch, SCHEDULE, 8, states)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times)

    assert fastest(512) < 0.75 * fastest(1024)
    batch.close()
    for c in ctxs:
        c.close()
