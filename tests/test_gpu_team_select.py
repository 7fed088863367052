"""The persistent batch's two forms of the rebalancing selection against jet_refine.

A multi-block team selects in shared memory while no block of the team owns
more than 4,096 records (and 32 blocks of the partition), else team-wide: few
blocks of many vertices, many blocks, weights with 64-bit and longer keys, and
every team size, from a start that overloads the lower blocks.
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


@pytest.mark.parametrize("n,k,c_max", [(40_000, 2, 1), (40_000, 8, 4), (30_000, 33, 1), (9_000, 200, 1), (9_000, 256, 700),
                                       (20_000, 5, 1000), (70, 64, 1)])
@pytest.mark.parametrize("team", [(8, 1024), (2, 256), (1, 512)])
def test_team_selection(n, k, c_max, team):
    h = synth.uniform(3 * n + k, n, int(1.1 * n), base=2, geo=(2, 5), size_cap=64, c_max=c_max, w_max=3)
    rng = np.random.RandomState(k)
    part = synth.part_perm(k, n, k)
    drift = rng.rand(n) < 0.2
    part[drift] = rng.randint(0, max(1, k // 3), int(drift.sum()))
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))
    want = jet.JetState(ctx, part)
    res = jet.jet_refine(ctx, SCHEDULE, 3, want.part, want.phi, want.block_w)
    got = jet.JetState(ctx, part)
    batch = jet.jet_batch_create([ctx])
    jet.jet_batch_set_team(batch, *team, 0)
    out = jet.jet_batch_refine(batch, SCHEDULE, 3, [got])[0]
    assert out == res
    assert torch.equal(got.part, want.part) and torch.equal(got.phi, want.phi)
    assert torch.equal(got.block_w, want.block_w)
    batch.close()
    ctx.close()
