"""Jet applies on both sides of the move count from which phi is counted anew, against the oracle.

phi just above the size from which the rule applies (256 MB); the first
iteration from a permuted start approves more moves than the rule's count, the
second fewer.  k = 255 has rows off the 16-byte boundary; the hub edges span
several segments.
"""
import numpy as np
import pytest

import oracle
from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402


@pytest.mark.parametrize("k", [255, 256])
@pytest.mark.parametrize("graph_mode", [0, 1])
def test_large_and_small_applies(k, graph_mode):
    hg = synth.rownet(7, 40_000, 252_000, n_hubs=5, hub_min=3_000, hub_max=8_000)
    part = synth.part_perm(7, hg.n, k)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(hg), jet.params(k))
    jet.jet_set_graph_mode(ctx, graph_mode)
    st = jet.JetState(ctx, part)
    orc = oracle.Oracle(hg)
    ost = oracle.State(orc, k, part)
    approved = []
    for r in range(2):
        st.round((3, 4))
        want = orc.refine_round(oracle.Params(k), (3, 4), ost.part, ost.phi, ost.bw, ost.locked)
        assert st.stats_dict() == want, f"iteration {r}"
        assert np.array_equal(st.part.cpu().numpy()[: hg.n], ost.part), f"iteration {r}: partition"
        assert np.array_equal(st.phi.cpu().numpy()[: hg.m * k].reshape(hg.m, k), ost.phi), f"iteration {r}: phi"
        assert np.array_equal(st.block_w.cpu().numpy(), ost.bw), f"iteration {r}: block weights"
        approved.append(want["approved"])
    assert 2 * approved[1] < approved[0]
    ctx.close()
