"""Rebalancing with the records in a segment per block against the oracle.

Sizes on both sides of every line of that form: 4,096 vertices per block
(segments or one list), 2^17 vertices (who keeps the block weights), segments
beyond one thread block's registers (4,096 records), beyond one thread block
(16,384: a cluster) and beyond the cluster's registers (32,768); keys of up to
64 bits and longer ones; c(V) on both sides of 2^32.
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

# (n, k, least and largest c(v), share of the vertices put into block 0)
CASES = [
    (131_071, 37, 1, 1, 0.02), (131_072, 37, 1, 4, 0.02), (131_073, 37, 1, 4, 0.02),
    (131_072, 200, 1, 1, 0.03), (131_073, 200, 1, 1, 0.03),
    (8_193, 2, 1, 1, 0.4), (8_194, 2, 1, 1, 0.4),        # 4,096 and 4,097 vertices per block
    (16_384, 8, 1, 1, 1.0), (16_385, 8, 1, 1, 1.0),      # no large segment possible; just one
    (12_000, 4, 1, 900, 1.0), (140_000, 40, 30_000, 32_767, 0.08),  # one block beyond its registers, longer keys
    (20_000, 8, 1, 4, 0.9), (30_000, 8, 1, 1000, 1.0),   # a cluster, the records held; with longer keys
    (90_000, 37, 1, 3, 1.0), (90_000, 37, 1, 900, 1.0),  # beyond the registers of the cluster
    (140_000, 64, 1, 2, 1.0),                            # ... where the apply keeps the block weights
    (140_000, 64, 30_000, 32_767, 0.5),                  # c(V) above 2^32
    (120_000, 64, 32_000, 32_767, 0.5),                  # just below
    (60_000, 16, 1, 1, -1.0),                            # three large segments
]


def _instance(n, k, c_lo, c_hi, share):
    h = synth.uniform(n + k, n, n + n // 10, base=2, geo=(1, 2), size_cap=32, w_max=3)
    rng = np.random.RandomState(k)
    h.vwgt[:] = rng.randint(c_lo, c_hi + 1, n)
    part = synth.part_perm(k, n, k)
    if share < 0:
        part = rng.randint(0, 3, n).astype(np.int32)
    else:
        part[rng.rand(n) < share] = 0
    return h, part


@pytest.mark.parametrize("n,k,c_lo,c_hi,share", CASES)
def test_rebalance_and_round(n, k, c_lo, c_hi, share):
    h, part = _instance(n, k, c_lo, c_hi, share)
    if c_lo == 30_000:
        assert int(h.vwgt.astype(np.int64).sum()) >= 1 << 32
    prm = oracle.Params(k, max_rebalance_rounds=4)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k, max_rebalance_rounds=4))
    orc = oracle.Oracle(h)
    ost = oracle.State(orc, k, part)
    st = jet.JetState(ctx, part)

    def same(what):
        assert np.array_equal(st.part.cpu().numpy(), ost.part), f"{what}: partition"
        assert np.array_equal(st.block_w.cpu().numpy(), ost.bw), f"{what}: block weights"
        assert np.array_equal(st.phi.cpu().numpy().reshape(h.m, k), ost.phi), f"{what}: phi"

    rounds, moves = orc.rebalance(prm, ost.part, ost.phi, ost.bw)
    jet.jet_rebalance(ctx, st.part, st.phi, st.block_w, st.stats)
    got = st.stats_dict()
    assert (got["rebalance_rounds"], got["rebalance_moves"]) == (rounds, moves) and rounds > 0
    same("rebalancing")
    for mode in (0, 1):  # kernel by kernel, then the captured iteration; from the skewed start again
        jet.jet_set_graph_mode(ctx, mode)
        ost = oracle.State(orc, k, part)
        st = jet.JetState(ctx, part)
        want = orc.refine_round(prm, (3, 4), ost.part, ost.phi, ost.bw, ost.locked)
        st.round((3, 4))
        assert st.stats_dict() == want, f"graph mode {mode}"
        same(f"iteration, graph mode {mode}")
    ctx.close()


def _fastest_rebalance(n, k):
    """Milliseconds of 32 rebalancing rounds that start with every vertex in block 0."""
    h = synth.uniform(n, n, n + n // 10, base=2, geo=(1, 2), size_cap=32)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))
    st = jet.JetState(ctx, np.zeros(n, np.int32))
    times = []
    for _ in range(6):
        st.part.zero_()
        jet.jet_build_pincounts(ctx, st.part, st.phi, st.block_w)
        torch.cuda.synchronize()
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        jet.jet_rebalance(ctx, st.part, st.phi, st.block_w, st.stats)
        t1.record()
        torch.cuda.synchronize()
        times.append(t0.elapsed_time(t1))
    assert st.stats_dict()["rebalance_rounds"] == 32
    ctx.close()
    return min(times)


def test_one_large_segment_is_no_slower_than_the_list_form():
    """100,000 vertices in one segment against 160,000 in one list: a selection by one thread block took 15 times
    the list form's time."""
    assert _fastest_rebalance(100_000, 37) < 2 * _fastest_rebalance(160_000, 37)
