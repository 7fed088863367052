"""The instance of test_gpu_recount.py has one iteration on each side of the move count from which phi is recounted.

The count follows from constants of launch_apply_jet, read from its source, so
that a change of them that puts both iterations on one side shows here.  The
moves are the oracle's.
"""
import os
import re

import pytest

import oracle
from paper_2504_12013_gb300 import build, synth


def _rebuild_min(hg, k):
    src = open(os.path.join(build.CSRC, "k_moves.cu")).read()
    body = src[src.index("cudaError_t launch_apply_jet("):]
    line = float(re.search(r"phi_bytes < ([0-9.e]+)\)", body).group(1))
    rate, per_move = map(float, re.search(r"bytes / \(([0-9.e]+) \* ([0-9.]+)\) \* c->n / ", body).groups())
    kwp = next(w for w in (1, 2, 4, 8) if 32 * w >= k)
    phi = 4.0 * hg.m * k
    assert phi >= line, "phi is below the size from which the rule applies"
    return int((phi + 8.0 * hg.m * kwp + 8.0 * hg.m + 8.0 * hg.P) / (rate * per_move) * hg.n / hg.P) + 1


@pytest.mark.parametrize("k", [255, 256])
def test_iterations_lie_on_both_sides(k):
    hg = synth.rownet(7, 40_000, 252_000, n_hubs=5, hub_min=3_000, hub_max=8_000)
    orc = oracle.Oracle(hg)
    st = oracle.State(orc, k, synth.part_perm(7, hg.n, k))
    first, second = (orc.refine_round(oracle.Params(k), (3, 4), st.part, st.phi, st.bw, st.locked)["approved"]
                     for _ in range(2))
    assert second < _rebuild_min(hg, k) <= first
