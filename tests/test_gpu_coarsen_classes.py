"""Clustering on the GPU vs the oracle at the edges of the rating classes.

A vertex is rated by a warp (up to 64 rated pins), a block of three sizes (256,
1,024, 4,096) or with its table in the pool; its edges go through the kernels
32, 128, 256 or 512 at a time.  The instance has vertices on both sides of
each of these bounds, made of two-pin edges and of edges of up to 1,000 pins.
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

# two-pin edges and edges of the given sizes of one vertex: rated pins = two + sum(size - 1)
SHAPES = [(127, ()), (129, ()), (256, ()), (257, ()), (31, ()), (32, ()), (33, ()), (64, ()), (65, ()), (25, (40,)), (26, (40,)), (255, (770,)), (257, (768,)),
          (1024, ()), (1025, ()), (25, (1000,)), (26, (1000,)), (513, (1000, 1000, 1000, 587)),
          (513, (1000, 1000, 1000, 588)), (4096, ()), (4097, ()), (600, (1000,) * 5), (3, (1001, 1500))]


def _instance(c_max, w_max):
    rng = np.random.RandomState(5)
    n, edges = 7000, []
    for v, (two, sizes) in enumerate(SHAPES):
        others = np.setdiff1d(np.arange(n), [v])
        edges += [[v, int(u)] for u in rng.choice(others, two, replace=False)]
        edges += [[v, *map(int, rng.choice(others, s - 1, replace=False))] for s in sizes]
    edges += [list(map(int, rng.choice(n, rng.randint(1, 6), replace=False))) for _ in range(6000)]
    rng.shuffle(edges)
    return synth.from_edges(n, edges, rng.randint(1, c_max + 1, n).astype(np.int32),
                            rng.randint(1, w_max + 1, len(edges)).astype(np.int32))


@pytest.mark.parametrize("c_max,w_max", [(1, 1), (4, 9)])
@pytest.mark.parametrize("frac,ns,cd", [(30, 100, 100), (30, 0, 1), (700, 20, 4), (1, 7100, 1)])
def test_rating_classes(c_max, w_max, frac, ns, cd):
    h = _instance(c_max, w_max)
    cmax = max(2, int(h.vwgt.sum()) // frac)
    order = synth.vertex_order(3, h.n)
    if ns == 7100:  # one vertex at a time, the listed ones first
        order = np.concatenate([np.arange(len(SHAPES)), order[order >= len(SHAPES)]]).astype(np.int32)
    want = oracle.Oracle(h).cluster(cmax, order, n_single=ns, cap_div=cd)
    got = jet.jet_cluster(jet.DeviceHypergraph(h), cmax, torch.as_tensor(order).cuda(), n_single=ns, cap_div=cd)
    assert np.array_equal(got.cpu().numpy(), want)
