"""Pin counts, block weights and the dense connectivity at the edges of their lane groups, against numpy.

The edges' sizes straddle the group widths (8, 16, 32 lanes), the thread-block
class (128 pins) and the segment length (2,048 pins); k straddles the mask
widths and the 16-byte rows; phi is also placed off a 16-byte boundary.
"""
import numpy as np
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402

SIZES = (0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 65, 127, 128, 129, 2047, 2048, 2049, 4096, 4097, 5000)


def _instance(c_max):
    rng = np.random.RandomState(11)
    n = 6000
    sizes = list(SIZES) + [int(x) for x in rng.randint(0, 12, 3000)]
    rng.shuffle(sizes)
    edges = [np.sort(rng.choice(n, s, replace=False)) for s in sizes]
    return synth.from_edges(n, edges, rng.randint(1, c_max + 1, n).astype(np.int32),
                            rng.randint(1, 9, len(edges)).astype(np.int32))


@pytest.mark.parametrize("c_max", [1, 32767])
@pytest.mark.parametrize("k", [2, 3, 4, 31, 32, 33, 36, 64, 65, 128, 130, 200, 255, 256])
@pytest.mark.parametrize("shift", [0, 1])
def test_pincounts_and_connectivity(k, c_max, shift):
    h = _instance(c_max)
    part = np.random.RandomState(k).randint(0, k, h.n).astype(np.int32)
    want = np.zeros((h.m, k), np.int32)
    np.add.at(want, (np.repeat(np.arange(h.m), np.diff(h.eptr)), part[h.pins]), 1)
    lam = (want > 0).sum(1).astype(np.int64)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))
    phi = torch.full((h.m * k + shift,), -7, dtype=torch.int32, device="cuda")[shift:]
    bw = torch.full((k,), -7, dtype=torch.int64, device="cuda")
    obj = torch.full((1,), -7, dtype=torch.int64, device="cuda")
    dpart = torch.as_tensor(part).cuda()
    jet.jet_build_pincounts(ctx, dpart, phi, bw)
    jet.jet_connectivity(ctx, phi, obj)
    assert np.array_equal(phi.cpu().numpy().reshape(h.m, k), want)
    assert np.array_equal(bw.cpu().numpy(), np.bincount(part, h.vwgt, k).astype(np.int64))
    objective = int((np.maximum(lam - 1, 0) * h.ewgt).sum())
    assert int(obj.item()) == objective
    # the bitmasks built beside phi give the same objective (the rebalancer's statistics read them)
    st = torch.zeros(8, dtype=torch.int64, device="cuda")
    ctx2 = jet.jet_ctx_create(ctx.hg, jet.params(k, eps=(1000, 1)))  # nothing is overloaded
    jet.jet_build_pincounts(ctx2, dpart, phi, bw)
    jet.jet_rebalance(ctx2, dpart, phi, bw, st)
    assert int(st[4].item()) == objective
    ctx.close()
    ctx2.close()
