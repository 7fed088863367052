"""Pin counts of many edges of more than 128 pins (a warp per segment) against numpy.

More than 19,456 segments of up to 1,024 pins (16 waves of thread blocks), among them
the last segments of edges beyond 2,048 pins, sizes on both sides of the
warp's 128 pins in flight and of both bounds, every mask width, phi off a
16-byte boundary; and the step in time from 128 to 129 pins.
"""
import numpy as np
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402


def _instance(sizes, n, seed):
    rng = np.random.RandomState(seed)
    edges = [np.sort((rng.randint(n) + np.arange(s) * (n // (s + 1) or 1)) % n) for s in sizes]
    return synth.from_edges(n, edges)


@pytest.mark.parametrize("k,shift", [(2, 0), (31, 1), (32, 0), (33, 0), (64, 1), (65, 0), (128, 0), (129, 1), (255, 0),
                                     (256, 1)])
def test_many_segments(k, shift):
    rng = np.random.RandomState(k)
    sizes = [129, 130, 159, 160, 161, 255, 256, 257, 1023, 1024, 1025, 2047, 2048, 2049, 2177, 3072, 3073, 4097, 5000,
             128, 3, 0, 1] + [int(x) for x in rng.randint(129, 200, 20_000)]
    rng.shuffle(sizes)
    h = _instance(sizes, 9000, k)
    part = rng.randint(0, k, h.n).astype(np.int32)
    want = np.zeros((h.m, k), np.int32)
    np.add.at(want, (np.repeat(np.arange(h.m), np.diff(h.eptr)), part[h.pins]), 1)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k, eps=(1000, 1)))  # nothing is overloaded
    phi = torch.full((h.m * k + shift,), -7, dtype=torch.int32, device="cuda")[shift:]
    bw = torch.zeros(k, dtype=torch.int64, device="cuda")
    dpart = torch.as_tensor(part).cuda()
    jet.jet_build_pincounts(ctx, dpart, phi, bw)
    assert np.array_equal(phi.cpu().numpy().reshape(h.m, k), want)
    st = torch.zeros(8, dtype=torch.int64, device="cuda")
    jet.jet_rebalance(ctx, dpart, phi, bw, st)  # its statistics read the bitmasks
    assert int(st[4].item()) == int((np.maximum((want > 0).sum(1) - 1, 0) * h.ewgt).sum())
    bad = part.copy()
    bad[int(h.pins[h.eptr[sizes.index(160)]])] = k
    jet.jet_build_pincounts(ctx, torch.as_tensor(bad).cuda(), phi, bw)
    with pytest.raises(jet.JetError):
        jet.jet_refine(ctx, ((0, 1),), 1, torch.as_tensor(bad).cuda(), phi, bw)
    ctx.close()


def _fastest(size, m, k):
    h = _instance([size] * m, 400_000, size)
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))
    st = jet.JetState(ctx, synth.part_perm(1, h.n, k))
    times = []
    for _ in range(12):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        jet.jet_build_pincounts(ctx, st.part, st.phi, st.block_w)
        t1.record()
        torch.cuda.synchronize()
        times.append(t0.elapsed_time(t1))
    ctx.close()
    return min(times)


def test_no_step_from_128_to_129_pins():
    """Edges of 129 pins went to a thread block each and took 1.7 times the time of edges of 128."""
    assert _fastest(129, 60_000, 16) < 1.45 * _fastest(128, 60_000, 16)
