"""jet_connectivity on rows off the 16-byte boundary: values at the edges of the loads per lane, and their time."""
import numpy as np
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402


def _context(k, m, seed=3):
    h = synth.uniform(seed, 5000, m, base=2, geo=(1, 2), size_cap=16, w_max=7)
    return h, jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(k))


@pytest.mark.parametrize("k", [2, 3, 5, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 95, 97, 127, 128, 129, 159, 161, 193, 223,
                               225, 255, 256])
@pytest.mark.parametrize("m", [1, 37, 5001])
def test_every_number_of_loads(k, m):
    h, ctx = _context(k, m)
    rng = np.random.RandomState(k)
    phi = rng.randint(0, 3, (m, k)).astype(np.int32) * (rng.rand(m, 1) < 0.9)  # any table: empty rows too
    phi = phi.astype(np.int32)
    out = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    buf = torch.empty(m * k + 1, dtype=torch.int32, device="cuda")
    buf[1:] = torch.as_tensor(phi.reshape(-1))
    jet.jet_connectivity(ctx, buf[1:], out)
    assert int(out.item()) == int((np.maximum((phi > 0).sum(1) - 1, 0).astype(np.int64) * h.ewgt).sum())
    ctx.close()


def test_rows_of_255_take_about_the_time_of_256():
    """1 M rows: 2.4 times the time of the aligned form while a row's loads were a loop."""
    times = {}
    for k in (255, 256):
        h, ctx = _context(k, 1_000_000)
        phi = torch.zeros(h.m * k, dtype=torch.int32, device="cuda")
        out = torch.zeros(1, dtype=torch.int64, device="cuda")
        best = []
        for _ in range(10):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            jet.jet_connectivity(ctx, phi, out)
            t1.record()
            torch.cuda.synchronize()
            best.append(t0.elapsed_time(t1))
        times[k] = min(best)
        ctx.close()
        del phi
    assert times[255] < 1.9 * times[256]
