"""jet_profile_work reports the radix-select levels of the selection in use, on both sides of 4,096 vertices per block."""
import pytest

from paper_2504_12013_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_12013_gb300 import jet  # noqa: E402


@pytest.mark.parametrize("n,segments", [(8193, True), (8194, False)])
@pytest.mark.parametrize("c_max", [1, 1000])
def test_select_levels(n, segments, c_max):
    h = synth.uniform(1, n, n, base=2, geo=(1, 2), size_cap=16, c_max=c_max)
    # key bits: the priority (64, or with unit weights those of (1 + lcm(1)) * max weighted degree) and the vertex id
    deg = int((h.vptr[1:] - h.vptr[:-1]).max())
    bits = (64 if c_max > 1 else (2 * deg).bit_length()) + (n - 1).bit_length()
    digit = 8 if segments else -(-bits // -(-bits // 11))  # 8-bit digits, or the fewest levels of at most 11 bits
    ctx = jet.jet_ctx_create(jet.DeviceHypergraph(h), jet.params(2))
    assert jet.jet_profile_work(ctx)["select_levels"] == -(-bits // digit)
    ctx.close()
