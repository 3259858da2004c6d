"""The many-row tensor-core GEMM (pairs of CTAs, stream-K) at the edges of its tiles and of its work split."""
import pytest
import torch

from paper_2211_17192_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n_out,k", [
    (129, 128, 64),      # one tile, one k-block: a single pair; two accumulators of 80 rows, the second nearly empty
    (129, 300, 72),      # features and inner dimension that end inside a tile; the last 128-feature tile does not exist
    (256, 256, 4096),    # one full tile shared by many pairs: a partial sum per pair
    (257, 1000, 200),    # two row tiles of 144
    (224, 5000, 1024),   # tiles shared by two or three pairs
    (513, 12800, 128),   # whole tiles first, the rest shared
    (2048, 37888, 8),    # whole tiles only
])
def test_many_rows_against_fp64(rows, n_out, k):
    gen = torch.Generator(device="cuda").manual_seed(rows + n_out + k)
    x = torch.randn((rows, k), device="cuda", generator=gen)
    w = (torch.randn((n_out, k), device="cuda", generator=gen) * 0.05).to(torch.bfloat16)
    packed = binding.spec_pack_weight(w)
    y = binding.spec_linear(x, packed, "tensor_packed", n_out=n_out)
    assert torch.equal(y, binding.spec_linear(x, w, "tensor"))
    ws = torch.full((binding.spec_linear_workspace_bytes(rows, n_out, k),), 255, dtype=torch.uint8, device="cuda")
    parts = binding.spec_linear_partials(x, packed, n_out, ws)  # (slots without a sum are zero, not what was there)
    total = parts[0].clone()
    for s in range(1, parts.shape[0]):
        total += parts[s]
    assert torch.equal(total, y)
    assert binding.spec_device_error() == 0
    for c in range(0, n_out, 8192):
        ref = x.double() @ w[c:c + 8192].double().T
        # x is kept to 2^-17 of its value by the two bf16 terms and sums of k products round to 2^-24 each:
        # (2^-17 + 2^-24 sqrt(k)) * sum |x w|, far below the bound
        bound = 2.0 ** -16 * (x.double().abs() @ w[c:c + 8192].double().abs().T)
        assert bool(((y[:, c:c + 8192].double() - ref).abs() <= bound + 1e-30).all())


@pytest.mark.parametrize("n_out", [8, 5])  # columns by fours, and one by one
@pytest.mark.parametrize("rows", [65535, 65536, 131073])
def test_more_rows_than_a_grid_has_along_y(rows, n_out):
    gen = torch.Generator(device="cuda").manual_seed(rows + n_out)
    x = torch.randn((rows, 64), device="cuda", generator=gen)
    w = (torch.randn((n_out, 64), device="cuda", generator=gen) * 0.05).to(torch.bfloat16)
    ref = x.double() @ w.double().T
    bound = 2.0 ** -16 * (x.double().abs() @ w.double().abs().T)  # (as above)
    for y in (binding.spec_linear(x, w, "tensor"), binding.spec_linear(x, binding.spec_pack_weight(w), "tensor_packed", n_out=n_out)):
        assert bool(((y.double() - ref).abs() <= bound + 1e-30).all())
