"""The bf16 product of the one-sided modes at the edges of its tile choice: CTA pairs (256 x 256) with ragged rows and
half a column tile, and single CTAs with 64, 128 and 256 columns."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K,N", [
    (2300, 256, 2176),     # pairs: 9 x 9 tiles, 252 rows in the last one, 128 columns in the last one
    (18945, 128, 128),     # pairs: one column tile, of which one CTA's half is missing; one row in the last row tile
    (9000, 128, 512),      # 142 tiles of 256 columns (128 would take two waves)
    (2300, 384, 640),      # 128 columns
    (65, 640, 384)])       # 64 columns
def test_tile_forms_of_the_bf16_product(T, K, N):
    """Against a float64 product of the same bf16 values: float32 accumulation of K exact products is within
    K * 2^-24 * sum|a b| of it, the result is rounded to bf16 once."""
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(T + N)
    x = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    w = (torch.randn(N, K, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    res = B.dense_one_sided(x, B.W16A16, w_bf16=w)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    want = x.double() @ w.double().t()
    mag = x.double().abs() @ w.double().abs().t()
    err = (res["out"].double() - want).abs()
    assert bool((err <= K * 2.0 ** -24 * mag + 2.0 ** -8 * want.abs() + 1e-30).all())
