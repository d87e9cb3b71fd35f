"""Linear attention whose state leaves the range of fp32, on the kernels that take it apart into three bf16 terms: an infinite sum stays
infinite (the terms behind it are zero, not inf - inf)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


def _positive(*shape):
    gen = torch.Generator(device=DEV).manual_seed(300 + shape[-1])
    return (torch.rand(shape, generator=gen, device=DEV) + 0.5).bfloat16()


def test_infinite_products_at_head_dim_128(jv):
    """One infinite value: its channel is infinite for every token, the others are what they are without it."""
    q, k, v = (_positive(1, 2, 200, 128) for _ in range(3))
    clean = jv.linear_attn(q, k, v, 10, 20)
    v[0, 1, 77, 5] = float("inf")
    o = jv.linear_attn(q, k, v, 10, 20)
    assert bool((o[0, 1, :, 5] == float("inf")).all())
    keep = torch.ones_like(o, dtype=torch.bool)
    keep[0, 1, :, 5] = False
    assert torch.equal(o[keep], clean[keep])


def test_infinite_denominators_of_the_block_with_a_convolution(jv):
    """Keys so large that their sum overflows, values so small that the products do not: the attention's share is x / inf = 0 and the output
    the convolution's alone (centre taps of 1: v itself)."""
    H, Hg, Wg = 2, 16, 24
    q, k, v = (_positive(1, H, Hg * Wg, 64) for _ in range(3))
    k[0, 1, 100:104, 7] = 2e38
    v *= 2.0 ** -6
    b2 = torch.zeros(H * 64, 3, 3, device=DEV)
    b2[:, 1, 1] = 1.0
    o = jv.linear_attn(q, k, v, Hg, Wg, dwc={"k": 3, "R": 0, "b2": b2.view(-1)})
    assert torch.equal(o[0, 1], v[0, 1])
    assert bool(torch.isfinite(o).all()) and not torch.equal(o[0, 0], v[0, 0])
