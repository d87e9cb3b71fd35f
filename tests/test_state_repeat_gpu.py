"""The state pass of the linear block where a head's last tile holds few tokens: the rows past them are zeros that no copy has to fetch, so
that tile is in shared memory almost at once, over a stage whose last readers have only just handed it back.  Every call gives
the first one's output bit for bit, and that is the formula's."""
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


# rings of three stages (more than 296 heads) and of six; a last tile of 4, 60 and 1 tokens
@pytest.mark.parametrize("B,H,N", [(24, 24, 2500), (12, 24, 4092), (5, 24, 1601)])
def test_last_tile_of_few_tokens(jv, B, H, N):
    gen = torch.Generator(device=DEV).manual_seed(6100 + N)
    q, k, v = (torch.randn((B, H, N, 64), generator=gen, device=DEV).bfloat16() for _ in range(3))
    out = torch.empty_like(q)
    first = jv.linear_attn(q, k, v, 1, N).clone()
    for rep in range(25):
        jv.linear_attn(q, k, v, 1, N, out=out)
        assert torch.equal(out, first), rep
    for b, h in ((0, 0), (B - 1, H - 1)):
        rq, rk, vv = q[b, h].double().clamp(min=0), k[b, h].double().clamp(min=0), v[b, h].double()
        ref = (rq @ (rk.T @ vv)) / ((rq @ rk.sum(0)) + 1e-6)[:, None]
        # KV rounded to bf16 (2^-9 of a term, 64 of them to a sum), the result rounded once more
        assert float((first[b, h].double() - ref).norm() / ref.norm()) <= 4e-3
