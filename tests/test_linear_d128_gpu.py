"""Linear attention at head_dim 128 on its tensor-core kernels: cluster sizes of the state pass from one to eight
chunks per head (chunks past the end among them), ragged 64- and 128-token tiles, one tile and many per CTA of the apply pass.

The state enters the product as three bf16 terms (24 bits), so the result differs from the oracle by the rounding of
the bf16 store; the bars are those of every bf16 comparison."""
import pytest
import torch

from paper_2605_26636_b200 import inputs
from tests._util import TOL, guarded_empty, rel_err, sample_heads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


CASES = [  # B, H, P, Hg, Wg
    (1, 1, 0, 1, 1),
    (1, 2, 0, 5, 13),        # 65 tokens: two tiles, two chunks
    (1, 3, 0, 8, 16),        # 128 tokens: exactly one apply tile
    (1, 2, 5, 17, 33),       # prefix tokens, 9 + tiles over eight chunks
    (2, 8, 0, 64, 64),
    (1, 8, 1, 37, 37),
    (3, 8, 0, 33, 40),       # 24 heads: six chunks
    (5, 10, 0, 20, 24),      # 50 heads: two chunks
    (1, 21, 0, 10, 64),      # seven chunks of two tiles: the last ones empty, shares of 19 rows
    (2, 80, 0, 9, 15),       # 160 heads: one chunk
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_linear_attention_head_dim_128(jv, oracle, case):
    B, H, P, Hg, Wg = case
    N = P + Hg * Wg
    q, k, v = inputs.custom_qkv(B, H, N, 128, "bf16", seed=12900 + N)
    heads = sample_heads(B, H, 4, N)
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    ws = jv.alloc_workspace("L", jv.make_shape(dq, Hg, Wg, P), None, DEV)
    ws.fill_(255)                                      # NaN: a state that is read before it is written shows
    launches = jv.launch_count()
    for _ in range(3):
        jv.linear_attn(dq, dk, dv, Hg, Wg, out=out, ws=ws, prefix=P)
    assert jv.launch_count() == launches + 6
    check()
    assert rel_err(pick(out.cpu()), oracle.linear_attn(pick(q), pick(k), pick(v), Hg, Wg, prefix=P)) <= TOL["bf16"], case
    again = jv.linear_attn(dq, dk, dv, Hg, Wg, prefix=P)
    assert torch.equal(out, again)                     # fixed summation order
