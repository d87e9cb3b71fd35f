"""The window kernel on windows smaller than its two query tiles: two windows of one 128-token tile per item, and four of 8 x 8
tokens (two side by side in a tile, each row attending its own half of the tile's keys).  Grids cut the windows in every way:
right halves of a tile outside the grid, one column or one row of a window left, a second tile or a second key step
missing; prefix tokens (one and the most the kernel takes), strided inputs, fewer items than SMs and several per CTA."""
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


CASES = [  # B, H, P, Hg, Wg, wh, ww, fused activation
    (1, 2, 0, 16, 16, 8, 8, False),
    (1, 3, 0, 9, 17, 8, 8, False),
    (1, 2, 0, 13, 24, 8, 8, True),
    (2, 2, 1, 21, 39, 8, 8, False),
    (1, 2, 16, 35, 25, 8, 8, False),
    (32, 12, 0, 16, 16, 8, 8, True),
    (4, 16, 5, 37, 53, 8, 8, False),
    (1, 2, 0, 17, 33, 8, 16, False),
    (8, 8, 3, 45, 50, 8, 16, False),
    (2, 3, 0, 21, 45, 4, 32, True),
    (1, 2, 7, 31, 20, 16, 8, False),
    (3, 5, 0, 41, 23, 16, 8, False),
    (8, 16, 5, 33, 47, 16, 16, False),
    (1, 16, 5, 64, 64, 16, 16, False),   # the prefix queries ahead of the windows although a few SMs are free
    (1, 24, 1, 40, 60, 16, 16, False),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_small_windows(jv, oracle, case):
    B, H, P, Hg, Wg, wh, ww, fused = case
    N = P + Hg * Wg
    q, k, v = inputs.custom_qkv(B, H, N, 64, "bf16", seed=8800 + N + wh)
    if fused:
        act = torch.stack([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2).to(DEV).contiguous()
        dq, dk, dv = (act[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    else:
        dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    for _ in range(2):
        launches = jv.launch_count()
        jv.window_attn(dq, dk, dv, Hg, Wg, wh, ww, out=out, prefix=P)
        assert jv.launch_count() == launches + (2 if P else 1)
    check()
    heads = sample_heads(B, H, 4, N)
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    assert rel_err(pick(out.cpu()), oracle.window_attn(pick(q), pick(k), pick(v), Hg, Wg, wh, ww, prefix=P)) <= TOL["bf16"], case


def test_a_dominant_key_of_an_8x8_window_weighs_exactly_one(jv):
    """Every window has one key 2^4 to 2^8 above another one, in the other half of its rows, and nothing else of weight; all values are
    1.5.  With the larger one's probability taken against itself it is 1 in bf16 too, the smaller one's rounding is 2^-8 of
    2^-4 at most, and the result rounds to 1.5 (the neighbours are 2^-7 away).  Against the smaller one the larger one's probability is
    rounded itself, by up to 2^-8 of the whole."""
    B, H, Hg, Wg = 2, 16, 40, 56
    gen = torch.Generator().manual_seed(8901)
    nwin = B * H * (Hg // 8) * (Wg // 8)
    score = torch.full((nwin, 64), -40.0)                   # in powers of two: the softmax scale below is ln 2
    low = torch.randint(0, 32, (nwin,), generator=gen)      # keys 0 .. 31 are the window's upper four rows
    high = torch.randint(32, 64, (nwin,), generator=gen)
    swap = torch.rand(nwin, generator=gen) < 0.25
    low, high = torch.where(swap, high, low), torch.where(swap, low, high)
    score[torch.arange(nwin), low] = 0.0
    score[torch.arange(nwin), high] = torch.randint(4 * 32, 8 * 32, (nwin,), generator=gen) / 32.0   # exact in bf16
    k0 = score.view(B, H, Hg // 8, Wg // 8, 8, 8).permute(0, 1, 2, 4, 3, 5).reshape(B, H, Hg * Wg)
    q, k = (torch.zeros(B, H, Hg * Wg, 64) for _ in range(2))
    q[..., 0] = 1.0
    k[..., 0] = k0
    q, k, v = (t.bfloat16().to(DEV) for t in (q, k, torch.full_like(q, 1.5)))
    out = jv.window_attn(q, k, v, Hg, Wg, 8, 8, scale=0.6931471805599453)
    assert bool((out == 1.5).all()), int((out != 1.5).sum())
