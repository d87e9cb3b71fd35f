"""Keys that are switched off by a score of -inf (a channel of k that is -inf where q's is positive): whole tiles of them for a part of
the kernel that sees only those at first, a group of warps, a key slot, a warp or half a window.  They weigh nothing; the
result is the softmax over the other keys."""
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


def attend(q, k, v):
    return torch.softmax(q @ k.transpose(-1, -2) / 8, -1) @ v


def reference(q, k, v, Hg, Wg, win, P):
    q, k, v = (t.double() for t in (q, k, v))
    o = torch.empty_like(q)
    o[:, :, :P] = attend(q[:, :, :P], k, v)
    idx = P + torch.arange(Hg * Wg, device=q.device).view(Hg, Wg)
    for y in range(0, Hg, win):
        for x in range(0, Wg, win):
            t = idx[y:y + win, x:x + win].reshape(-1)
            s = torch.cat([torch.arange(P, device=q.device), t])
            o[:, :, t] = attend(q[:, :, t], k[:, :, s], v[:, :, s])
    return o


# mask: which tokens are off.  Behind the first 64 (of a window: the first row of 16); every other 16; the upper half of every 8 x 8 window
TAIL, ODD, UPPER = (lambda t, y, x: t >= 64), (lambda t, y, x: t % 32 >= 16), (lambda t, y, x: y % 8 < 4)
CASES = [  # dtype, B, H, P, Hg, Wg, win, mask
    ("f32", 1, 3, 0, 1, 300, 512, TAIL),               # keys over four groups
    ("f32", 2, 40, 0, 1, 300, 512, TAIL),
    ("f32", 1, 3, 2, 32, 32, 16, ODD),
    ("f32", 1, 2, 1, 40, 30, 16, TAIL),                # prefix queries: keys over eight groups
    ("bf16", 1, 2, 0, 1, 600, 1024, TAIL),             # keys over four slots
    ("bf16", 1, 2, 0, 1, 1370, 2048, TAIL),
    ("bf16", 1, 6, 1, 37, 37, 16, ODD),                # prefix queries: 16 keys per warp
    ("bf16", 1, 2, 0, 24, 40, 8, UPPER),
    ("bf16", 2, 2, 3, 21, 39, 8, UPPER),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:-1])))
def test_keys_of_score_minus_infinity(jv, case):
    dtype, B, H, P, Hg, Wg, win, mask = case
    N = P + Hg * Wg
    gen = torch.Generator(device=DEV).manual_seed(7400 + N)
    q, k, v = (torch.randn((B, H, N, 64), generator=gen, device=DEV) for _ in range(3))
    q[..., 0] = 1.0
    t = torch.arange(N, device=DEV)
    off = mask(t, (t - P).clamp(min=0) // Wg, (t - P).clamp(min=0) % Wg) & (t >= P)
    if win < Hg and mask is TAIL:
        off &= (t - P) % Wg % win >= 4                 # some keys in every window's every row
    k[:, :, off, 0] = float("-inf")
    if dtype == "bf16":
        q, k, v = (x.bfloat16() for x in (q, k, v))
    o = jv.full_attn(q, k, v) if win >= Hg and win >= Wg else jv.window_attn(q, k, v, Hg, Wg, win, win, prefix=P)
    ref = reference(q, k, v, Hg, Wg, win, P)
    assert bool(torch.isfinite(ref).all()) and bool(torch.isfinite(o).all())
    # fp32: sums of up to 1400 terms; bf16: probabilities and result rounded to 2^-9
    assert float((o.double() - ref).norm() / ref.norm()) <= (3e-6 if dtype == "f32" else 1e-2)


def test_a_row_without_any_key_is_nan(jv):
    q, k, v = (torch.randn((1, 2, 300, 64), device=DEV) for _ in range(3))
    q[..., 0], k[..., 0] = 1.0, float("-inf")
    assert bool(torch.isnan(jv.full_attn(q, k, v)).all())
    q, k, v = (t[:, :, :256].bfloat16().contiguous() for t in (q, k, v))
    assert bool(torch.isnan(jv.window_attn(q, k, v, 16, 16, 8, 8)).all())
    q, k, v = (t.repeat(1, 1, 3, 1) for t in (q, k, v))
    assert bool(torch.isnan(jv.full_attn(q, k, v)).all())
