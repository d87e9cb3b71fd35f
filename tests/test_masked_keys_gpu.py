"""Keys that are switched off by a score of -inf (a channel of k that is -inf where q's is positive): whole tiles of them for a part of
the kernel that sees only those at first, a group of warps, a key slot, a warp or half a window.  They weigh nothing; the
result is the softmax over the other keys.  And keys whose score is +inf or no number: a softmax with one of those is no number,
wherever the key lies."""
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
    return torch.softmax(q @ k.transpose(-1, -2) * q.shape[-1] ** -0.5, -1) @ v


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


# One call for each kernel (and dtype, head_dim, prefix) that takes exponentials of scores, windows of 0 being full attention
ROUTES = [  # dtype, D, B, H, P, Hg, Wg, win
    ("bf16", 64, 1, 48, 0, 1, 1024, 0),                # four query tiles per CTA
    ("bf16", 64, 1, 24, 0, 1, 1024, 0),                # two
    ("bf16", 64, 1, 24, 0, 1, 600, 0),                 # keys over four slots
    ("bf16", 64, 1, 24, 0, 1, 200, 0),                 # short sequences on the window kernel
    ("bf16", 64, 1, 4, 0, 40, 36, 16),
    ("bf16", 64, 1, 4, 5, 40, 36, 16),
    ("bf16", 64, 1, 4, 0, 40, 36, 8),
    ("bf16", 64, 1, 4, 5, 40, 36, 8),
    ("bf16", 64, 2, 8, 0, 65, 33, 32),                 # windows of eight tiles
    ("bf16", 128, 2, 8, 0, 1, 1200, 0),
    ("bf16", 128, 2, 8, 0, 40, 30, 16),
    ("f32", 64, 1, 24, 0, 1, 1000, 0),                 # tensor cores
    ("f32", 64, 2, 12, 1, 25, 27, 8),                  # two windows to a block
    ("f32", 64, 1, 12, 70, 20, 20, 16),
    ("f32", 64, 1, 3, 0, 1, 300, 0),                   # multiply-adds
    ("f32", 64, 1, 3, 5, 20, 20, 16),
]
BAR = {"f32": 3e-6, "bf16": 1e-2}      # (as above)


def _call(jv, case, seed):
    dtype, D, B, H, P, Hg, Wg, win = case
    N = P + Hg * Wg
    gen = torch.Generator(device=DEV).manual_seed(seed + N)
    q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV) for _ in range(3))
    q[..., 0] = 1.0

    def run():
        a = [x.bfloat16() if dtype == "bf16" else x for x in (q, k, v)]
        o = jv.full_attn(*a) if win == 0 else jv.window_attn(*a, Hg, Wg, win, win, prefix=P)
        return o.double(), reference(*a, Hg, Wg, win if win else max(Hg, Wg), P)
    return q, k, v, run


def _compare(o, ref, dtype, what):
    assert torch.equal(torch.isnan(o), torch.isnan(ref)), what
    f = torch.isfinite(ref)
    assert bool(torch.isfinite(o[f]).all()), what
    assert float((o - ref)[f].norm() / ref[f].norm()) <= BAR[dtype], what


@pytest.mark.parametrize("case", ROUTES, ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("value", [float("nan"), float("inf")], ids=str)
def test_a_score_that_is_no_number_or_plus_infinity(jv, case, value):
    """At every position of a tile of 32 scores: in full attention one key per head, a head on, in windows one per window."""
    dtype, D, B, H, P, Hg, Wg, win = case
    N = P + Hg * Wg
    for off in (0, 15, 30, N - 20) if win == 0 else (0, 23):
        q, k, v, run = _call(jv, case, 7500)
        kf = k.view(B * H, N, D)
        for h in range(B * H - 1):
            if win == 0:
                kf[h, (off + h) % N, 0] = value
                continue
            for w, (y0, x0) in enumerate((y, x) for y in range(0, Hg, win) for x in range(0, Wg, win)):
                i = (off + 7 * h + w) % (win * win)
                y, x = y0 + i // win, x0 + i % win
                if w % 5 != 4 and y < Hg and x < Wg:
                    kf[h, P + y * Wg + x, 0] = value
        o, ref = run()
        assert bool(torch.isnan(ref).any()) and bool(torch.isfinite(ref).any())
        _compare(o, ref, dtype, off)


@pytest.mark.parametrize("case", ROUTES, ids=lambda c: "x".join(map(str, c)))
def test_first_keys_of_score_minus_infinity(jv, case):
    """The first steps of a row see no key of weight: 64 keys, and two tiles and a bit; in windows the first 1/4 and all but the last row."""
    dtype, D, B, H, P, Hg, Wg, win = case
    N = P + Hg * Wg
    t = torch.arange(N, device=DEV)
    y = (t - P).clamp(min=0) // Wg
    masks = [t < n for n in (64, 128 if N < 300 else 261)] if win == 0 else [(y % win < n) & (t >= P) & (y < Hg - Hg % win) for n in (win // 4, win - 1)]
    for off in masks + ([t < P + 64] if win and P else []):          # (with the prefix keys, which the prefix queries see first)
        q, k, v, run = _call(jv, case, 7600)
        k[:, :, off, 0] = float("-inf")
        o, ref = run()
        assert bool(torch.isfinite(ref).any())
        _compare(o, ref, dtype, int(off.sum()))


@pytest.mark.parametrize("case", ROUTES, ids=lambda c: "x".join(map(str, c)))
def test_rows_without_any_key_are_nan(jv, case):
    """Every key of the first head, and in windows every key of the first window, its prefix keys included."""
    dtype, D, B, H, P, Hg, Wg, win = case
    q, k, v, run = _call(jv, case, 7700)
    k[0, 0, :, 0] = float("-inf")
    if win:
        t = torch.arange(P + Hg * Wg, device=DEV) - P
        k[:, :, (t < 0) | ((t // Wg < win) & (t % Wg < win)), 0] = float("-inf")
    o, ref = run()
    assert bool(torch.isnan(ref).any()) and bool(torch.isfinite(ref).any())
    _compare(o, ref, dtype, 0)


@pytest.mark.parametrize("what", ["q zero", "two channels", "two signs", "beside large", "large q", "larger q", "small q", "tiny q", "large scores", "lowest", "mixed"])
@pytest.mark.parametrize("case", [c for c in ROUTES if c[0] == "f32"], ids=lambda c: "x".join(map(str, c)))
def test_infinities_in_fp32_keys(jv, case, what):
    """Where an infinite channel of k does not simply switch its key off, or does so among values that come close to the bounds of the kernels: the rows
    that are no numbers are, and the others are as accurate as ever."""
    dtype, D, B, H, P, Hg, Wg, win = case
    N = P + Hg * Wg
    q, k, v, run = _call(jv, case, 7800)
    t = torch.arange(N, device=DEV)
    off, rows = t % 9 == 4, t % 5 == 2
    k[:, :, off, 0] = float("-inf")
    if what == "q zero":                                   # 0 * inf: no number
        q[:, :, rows, 0] = 0.0
        q[..., 1] = 0.0                                    # (and zeros that meet nothing)
    elif what == "two channels":                           # of one sign or two, by q's
        k[:, :, t % 90 == 4, 40] = float("-inf")
    elif what == "two signs":
        k[:, :2, t % 90 == 4, 40] = float("inf")
        q[..., 40] = 0.5
    elif what == "beside large":                           # finite, and against the infinity
        k[:, :, t % 90 == 4, 40] = 3e38
        q[..., 40] = 0.5
    elif what in ("large q", "larger q"):
        k[:, :, ~off, 0] = 0.0
        q[:, :, rows, 0] = 5e4 if what == "large q" else 1e9
    elif what == "small q":
        q[:, :, rows, 0] = 1e-9
    elif what == "tiny q":
        q[:, :, rows, 0] = 1e-36
    elif what == "large scores":                           # the others are far below
        k[:, :, ~off, 3], q[..., 3] = -1e12, 0.0
        q[:, :, rows, 3] = 1e9
    elif what == "lowest":
        k[:, :, off, 0] = torch.finfo(torch.float32).min
    elif what == "mixed":                                  # one key left in some windows and rows
        k[:, :, t % 8 != 1, 0] = float("-inf")
    o, ref = run()
    assert bool(torch.isfinite(ref).any())
    if what == "large scores":                             # weights of scores of 1e20: only the largest one's counts, and rounding decides which is
        assert torch.equal(torch.isnan(o), torch.isnan(ref))
        o, ref = o[:, :, ~rows], ref[:, :, ~rows]
    _compare(o, ref, dtype, what)


@pytest.mark.parametrize("what", ["v inf", "v nan", "v 1e35", "v 1e-37", "q inf", "q nan"])
@pytest.mark.parametrize("case", [c for c in ROUTES if c[0] == "f32"], ids=lambda c: "x".join(map(str, c)))
def test_fp32_values_beyond_the_ordinary(jv, case, what):
    """In one channel, of every 50th token or (very small ones) of all: what comes out infinite or no number is where fp64 has it, the rest, channel by channel, as
    accurate as ever."""
    dtype, D, B, H, P, Hg, Wg, win = case
    q, k, v, run = _call(jv, case, 7900)
    name, value = what.split()
    t = q if name == "q" else v
    if value == "1e-37":
        t[..., 3] *= 1e-37
    else:
        t[:, ::2, 7::50, 3] = float(value)
    o, ref = run()
    assert torch.equal(torch.isnan(o), torch.isnan(ref)) and torch.equal(torch.isinf(o), torch.isinf(ref))
    for c in (slice(3, 4), slice(4, D)):
        f = torch.isfinite(ref[..., c])
        assert float((o - ref)[..., c][f].norm()) <= BAR[dtype] * float(ref[..., c][f].norm())
