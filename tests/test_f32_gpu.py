"""The fp32 kernels (attention and the linear block at head_dim 64) at the sizes where they can go wrong.  Attention on multiply-adds: the
splits of a CTA into row warps and key groups, windows of a single key tile and ragged ones, prefix tokens alone in a
tile; on the tensor cores: ragged tiles, two windows to a block, values that its terms hold only just.  The linear block: chunk and tile
remainders, one-column grids, rows shorter than a thread's run of tokens.

Tolerance: a score is a sum of 64 products in fp32, magnitude up to about 60 before scaling by 1 / 8: its error stays
below 64 * 2^-24 * 60 / 8 = 3e-5, usually a tenth of that, and the result is off by that fraction of the values; the bar
of every fp32 comparison here, 1e-4 of the rms, covers it."""
import pytest
import torch

from paper_2605_26636_b200 import inputs
from tests._util import TOL, dwc_to_device, guarded_empty, rel_err, sample_heads

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


CASES = [  # B, H, P, Hg, Wg, win
    (1, 1, 0, 1, 1, 1),          # one token
    (1, 2, 0, 5, 13, 64),        # 65 tokens: two key tiles, the second of one key; one window
    (1, 6, 0, 16, 16, 8),        # F: 16-row tiles, eight key groups
    (1, 2, 5, 9, 23, 8),         # edge windows, windows of 64 + 5 keys
    (2, 8, 1, 17, 31, 16),       # on the tensor cores
    (4, 37, 0, 8, 8, 8),         # one key tile per window
    (3, 50, 3, 12, 17, 7),       # windows whose width is not a power of two
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_fp32_kernels(jv, oracle, case):
    B, H, P, Hg, Wg, win = case
    N = P + Hg * Wg
    q, k, v = inputs.custom_qkv(B, H, N, 64, "f32", seed=3200 + N)
    dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    heads = sample_heads(B, H, 6, N)
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)      # as one batch of sampled heads
    qs, ks, vs = pick(q), pick(k), pick(v)
    for name, call, ref in (
            ("F", lambda o: jv.full_attn(dq, dk, dv, out=o), lambda: oracle.full_attn(qs, ks, vs)),
            ("W", lambda o: jv.window_attn(dq, dk, dv, Hg, Wg, win, win, out=o, prefix=P),
             lambda: oracle.window_attn(qs, ks, vs, Hg, Wg, win, win, prefix=P)),
            ("L", lambda o: jv.linear_attn(dq, dk, dv, Hg, Wg, out=o, prefix=P),
             lambda: oracle.linear_attn(qs, ks, vs, Hg, Wg, prefix=P))):
        out, check = guarded_empty(q.shape, torch.float32, DEV)
        out.fill_(float("nan"))
        call(out)
        check()
        assert rel_err(pick(out.cpu()), ref()) <= TOL["f32"], (name, case)


# Calls that fill the chip go to the tensor cores, each value as three bf16 terms: ragged last tiles of rows and keys, prefix tokens in front of a window's
# keys, windows two to a block (an odd number of them, small ones at the edges, one to five key tiles that go through rings of two; more than 64
# keys come of prefix tokens only).  Heads: the dispatch asks for up to 2 row tiles of 32 per SM, these have twice that on 148 SMs.
TC_CASES = [  # B, H, P, Hg, Wg, window
    (1, 24, 0, 20, 20, (20, 20)),
    (2, 24, 0, 13, 17, (16, 16)),
    (1, 24, 5, 33, 35, (16, 16)),
    (4, 24, 1, 17, 23, (8, 8)),
    (2, 24, 70, 18, 23, (7, 9)),
    (4, 24, 70, 17, 17, (8, 8)),
    (2, 24, 200, 17, 23, (8, 8)),
    (2, 24, 70, 19, 10, (10, 10)),
    (8, 24, 0, 10, 11, (11, 11)),
]


def _tc_heads(q, k, v, heads):
    return tuple(torch.stack([t[b, h] for b, h in heads]).unsqueeze(0) for t in (q, k, v))


def _on_tensor_cores(jv, call, out):
    """Whether the call's attention goes there: those kernels leave the output alone while the status word is set, the others write it."""
    assert jv.device_status() == jv.JV_OK
    out.fill_(1234.5)
    jv.selftest_wait_timeout(1000)
    call(out)
    torch.cuda.synchronize()
    left = bool((out == 1234.5).all())
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    out.fill_(float("nan"))
    return left


@pytest.mark.parametrize("case", TC_CASES, ids=lambda c: "x".join(map(str, c[:5])) + "x%dx%d" % c[5])
def test_fp32_tensor_cores(jv, oracle, case):
    """Beside the bar of this file, the 2-norm of the error: 1.6e-7 to 2.3e-7 with all six products of terms in both contractions, 1.9e-6 at least
    without one of the three smallest in either (that arithmetic on the CPU, these inputs, 64 to 1155 keys)."""
    B, H, P, Hg, Wg, (wh, ww) = case
    q, k, v = inputs.custom_qkv(B, H, P + Hg * Wg, 64, "f32", seed=3600 + P + Hg)
    dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    heads = sample_heads(B, H, 4, P + Hg)
    qs, ks, vs = _tc_heads(q, k, v, heads)
    for name, call, ref in (
            ("F", lambda o: jv.full_attn(dq, dk, dv, out=o), lambda: oracle.full_attn(qs, ks, vs)),
            ("W", lambda o: jv.window_attn(dq, dk, dv, Hg, Wg, wh, ww, out=o, prefix=P),
             lambda: oracle.window_attn(qs, ks, vs, Hg, Wg, wh, ww, prefix=P))):
        out, check = guarded_empty(q.shape, torch.float32, DEV)
        assert _on_tensor_cores(jv, call, out), (name, case)
        call(out)
        check()
        o, r = _tc_heads(out.cpu(), out.cpu(), out.cpu(), heads)[0], ref()
        assert rel_err(o, r) <= TOL["f32"], (name, case)
        d = o.double().numpy() - r
        assert float((d * d).sum() ** 0.5) <= 6e-7 * float((r * r).sum() ** 0.5), (name, case)


@pytest.mark.parametrize("term", ["00", "01", "10", "02", "11", "20"])
def test_fp32_tensor_cores_terms(jv, term):
    """Scores that are one product of terms, q's i-th by k's j-th, all others cancelling between two channels: without it every key weighs the same."""
    B, H, N = 1, 24, 400
    a, b = 2.0 ** -9, 2.0 ** -18                             # behind 1, what the second and the third term hold
    qc, kc = {"00": ((1, 0), (1, 0)), "01": ((1, -1), (1 + a, 1)), "10": ((1 + a, -1), (1, 1)), "02": ((1, -1), (1 + a + b, 1 + a)),
              "11": ((1 + a, -1), (1 + a, 1 + 2 * a)), "20": ((1 + a + b, -1 - a), (1, 1))}[term]
    size = 4 / sum(x * y for x, y in zip(qc, kc))             # scores of up to 4
    q, k = torch.zeros(B, H, N, 64), torch.zeros(B, H, N, 64)
    v = inputs.normal((B, H, N, 64), 3790, "f32")
    row, key = 2.0 ** -(torch.arange(N) % 3).float(), 2.0 ** -(torch.arange(N) % 4).float() * (1 - 2 * (torch.arange(N) % 7 == 0).float())
    for c in range(2):
        q[..., 5 + 20 * c], k[..., 5 + 20 * c] = row * qc[c], key * kc[c] * size
    ref = torch.softmax(q.double() @ k.double().transpose(-1, -2), -1) @ v.double()
    assert float((torch.softmax(4 * row[:, None] * key[None], -1).double() @ v.double() - ref).norm() / ref.norm()) < 1e-6
    out = torch.empty(B, H, N, 64, device=DEV)
    call = lambda o: jv.full_attn(q.to(DEV), k.to(DEV), v.to(DEV), scale=1.0, out=o)
    assert _on_tensor_cores(jv, call, out)
    call(out)
    assert float((out.cpu().double() - ref).norm() / ref.norm()) <= 6e-7


@pytest.mark.parametrize("what", ["k -inf", "k lowest", "k inf", "q nan", "v inf", "v large"])
def test_fp32_tensor_cores_special_values(jv, what):
    """What is no finite number, or so large that products of bf16 terms overflow, gives what fp64 gives."""
    B, H, N = 1, 24, 400
    q, k, v = inputs.custom_qkv(B, H, N, 64, "f32", seed=3700)
    name, value = what.split()
    t = {"q": q, "k": k, "v": v}[name]
    x = {"-inf": float("-inf"), "inf": float("inf"), "lowest": torch.finfo(torch.float32).min, "nan": float("nan"), "large": 1e37}[value]
    q[0, 2, :, 3] = q[0, 2, :, 3].abs() + 0.5              # (an infinite score has one sign)
    q[0, 2, :, 3] = (q[0, 2, :, 3] * 4).round() / 4         # (values that are one bf16 term)
    t[0, 2, 130:140, 3] = x
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    jv.full_attn(*(a.to(DEV) for a in (q, k, v)), out=out)
    check()
    s = (q.double() @ k.double().transpose(-1, -2)).clamp(-1e300, 1e300) if value == "lowest" else q.double() @ k.double().transpose(-1, -2)
    ref = torch.softmax(s / 8.0, -1) @ v.double()
    got = out.cpu().double()
    assert torch.equal(got.isfinite(), ref.isfinite())
    f = ref.isfinite()
    assert bool(((got - ref).abs()[f] <= 1e-4 * ref.abs()[f].clamp(min=ref[0, 0].square().mean().sqrt())).all())


@pytest.mark.parametrize("size", [1e-27, 1e-30, 1e-34, 1e-36, 1e-37])
@pytest.mark.parametrize("H,Hg,Wg", [(3, 24, 16), (24, 24, 16)], ids=["multiply-adds", "tensor cores"])
def test_fp32_small_values(jv, H, Hg, Wg, size):
    """V of this size in some channels, or q against a large k: results as accurate as those of other sizes, down to fp32's subnormals (results of
    5e-39, in steps of 1.4e-45)."""
    q, k, v = (t.to(DEV) for t in inputs.custom_qkv(1, H, Hg * Wg, 64, "f32", seed=3770))
    v[..., 5:60] *= size
    v[..., 7] = 0.0
    v[:, 1, 33] = 0.0
    ref = torch.softmax(q.double() @ k.double().transpose(-1, -2) / 8, -1) @ v.double()
    o = jv.full_attn(q, k, v).double()
    for c in (slice(0, 5), slice(5, 60)):
        assert float((o - ref)[..., c].norm() / ref[..., c].norm()) <= 6e-7
    assert bool((o[..., 7] == 0).all())
    o = jv.full_attn(q * size, k * 1e9, v, scale=1 / (8 * size * 1e9)).double()
    assert float((o - ref).norm() / ref.norm()) <= 6e-7


@pytest.mark.parametrize("size", [3e4, 1e5, 1e6, 1e9])
@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("H,Hg,Wg", [(3, 24, 16), (24, 24, 16)], ids=["multiply-adds", "tensor cores"])
def test_fp32_large_scores(jv, H, Hg, Wg, size, sign):
    """q and k of this size: one key takes all of a row's weight.  sign -1: all scores are negative.  Rows whose two largest scores are closer
    than the rounding of a sum of 64 products in 32 bits (64 * 2^-24 of the largest at most) need only be finite."""
    q, k, v = (t.to(DEV) for t in inputs.custom_qkv(1, H, Hg * Wg, 64, "f32", seed=3750))
    q, k = q * size, k * size
    if sign < 0:
        q, k = q.abs(), -k.abs()

    def windows(t):                                          # 8 x 8 windows as heads
        return t.view(1, H, Hg // 8, 8, Wg // 8, 8, 64).transpose(3, 4).reshape(1, -1, 64, 64)

    for o, (a, b, c) in ((jv.full_attn(q, k, v), (q, k, v)), (windows(jv.window_attn(q, k, v, Hg, Wg, 8, 8)), map(windows, (q, k, v)))):
        s = a.double() @ b.double().transpose(-1, -2) / 8
        top = s.topk(2, -1)
        gap = top.values[..., 0] - top.values[..., 1]
        clear = (gap > 64 * 2.0 ** -24 * s.abs().amax(-1)) & (gap > 100)
        assert float(clear.double().mean()) > 0.98
        assert bool(torch.isfinite(o).all())
        want = torch.gather(c, 2, top.indices[..., :1].expand(-1, -1, -1, 64))
        assert float((o - want).abs()[clear].max()) <= 1e-5


@pytest.mark.parametrize("B,H,P,Hg,Wg,win", [(1, 1, 1, 5, 5, 4), (1, 2, 17, 16, 31, 8), (1, 6, 5, 37, 37, 8), (3, 50, 3, 12, 17, 7),
                                             (1, 12, 100, 17, 23, 4), (1, 12, 120, 9, 9, 5), (1, 6, 120, 20, 20, 5), (4, 24, 120, 24, 24, 5), (4, 24, 97, 21, 23, 6)])
def test_fp32_prefix_queries(jv, oracle, B, H, P, Hg, Wg, win):
    """The prefix queries' keys over 4 to 32 groups in clusters of 1 to 8 blocks or over 8 of one block, some of them without a key; windows of 9 to 32 tokens with
    more than 128 keys, few (16 rows to a CTA) and many (32 rows)."""
    q, k, v = inputs.custom_qkv(B, H, P + Hg * Wg, 64, "f32", seed=3800 + P)
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    out.fill_(float("nan"))
    jv.window_attn(*(t.to(DEV) for t in (q, k, v)), Hg, Wg, win, win, out=out, prefix=P)
    check()
    heads = sample_heads(B, H, 4, P)
    qs, ks, vs = _tc_heads(q, k, v, heads)
    o = _tc_heads(out.cpu(), k, v, heads)[0]
    assert rel_err(o, oracle.window_attn(qs, ks, vs, Hg, Wg, win, win, prefix=P)) <= TOL["f32"]


# Windows of up to eight tokens are the kernel of one warp per query row's, with prefix tokens where there are many of them (B = 4) and a window's keys
# are at most 32; their prefix queries are not; windows of nine tokens are one launch of this kernel.
@pytest.mark.parametrize("B,P", [(2, 0), (2, 1), (4, 1), (4, 24), (4, 31), (4, 70)])
@pytest.mark.parametrize("wh,ww", [(1, 1), (2, 2), (2, 4), (8, 1), (3, 3), (1, 9)])
def test_fp32_small_windows(jv, oracle, B, P, wh, ww):
    H, Hg, Wg = 8, 15, 19
    q, k, v = inputs.custom_qkv(B, H, P + Hg * Wg, 64, "f32", seed=3400 + P + wh)
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    out.fill_(float("nan"))
    launches = jv.launch_count()
    jv.window_attn(*(t.to(DEV) for t in (q, k, v)), Hg, Wg, wh, ww, out=out, prefix=P)
    assert jv.launch_count() - launches == (2 if P else 1)
    check()
    heads = sample_heads(B, H, 4, P + wh)
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    assert rel_err(pick(out.cpu()), oracle.window_attn(pick(q), pick(k), pick(v), Hg, Wg, wh, ww, prefix=P)) <= TOL["f32"]


@pytest.mark.parametrize("N", [1, 2, 7, 8, 9])
def test_fp32_short_sequences(jv, oracle, N):
    q, k, v = inputs.custom_qkv(2, 5, N, 64, "f32", seed=3500 + N)
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    out.fill_(float("nan"))
    jv.full_attn(*(t.to(DEV) for t in (q, k, v)), out=out)
    check()
    assert rel_err(out, oracle.full_attn(q, k, v)) <= TOL["f32"]


@pytest.mark.parametrize("N", [31, 33, 64, 65, 97, 128, 129, 225, 256, 257])
def test_fp32_short_rows_of_keys(jv, oracle, N):
    """Tiles of 32 keys over two, four and eight groups: the last group full, ragged and without a key; one key more than they take."""
    q, k, v = inputs.custom_qkv(1, 3, N, 64, "f32", seed=3900 + N)
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    out.fill_(float("nan"))
    jv.full_attn(*(t.to(DEV) for t in (q, k, v)), out=out)
    check()
    assert rel_err(out, oracle.full_attn(q, k, v)) <= TOL["f32"]


@pytest.mark.parametrize("static", [False, True], ids=["squeeze", "static"])
@pytest.mark.parametrize("case", [(1, 1, 0, 1, 1), (1, 2, 0, 70, 1), (2, 3, 5, 11, 13), (1, 12, 1, 32, 32), (2, 2, 3, 3, 130), (2, 12, 0, 32, 32)],
                         ids=lambda c: "x".join(map(str, c)))
def test_fp32_linear_with_convolution(jv, oracle, case, static):
    B, H, P, Hg, Wg = case
    q, k, v = inputs.custom_qkv(B, H, P + Hg * Wg, 64, "f32", seed=3300 + Hg + Wg)
    d = inputs.dwc_weights(H * 64, 18, 3, 3301)                 # R = 18: rows of W2 that no float4 divides
    if static:
        d = {"k": 3, "R": 0, "b2": inputs.normal((H * 64 * 9,), inputs.SEED_BASE + 3302) * 0.2}
    out, check = guarded_empty(q.shape, torch.float32, DEV)
    out.fill_(float("nan"))
    jv.linear_attn(*(t.to(DEV) for t in (q, k, v)), Hg, Wg, dwc=dwc_to_device(d, DEV), out=out, prefix=P)
    check()
    assert rel_err(out, oracle.linear_attn(q, k, v, Hg, Wg, dwc=d, prefix=P)) <= TOL["f32"]
