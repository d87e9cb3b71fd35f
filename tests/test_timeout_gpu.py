"""The bounded waits of the tensor-core kernels, driven to their limit without hanging or
faulting anything: jv_selftest_wait_timeout enqueues a one-warp kernel that waits (through the
mixers' own bounded wait, limit 1 ms) on a barrier nothing completes.  Checked: the wait gives
up and the kernel returns; jv_device_status reports JV_ERR_TIMEOUT once and JV_OK afterwards;
tensor-core mixer calls enqueued while the status word is set leave their output untouched
(the behaviour include/jetvit.h documents); the next calls compute correctly."""
import pytest
import torch

from paper_2605_26636_b200 import inputs
from tests._util import TOL, dwc_to_device, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    return jetvit


def test_a_wait_that_runs_out_sets_the_status_and_nothing_hangs(jv, oracle):
    Hg, Wg = 40, 32                                   # two heads of 1280 tokens, or of 512: F with its keys over four slots
    qh, kh, vh = inputs.custom_qkv(1, 2, Hg * Wg, 64, "bf16", seed=31)
    q, k, v = (t.to(DEV) for t in (qh, kh, vh))
    qs, ks, vs = (t[:, :, :512].contiguous() for t in (q, k, v))
    dh = inputs.dwc_weights(2 * 64, 16, 3, 32)
    d = dwc_to_device(dh, DEV)
    calls = {
        "L": lambda out: jv.linear_attn(q, k, v, Hg, Wg, out=out),
        "L+dwc": lambda out: jv.linear_attn(q, k, v, Hg, Wg, dwc=d, out=out),
        "W": lambda out: jv.window_attn(q, k, v, Hg, Wg, 16, 16, out=out),
        "F": lambda out: jv.full_attn(q, k, v, out=out),
        "F short": lambda out: jv.full_attn(qs, ks, vs, out=out.view(-1)[:qs.numel()].view(qs.shape)),
    }
    assert jv.device_status() == jv.JV_OK
    good = {}
    for name, fn in calls.items():
        good[name] = torch.empty_like(q)
        fn(good[name])
    assert jv.device_status() == jv.JV_OK

    gave_up = torch.zeros(1, dtype=torch.int32, device=DEV)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    jv.selftest_wait_timeout(1000, gave_up)           # 1 ms
    t1.record()
    # calls enqueued while the status word is set: their kernels leave at once, o keeps the canary
    outs = {}
    for name, fn in calls.items():
        outs[name] = torch.full_like(q, 1234.5)
        fn(outs[name])
    torch.cuda.synchronize()
    assert int(gave_up.item()) == 1
    assert 0.9 <= t0.elapsed_time(t1) < 200.0         # the wait lasted about its limit, not the 2 s default
    for name, o in outs.items():
        assert bool((o == 1234.5).all()), f"{name}: output written while the status word was set"
    assert jv.device_status() == jv.JV_ERR_TIMEOUT    # reported once ...
    assert jv.device_status() == jv.JV_OK             # ... and cleared
    # the context is intact and the next calls compute what they computed before, and what the oracle says
    for name, fn in calls.items():
        o = torch.full_like(q, 1234.5)
        fn(o)
        torch.cuda.synchronize()
        n = qs.numel() if name == "F short" else q.numel()
        assert torch.equal(o.view(-1)[:n], good[name].view(-1)[:n]), name
    assert rel_err(good["L+dwc"], oracle.linear_attn(qh, kh, vh, Hg, Wg, dwc=dh)) <= TOL["bf16"]
    assert rel_err(good["F"], oracle.full_attn(qh, kh, vh)) <= TOL["bf16"]
    assert jv.device_status() == jv.JV_OK


def test_every_tensor_core_kernel_leaves_at_once(jv):
    """One call for each of the kernels that look at the status word, twice while it is set (tensor memory that the first one had not given back
    would make the second one wait until its limit): the output keeps its contents, the call after the word has been
    cleared computes what it computed before."""
    def qkv(B, H, N, D=64, seed=0):
        return tuple(t.to(DEV) for t in inputs.custom_qkv(B, H, N, D, "bf16", seed=500 + seed))

    def proj(B, N, H):
        C = 64 * H
        x = inputs.normal((B, N, C), 5100 + N, "bf16").to(DEV)
        (w, b), (wo, bo) = inputs.proj_weights(3 * C, C, 5200), inputs.proj_weights(C, C, 5201)
        return x, w.to(DEV), b.to(DEV), wo.to(DEV), bo.to(DEV)

    d = dwc_to_device(inputs.dwc_weights(4 * 64, 16, 3, 501), DEV)
    calls = {}

    def mixer(name, q, fn):
        calls[name] = (lambda o: fn(o[0]), [torch.empty_like(q)])

    q1, k1, v1 = qkv(1, 48, 1024, seed=1)             # 96 groups of four query tiles
    mixer("F, four-tile kernel", q1, lambda o: jv.full_attn(q1, k1, v1, out=o))
    q2, k2, v2 = qkv(1, 24, 1024, seed=2)             # 96 pairs
    mixer("F, two-tile kernel", q2, lambda o: jv.full_attn(q2, k2, v2, out=o))
    q3, k3, v3 = qkv(2, 20, 2100, seed=3)
    mixer("F, keys over four slots behind a round of the four-tile kernel", q3, lambda o: jv.full_attn(q3, k3, v3, out=o))
    q4, k4, v4 = qkv(1, 300, 200, seed=4)
    mixer("F, window kernel", q4, lambda o: jv.full_attn(q4, k4, v4, out=o))
    q5, k5, v5 = qkv(1, 4, 5 + 40 * 36, seed=5)
    for win in (8, 16, 32):
        mixer(f"W {win} with prefix tokens", q5, lambda o, win=win: jv.window_attn(q5, k5, v5, 40, 36, win, win, out=o, prefix=5))
    mixer("L with prefix tokens", q5, lambda o: jv.linear_attn(q5, k5, v5, 40, 36, dwc=d, out=o, prefix=5))
    q6, k6, v6 = qkv(2, 8, 40 * 30, 128, seed=6)
    mixer("F, head_dim 128", q6, lambda o: jv.full_attn(q6, k6, v6, out=o))
    mixer("W, head_dim 128", q6, lambda o: jv.window_attn(q6, k6, v6, 40, 30, 16, 16, out=o))
    mixer("L, head_dim 128", q6, lambda o: jv.linear_attn(q6, k6, v6, 40, 30, out=o))
    q7, k7, v7 = (t.to(DEV) for t in inputs.custom_qkv(1, 24, 5 + 33 * 29, 64, "f32", seed=507))
    mixer("F, fp32", q7, lambda o: jv.full_attn(q7, k7, v7, out=o))
    for win in (8, 16):
        mixer(f"W {win} with prefix tokens, fp32", q7, lambda o, win=win: jv.window_attn(q7, k7, v7, 33, 29, win, win, out=o, prefix=5))
    for name, (B, N, H) in (("one CTA", (1, 300, 6)), ("pairs", (3, 3100, 8))):
        x, w, b, wo, bo = proj(B, N, H)
        outs = [torch.empty((B, H, N, 64), dtype=torch.bfloat16, device=DEV) for _ in range(3)]
        calls[f"qkv_proj, {name}"] = (lambda o, x=x, w=w, b=b, H=H, N=N: jv.qkv_proj(x, w, b, H, 1, N, out=tuple(o)), outs)
        src = torch.randn((B, H, N, 64), device=DEV).bfloat16()
        calls[f"out_proj, {name}"] = (lambda o, src=src, wo=wo, bo=bo, N=N: jv.out_proj(src, wo, bo, 1, N, out=o[0]), [torch.empty_like(x)])

    assert jv.device_status() == jv.JV_OK
    good = {}
    for name, (fn, outs) in calls.items():
        fn(outs)
        good[name] = [o.clone() for o in outs]
    assert jv.device_status() == jv.JV_OK
    jv.selftest_wait_timeout(1000)
    for fn, outs in calls.values():
        for o in outs:
            o.fill_(1234.5)
        fn(outs)
        fn(outs)
    torch.cuda.synchronize()
    for name, (fn, outs) in calls.items():
        assert all(bool((o == 1234.5).all()) for o in outs), name
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    for name, (fn, outs) in calls.items():
        fn(outs)
        assert all(torch.equal(a, b) for a, b in zip(outs, good[name])), name
    assert jv.device_status() == jv.JV_OK


def test_selftest_rejects_bad_limits(jv):
    with pytest.raises(jv.JetVitError):
        jv.selftest_wait_timeout(0)
    with pytest.raises(jv.JetVitError):
        jv.selftest_wait_timeout(5_000_000)
    assert jv.device_status() == jv.JV_OK


def test_windows_that_leave_at_once_end_behind_their_prefix_queries(jv):
    """Window attention with prefix tokens while the status word is set: the windows' launch, which runs beside that of the prefix queries,
    leaves at once.  It must not be complete before the other one is, or what is enqueued behind the call could
    be overwritten by it."""
    H, Hg, Wg, P = 6, 37, 37, 5
    q, k, v = (t.to(DEV) for t in inputs.custom_qkv(1, H, P + Hg * Wg, 64, "bf16", seed=37))
    o = torch.empty_like(q)
    assert jv.device_status() == jv.JV_OK
    jv.selftest_wait_timeout(1000)
    for _ in range(20):
        jv.window_attn(q, k, v, Hg, Wg, 16, 16, out=o, prefix=P)
        o.fill_(1234.5)
        seen = o.clone()
        assert bool((seen == 1234.5).all()) and bool((o == 1234.5).all())
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    assert jv.device_status() == jv.JV_OK


@pytest.mark.parametrize("H", [8, 21, 50])                # clusters of eight, seven and two CTAs
def test_head_dim_128_state_pass_while_the_word_is_set(jv, oracle, H):
    """The CTAs of a cluster exchange their partial states also when they have given up, and each stays until what is sent to it has
    landed: many such calls in a row leave the device in order and the output alone."""
    Hg, Wg = 31, 21
    qh, kh, vh = inputs.custom_qkv(1, H, Hg * Wg, 128, "bf16", seed=128 + H)
    q, k, v = (t.to(DEV) for t in (qh, kh, vh))
    o = torch.full_like(q, 1234.5)
    assert jv.device_status() == jv.JV_OK
    jv.selftest_wait_timeout(1000)
    for _ in range(20):
        jv.linear_attn(q, k, v, Hg, Wg, out=o)
    torch.cuda.synchronize()
    assert bool((o == 1234.5).all())
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    jv.linear_attn(q, k, v, Hg, Wg, out=o)
    assert rel_err(o[:, :2], oracle.linear_attn(qh[:, :2], kh[:, :2], vh[:, :2], Hg, Wg)) <= TOL["bf16"]
    assert jv.device_status() == jv.JV_OK


@pytest.mark.parametrize("P", [1, 5, 16, 20])             # 20: the linear block's prefix rows by the apply pass, W on the kernel of large windows
def test_prefix_rows_stay_while_the_word_is_set(jv, oracle, P):
    """The rows of the prefix tokens have kernels of their own in W and in the linear block with a convolution; they leave o alone as the
    others do.  The linear block's scratch holds NaN: its state pass leaves without writing it."""
    H, Hg, Wg = 4, 33, 29
    qh, kh, vh = inputs.custom_qkv(1, H, P + Hg * Wg, 64, "bf16", seed=90 + P)
    q, k, v = (t.to(DEV) for t in (qh, kh, vh))
    dh = inputs.dwc_weights(H * 64, 16, 3, 91)
    d = dwc_to_device(dh, DEV)
    static = {"k": 3, "R": 0, "b2": d["b2"]}
    ws = jv.alloc_workspace("L", jv.make_shape(q, Hg, Wg, P), jv.make_dwc(d, DEV), DEV)
    calls = [lambda o: jv.linear_attn(q, k, v, Hg, Wg, dwc=d, out=o, ws=ws, prefix=P),
             lambda o: jv.linear_attn(q, k, v, Hg, Wg, dwc=static, out=o, ws=ws, prefix=P),
             lambda o: jv.linear_attn(q, k, v, Hg, Wg, out=o, ws=ws, prefix=P),
             lambda o: jv.window_attn(q, k, v, Hg, Wg, 16, 16, out=o, prefix=P),
             lambda o: jv.window_attn(q, k, v, Hg, Wg, 8, 8, out=o, prefix=P)]
    assert jv.device_status() == jv.JV_OK
    ws.fill_(255)
    jv.selftest_wait_timeout(1000)
    outs = [torch.full_like(q, 1234.5) for _ in calls]
    for fn, o in zip(calls, outs):
        fn(o)
        fn(o)
    torch.cuda.synchronize()
    for i, o in enumerate(outs):
        assert bool((o == 1234.5).all()), (i, (o != 1234.5).nonzero()[:4].tolist())
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    assert rel_err(calls[0](outs[0]), oracle.linear_attn(qh, kh, vh, Hg, Wg, dwc=dh, prefix=P)) <= TOL["bf16"]
    assert rel_err(calls[3](outs[3]), oracle.window_attn(qh, kh, vh, Hg, Wg, 16, 16, prefix=P)) <= TOL["bf16"]
    assert jv.device_status() == jv.JV_OK


@pytest.mark.parametrize("H,stays", [(16, True), (1, False)], ids=["tensor cores", "multiply-adds"])
@pytest.mark.parametrize("P,win", [(1, 8), (5, 16), (40, 8)])
def test_fp32_windows_stay_whole_while_the_word_is_set(jv, oracle, H, stays, P, win):
    """Window attention of fp32 tensors, prefix rows and windows: large calls leave all of o alone, small ones write all of it."""
    Hg, Wg = (33, 29) if stays else (13, 11)
    qh, kh, vh = inputs.custom_qkv(1, H, P + Hg * Wg, 64, "f32", seed=93 + P)
    q, k, v = (t.to(DEV) for t in (qh, kh, vh))
    ref = oracle.window_attn(qh, kh, vh, Hg, Wg, win, win, prefix=P)
    o = torch.full_like(q, 1234.5)
    assert jv.device_status() == jv.JV_OK
    jv.selftest_wait_timeout(1000)
    for _ in range(2):
        jv.window_attn(q, k, v, Hg, Wg, win, win, out=o, prefix=P)
    torch.cuda.synchronize()
    assert bool((o == 1234.5).all()) if stays else rel_err(o, ref) <= TOL["f32"]
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    assert rel_err(jv.window_attn(q, k, v, Hg, Wg, win, win, out=o, prefix=P), ref) <= TOL["f32"]
    assert jv.device_status() == jv.JV_OK


@pytest.mark.parametrize("k,R,token_wise", [(5, 16, 0), (3, 64, 1)])
def test_convolutions_that_add_to_the_output_stay_away_while_the_word_is_set(jv, oracle, k, R, token_wise):
    """5 x 5 kernels and token-wise ones are a pass of their own that reads o and adds to it."""
    H, Hg, Wg = 2, 24, 20
    qh, kh, vh = inputs.custom_qkv(1, H, Hg * Wg, 64, "bf16", seed=95 + k)
    q, kk, v = (t.to(DEV) for t in (qh, kh, vh))
    dh = dict(inputs.dwc_weights(H * 64, R, k, 96), token_wise=token_wise)
    d = dwc_to_device(dh, DEV)
    o = torch.full_like(q, 1234.5)
    assert jv.device_status() == jv.JV_OK
    jv.selftest_wait_timeout(1000)
    jv.linear_attn(q, kk, v, Hg, Wg, dwc=d, out=o)
    torch.cuda.synchronize()
    assert bool((o == 1234.5).all())
    assert jv.device_status() == jv.JV_ERR_TIMEOUT
    ref = oracle.linear_attn(qh, kh, vh, Hg, Wg, dwc=dh)
    # o is rounded to bf16 twice on these paths: the bars of tests/test_parity_gpu.py for them
    assert rel_err(jv.linear_attn(q, kk, v, Hg, Wg, dwc=d, out=o), ref, rms_tol=4.5e-3) <= TOL["bf16"]
    assert jv.device_status() == jv.JV_OK
