"""Calls enqueued one behind the other without a synchronisation, each on what the one before it wrote, over the same buffers with
other values every time.  A kernel is launched while the one ahead of it drains; one that read its inputs too early would find
the values of the pass before.  Every kernel is deterministic, so the outputs are those of the same chain run
one call at a time, bit for bit; the last one is checked against the oracle."""
import pytest
import torch

from paper_2605_26636_b200 import inputs
from tests._util import TOL, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PASSES = 6


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


def run_passes(chain, sources, sync):
    """chain(source, step) for every source, step() behind every call; returns copies of all that it yields."""
    outs = []
    for src in sources:
        for o in chain(src, torch.cuda.synchronize if sync else lambda: None):
            outs.append(o.clone())
    torch.cuda.synchronize()
    return outs


def check(chain, sources):
    ref = run_passes(chain, sources, True)
    for rep in range(3):
        got = run_passes(chain, sources, False)
        for i, (a, r) in enumerate(zip(got, ref)):
            assert torch.equal(a, r), (rep, i)
    return ref


# Window attention with prefix tokens behind its projection: the prefix queries' launch beside the windows (6 heads of 37 x 37
# tokens) and ahead of them (32 heads of 64 x 64 tokens fill the chip; 20 prefix tokens: the kernel of large windows)
@pytest.mark.parametrize("B,H,Hg,Wg,P", [(1, 6, 37, 37, 1), (2, 16, 64, 64, 5), (1, 2, 24, 24, 20)])
def test_block_with_prefix_tokens(jv, oracle, B, H, Hg, Wg, P):
    N, C = P + Hg * Wg, 64 * H
    xs = [inputs.normal((B, N, C), 4100 + i, "bf16").to(DEV) for i in range(PASSES)]
    w, b = (t.to(DEV) for t in inputs.proj_weights(3 * C, C, 4201))
    wo, bo = (t.to(DEV) for t in inputs.proj_weights(C, C, 4202))
    qkv = tuple(torch.empty((B, H, N, 64), dtype=torch.bfloat16, device=DEV) for _ in range(3))
    o, y = torch.empty_like(qkv[0]), torch.empty_like(xs[0])

    def chain(x, step):
        jv.qkv_proj(x, w, b, H, Hg, Wg, out=qkv, prefix=P)
        step()
        jv.window_attn(*qkv, Hg, Wg, 16, 16, out=o, prefix=P)
        step()
        jv.out_proj(o, wo, bo, Hg, Wg, out=y, prefix=P)
        step()
        return o, y

    ref = check(chain, xs)
    q, k, v = (t[:1, :2].cpu() for t in qkv)               # of the last pass
    assert rel_err(ref[-2][:1, :2], oracle.window_attn(q, k, v, Hg, Wg, 16, 16, prefix=P)) <= TOL["bf16"]


def test_full_attention_split_behind_whole_rounds(jv, oracle):
    """40 heads of 17 query tiles: one whole round of the four-tile kernel and, beside its end, the split-key kernel on what is left.  The second
    call reads what both of the first one's launches wrote."""
    B, H, N = 2, 20, 2100
    q, k, v = (t.to(DEV) for t in inputs.custom_qkv(B, H, N, 64, "bf16", seed=430))
    sources = [torch.roll(q, 7 * i, dims=2) for i in range(PASSES)]
    o1, o2 = torch.empty_like(q), torch.empty_like(q)
    launches = jv.launch_count()
    jv.full_attn(q, k, v, out=o1)
    assert jv.launch_count() - launches == 2

    def chain(src, step):
        jv.full_attn(src, k, v, out=o1)
        step()
        jv.full_attn(o1, k, src, out=o2)
        step()
        return o1, o2

    ref = check(chain, sources)
    pick = lambda t: t[1:, 19:].cpu()
    assert rel_err(pick(ref[-1]), oracle.full_attn(pick(ref[-2]), pick(k), pick(sources[-1]))) <= TOL["bf16"]


@pytest.mark.parametrize("dtype,D,H,Hg,Wg,P", [("f32", 64, 6, 37, 37, 5), ("f32", 64, 12, 16, 16, 0), ("bf16", 128, 8, 32, 33, 0), ("bf16", 128, 3, 9, 7, 0)])
def test_one_mixer_behind_the_other(jv, oracle, dtype, D, H, Hg, Wg, P):
    """Window, linear (fp32: with generated kernels) and full attention, each on the one before, on the fp32 kernels and at head_dim 128."""
    N = P + Hg * Wg
    q, k, v = (t.to(DEV) for t in inputs.custom_qkv(1, H, N, D, dtype, seed=440 + N))
    d = {a: (t.to(DEV) if hasattr(t, "to") else t) for a, t in inputs.dwc_weights(H * D, 48, 3, 441).items()} if dtype == "f32" else None
    sources = [torch.roll(q, 5 * i, dims=2) for i in range(PASSES)]
    outs = [torch.empty_like(q) for _ in range(3)]

    def chain(src, step):
        jv.window_attn(src, k, v, Hg, Wg, 16, 16, out=outs[0], prefix=P)
        step()
        jv.linear_attn(src, k, outs[0], Hg, Wg, dwc=d, out=outs[1], prefix=P)
        step()
        jv.full_attn(src, k, outs[1], out=outs[2])
        step()
        return outs

    ref = check(chain, sources)
    src, o1, o2, o3 = (t[:, :2].cpu() for t in (sources[-1], *ref[-3:]))
    kk, vv = k[:, :2].cpu(), v[:, :2].cpu()
    assert rel_err(o1, oracle.window_attn(src, kk, vv, Hg, Wg, 16, 16, prefix=P)) <= TOL[dtype]
    if d is None:
        assert rel_err(o2, oracle.linear_attn(src, kk, o1, Hg, Wg, prefix=P)) <= TOL[dtype]
    assert rel_err(o3, oracle.full_attn(src, kk, o2)) <= TOL[dtype]
