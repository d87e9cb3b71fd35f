"""The projections on pairs of CTAs: an odd number of token tiles (the last pair has one tile only, of the last batch element),
a ragged last tile per batch element, feature tiles that are full, a quarter full and half full."""
import pytest
import torch

from paper_2605_26636_b200 import inputs
from tests._util import TOL, guarded_empty, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


@pytest.mark.parametrize("H,which", [(7, "qkv"), (24, "out"), (23, "out")])
def test_projection_on_pairs(jv, oracle, H, which):
    B, Hg, Wg = 3, 50, 62                              # 25 token tiles per batch element, 28 tokens in the last
    N, C = Hg * Wg, 64 * H
    x = inputs.normal((B, N, C) if which == "qkv" else (B, H, N, 64), inputs.SEED_BASE + 9900 + H, "bf16")
    w, b = inputs.proj_weights(3 * C if which == "qkv" else C, C, 9901 + H)
    dx, dw, db = x.to(DEV), w.to(DEV), b.to(DEV)
    shapes = [(B, H, N, 64)] * 3 if which == "qkv" else [(B, N, C)]
    outs, checks = zip(*[guarded_empty(s, torch.bfloat16, DEV) for s in shapes])
    for _ in range(3):
        for o in outs:
            o.fill_(float("nan"))
        if which == "qkv":
            jv.qkv_proj(dx, dw, db, H, Hg, Wg, out=outs)
        else:
            jv.out_proj(dx, dw, db, Hg, Wg, out=outs[0])
    for check in checks:
        check()
    for bi in (0, 2):
        sl = slice(bi, bi + 1)
        refs = oracle.qkv_proj(x[sl], w, b, H) if which == "qkv" else [oracle.out_proj(x[sl], w, b)]
        for got, want in zip(outs, refs):
            assert rel_err(got[sl], want) <= TOL["bf16"]
    assert all(bool(torch.isfinite(o).all()) for o in outs)


def test_pairs_one_behind_the_other(jv):
    """Many launches of pairs in a row, each reading what the one before wrote: no CTA of a pair may leave while the other's commits are
    still to arrive in it, nor start on tensor memory that is not free yet.  All rounds give the same bits."""
    B, H, Hg, Wg = 3, 12, 50, 62
    C = 64 * H
    x = inputs.normal((B, Hg * Wg, C), inputs.SEED_BASE + 9950, "bf16").to(DEV)
    w, b = (t.to(DEV) for t in inputs.proj_weights(3 * C, C, 9951))
    wo, bo = (t.to(DEV) for t in inputs.proj_weights(C, C, 9952))
    qkv = jv.qkv_proj(x, w, b, H, Hg, Wg)
    y = jv.out_proj(qkv[0], wo, bo, Hg, Wg)
    ref = [t.clone() for t in (*qkv, y)]
    for _ in range(50):
        jv.qkv_proj(x, w, b, H, Hg, Wg, out=qkv)
        jv.out_proj(qkv[0], wo, bo, Hg, Wg, out=y)
    for got, want in zip((*qkv, y), ref):
        assert torch.equal(got, want)
