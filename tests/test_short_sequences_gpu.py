"""Full attention by length and heads.  Below 1024 tokens: at most two tiles on the window kernel (one token, a tile less one, a tile,
a tile and one, two tiles), the rest by heads and tiles on the split-key, the four-tile or the two-tile kernel; q, k, v contiguous and
in a fused activation."""
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


CASES = [(1, 1, 1), (1, 3, 15), (2, 5, 63), (1, 2, 64), (1, 3, 65), (2, 2, 127), (1, 4, 128), (3, 2, 129), (32, 12, 200), (1, 2, 255),
         (2, 80, 256), (1, 2, 257), (40, 2, 257), (40, 2, 385), (20, 4, 511), (80, 1, 513), (80, 1, 640), (80, 1, 770), (40, 1, 1000)]


@pytest.mark.parametrize("fused", [False, True], ids=["bhnd", "fused"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_short_sequences(jv, oracle, case, fused):
    B, H, N = case
    q, k, v = inputs.custom_qkv(B, H, N, 64, "bf16", seed=4100 + N + H)
    if fused:
        act = torch.stack([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2).to(DEV).contiguous()
        dq, dk, dv = (act[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    else:
        dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    for _ in range(2):
        jv.full_attn(dq, dk, dv, out=out)
    check()
    heads = sample_heads(B, H, 5, N)
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    assert rel_err(pick(out.cpu()), oracle.full_attn(pick(q), pick(k), pick(v))) <= TOL["bf16"], case
    assert bool(torch.isfinite(out).all())


# B, H, N: groups of three (the last of a head with two tiles, and whole), the split-key kernel behind a round of the four-tile one, pairs on the two-tile
# kernel, the split-key kernel alone in two rounds
SPLITS = [(1, 16, 2880), (1, 16, 3070), (2, 19, 2048), (2, 19, 1600), (1, 26, 4096), (2, 13, 4000), (1, 12, 3025)]


@pytest.mark.parametrize("case", SPLITS, ids=lambda c: "x".join(map(str, c)))
def test_items_of_three_tiles_and_pieces(jv, oracle, case):
    B, H, N = case
    q, k, v = inputs.custom_qkv(B, H, N, 64, "bf16", seed=4200 + N + H)
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    jv.full_attn(*(t.to(DEV) for t in (q, k, v)), out=out)
    check()
    assert bool(torch.isfinite(out).all())
    heads = [(0, 0), (B - 1, H - 1)]                   # the last head's groups are the ones cut into pieces
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    assert rel_err(pick(out.cpu()), oracle.full_attn(pick(q), pick(k), pick(v))) <= TOL["bf16"], case
