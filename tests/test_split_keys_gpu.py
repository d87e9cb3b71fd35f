"""Full attention with at most a query tile per SM: the keys of a tile over four slots.  One box of keys to three of the slots and two
to the fourth (the last of one key), whole boxes, ragged last tiles and boxes, more boxes than a slot's rings hold, as many
tiles as SMs; scores so spread that the slots' maxima differ widely and a slot's reference moves; tiles left over by whole rounds
of the four-tile kernel, with and without tiles behind the last group of four of a head."""
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


CASES = [(1, 1, 257, 1), (2, 3, 320, 1), (1, 5, 321, 1), (1, 6, 1370, 1), (1, 6, 1370, 6), (1, 37, 512, 1), (1, 21, 895, 4),
         (2, 1, 9400, 1), (1, 12, 7000, 1), (2, 12, 4088, 1)]


@pytest.mark.parametrize("fused", [False, True], ids=["bhnd", "fused"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_split_keys(jv, oracle, case, fused):
    B, H, N, spread = case
    q, k, v = inputs.custom_qkv(B, H, N, 64, "bf16", seed=4300 + N + H)
    q = q * spread                                    # small whole factors: exact in bf16 up to one rounding, on both sides
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
    assert bool(torch.isfinite(out).all())
    rows = list(range(N)) if N < 2000 else list(range(130)) + list(range(N - 700, N))
    heads = [(0, 0), (B - 1, H - 1)]
    pick = lambda t: torch.stack([t[b, h] for b, h in heads]).unsqueeze(0)
    assert rel_err(pick(out.cpu())[:, :, rows], oracle.full_attn(pick(q)[:, :, rows], pick(k), pick(v))) <= TOL["bf16"], case
