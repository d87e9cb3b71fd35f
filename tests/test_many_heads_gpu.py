"""The linear block with more heads than the state pass has CTAs at two to an SM (its rings are then half as deep): fewer tiles than a
ring holds, the last one of a few tokens, and several times round it; two chunks, one or three spans per head; prefix tokens, strided inputs."""
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


@pytest.mark.parametrize("conv", [False, True], ids=["none", "squeeze"])
@pytest.mark.parametrize("case", [(50, 6, 0, 5, 13, True), (99, 3, 1, 8, 8, False), (25, 12, 0, 24, 24, True), (31, 10, 5, 17, 23, False), (20, 8, 3, 32, 33, False),
                                  (10, 16, 0, 53, 52, False), (10, 16, 2, 65, 66, False)],
                         ids=lambda c: "x".join(map(str, c)))
def test_many_heads(jv, oracle, case, conv):
    B, H, P, Hg, Wg, fused = case
    N = P + Hg * Wg
    q, k, v = inputs.custom_qkv(B, H, N, 64, "bf16", seed=5200 + N + H)
    dwc = inputs.dwc_weights(H * 64, 8 * H, 3, seed=5300 + H) if conv else None
    if fused:
        act = torch.stack([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2).to(DEV).contiguous()
        dq, dk, dv = (act[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    else:
        dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    for _ in range(2):
        jv.linear_attn(dq, dk, dv, Hg, Wg, dwc=dwc_to_device(dwc, DEV) if conv else None, out=out, prefix=P)
    check()
    assert bool(torch.isfinite(out).all())
    for b in (0, B - 1):                              # whole samples: the generator sees every channel of one
        ref = oracle.linear_attn(q[b:b + 1], k[b:b + 1], v[b:b + 1], Hg, Wg, dwc=dwc, prefix=P)
        assert rel_err(out[b:b + 1].cpu(), ref) <= TOL["bf16"], (case, b)
