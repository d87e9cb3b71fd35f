"""The kernel generator of the pooled dynamic convolution at its edges: fewer hidden units than a CTA's 32 rows, more than one
128-value stretch of a weight row, more than 1024 channels, one sample and more than a group of eight, several groups
(many samples of many hidden units), weights that no 128-bit load can read, static kernels off 16 bytes; prefix tokens
beside the generator (one, the most it takes, none of them with static kernels) and behind it (one more)."""
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


def _off(t):
    """A copy of t whose data starts 4 bytes off a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=DEV)
    view = buf[1:1 + t.numel()].view(t.shape)
    view.copy_(t)
    return view


CASES = [  # B, H, P, Hg, Wg, R (0: static), k, weights off 16 bytes
    (1, 1, 0, 5, 7, 1, 3, False),
    (9, 2, 0, 6, 18, 20, 3, False),
    (1, 6, 1, 37, 37, 48, 3, False),
    (2, 3, 16, 9, 20, 18, 3, False),
    (2, 3, 17, 9, 20, 36, 3, False),
    (1, 24, 5, 11, 19, 192, 3, False),
    (33, 2, 2, 8, 9, 1024, 3, False),
    (3, 2, 0, 12, 13, 140, 5, False),
    (2, 4, 3, 10, 17, 64, 3, True),
    (2, 4, 0, 10, 17, 33, 5, True),
    (2, 3, 5, 10, 17, 0, 3, False),
    (2, 3, 5, 10, 17, 0, 3, True),
    (2, 3, 0, 10, 17, 0, 5, True),
]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_generator(jv, oracle, case, dtype):
    B, H, P, Hg, Wg, R, ksz, off = case
    q, k, v = inputs.custom_qkv(B, H, P + Hg * Wg, 64, dtype, seed=6100 + Hg + Wg + R)
    if R:
        d = inputs.dwc_weights(H * 64, R, ksz, 6101)
        d["b1"] = 0.1 * inputs.normal((R,), inputs.SEED_BASE + 6102)
    else:
        d = {"k": ksz, "R": 0, "b2": 0.2 * inputs.normal((H * 64 * ksz * ksz,), inputs.SEED_BASE + 6103)}
    dd = {key: ((_off(t) if off else t.to(DEV)) if hasattr(t, "to") else t) for key, t in d.items()}
    dq, dk, dv = (t.to(DEV) for t in (q, k, v))
    out, check = guarded_empty(q.shape, dq.dtype, DEV)
    ws = jv.alloc_workspace("L", jv.make_shape(dq, Hg, Wg, P), jv.make_dwc(dd, DEV), DEV)
    for _ in range(3):
        ws.fill_(255)                                  # NaN: what is read before it is written shows
        out.fill_(float("nan"))
        jv.linear_attn(dq, dk, dv, Hg, Wg, dwc=dd, out=out, ws=ws, prefix=P)
    check()
    assert rel_err(out, oracle.linear_attn(q, k, v, Hg, Wg, dwc=d, prefix=P)) <= TOL[dtype], case
