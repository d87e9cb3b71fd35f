"""Full attention on every cut that its rules make of a call: the four-tile kernel in whole groups of four or three query tiles, with the last
round in pieces of two tiles or one, and the two-tile kernel; by tile counts per head that leave every remainder.  (Few heads take the
split-key kernel at these lengths: tests/test_split_keys_gpu.py.)  Each on ordinary scores and on scores that make the
running reference move again and again, with a jump far beyond 2^64 in the middle.  Reference: the formula in fp64, all heads.

Bound of every value: probabilities are rounded to bf16 (each off by 2^-8 of itself at most), a part of the exponentials is a polynomial (7.5e-5, in
the sum of the row, too), the result is rounded to bf16: |o - r| <= (2^-8 + 2e-4) sum_j p_j |v_j| + 2^-8 |r|.  (The bar of 2e-2 rms that
samples of heads are held to elsewhere is a typical maximum, not a bound: over all 1.6 million values of a case here 2.2e-2
occurs.)  The rms of the error is held to 3e-3 of the result's as everywhere."""
import pytest
import torch

from tests._util import RMS_TOL_BF16, guarded_empty

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def jv():
    from paper_2605_26636_b200 import jetvit
    jetvit.lib()
    yield jetvit
    assert jetvit.device_status() == jetvit.JV_OK


CASES = [  # B, H, N
    (5, 15, 400), (2, 19, 1207), (1, 38, 1329), (2, 15, 1573),                # groups of four: 4, 10, 11 and 13 tiles a head
    (5, 15, 300), (2, 19, 900), (3, 11, 1085), (2, 15, 1207), (3, 16, 1024),  # groups of three: 3, 8, 9, 10 and 8 tiles
    (6, 31, 300), (6, 31, 400), (3, 22, 1085), (2, 31, 1207),                 # groups of four, the last round in pairs: 3, 4, 9 and 10 tiles
    (1, 149, 300), (3, 20, 1085), (4, 15, 1207),                              # the last round in single tiles: 3, 9 and 10
    (2, 12, 1024), (2, 19, 1600), (5, 16, 513), (8, 8, 330),                  # pairs on the two-tile kernel: 8, 13, 5 and 3
]


@pytest.mark.parametrize("rising", [False, True], ids=["plain", "rising"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_full_attention_routes(jv, case, rising):
    B, H, N = case
    gen = torch.Generator(device=DEV).manual_seed(4700 + N + H)
    q, k, v = (torch.randn((B, H, N, 64), generator=gen, device=DEV).bfloat16() for _ in range(3))
    if rising:                                           # keys lean more and more towards the first query; one sharply
        u = q[:, :, :1].float()
        k = (k.float() + 6.0 * torch.linspace(0.0, 1.0, N, device=DEV).view(N, 1) * u).bfloat16()
        k[:, :, N // 2] = (40.0 * u[:, :, 0]).bfloat16()
    out, check = guarded_empty(q.shape, torch.bfloat16, DEV)
    out.fill_(float("nan"))
    launches = jv.launch_count()
    jv.full_attn(q, k, v, out=out)
    assert jv.launch_count() - launches == 1
    check()
    err = ref = 0.0
    for b in range(B):
        p = torch.softmax(q[b].double() @ k[b].double().transpose(1, 2) / 8, -1)
        r = p @ v[b].double()
        d = (out[b].double() - r).abs()
        bound = (2.0 ** -8 + 2e-4) * (p @ v[b].double().abs()) + 2.0 ** -8 * r.abs()
        assert bool((d <= bound).all()), (case, b, float((d / bound).max()))
        err, ref = err + float((d * d).sum()), ref + float((r * r).sum())
    assert (err / ref) ** 0.5 <= RMS_TOL_BF16, case
