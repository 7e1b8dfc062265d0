"""tcgen05 attention with two CTAs of one row tile per SM (three or more such CTAs per SM): the bits of the form whose CTAs
take two row tiles, and the values of a float64 reference."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    yield torch, dllm
    dllm._check(dllm.lib.dllm_debug_attention_plan(0, 0, 1, 0))


# (B, queries, keys, H, Hkv): one, two and three row tiles, the last one with 1, 44 and 128 rows; one key, whole and ragged key
# tiles, fewer and more than the ring holds; grouped heads whose rows start inside a query
CASES = [(16, 128, 1, 32, 32), (16, 129, 63, 32, 32), (16, 129, 64, 32, 32), (8, 300, 193, 32, 32), (16, 70, 449, 32, 32),
         (4, 512, 1000, 32, 32), (32, 100, 130, 28, 4), (16, 256, 511, 14, 2)]


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("ramp", [False, True], ids=["flat", "growing maxima"])
@pytest.mark.parametrize("B,a,n,H,Hkv", CASES)
def test_two_ctas_per_sm(env, B, a, n, H, Hkv, hd, ramp):
    torch, dllm = env
    gen = torch.Generator(device="cuda").manual_seed(n)
    q = torch.randn(B * a, H * hd, device="cuda", generator=gen).bfloat16()
    k, v = (torch.randn(B, n, Hkv * hd, device="cuda", generator=gen).bfloat16() for _ in range(2))
    if ramp:
        k *= torch.linspace(0.1, 6, n, device="cuda").view(1, n, 1)
    G, tiles = H // Hkv, (a * (H // Hkv) + 127) // 128
    assert tiles * Hkv * B >= 3 * 148                     # enough row tiles for this form
    dllm._check(dllm.lib.dllm_debug_attention_plan(0, 0, 1, 0))
    got = dllm.attention(q, k, v, B, a, n, H, Hkv, hd)
    if tiles > 1:                                         # a lone row tile is shared by two groups there: other sums
        dllm._check(dllm.lib.dllm_debug_attention_plan(1, 0, 1, 2))
        want = dllm.attention(q, k, v, B, a, n, H, Hkv, hd)
        dllm._check(dllm.lib.dllm_debug_attention_plan(0, 0, 1, 0))
        if a * G % 256 == 0 or a * G % 256 > 128:         # (as is an odd last one)
            assert torch.equal(got, want)
    b = B - 1
    qq = q.view(B, a, H, hd)[b].double()
    kk, vv = (t.view(B, n, Hkv, hd)[b].repeat_interleave(G, 1).double() for t in (k, v))
    p = torch.softmax(torch.einsum("ahd,nhd->han", qq, kk) / hd ** 0.5, -1)
    ref = torch.einsum("han,nhd->ahd", p, vv).reshape(a, H * hd)
    got = got.view(B, a, H * hd)[b].double()
    assert float((got - ref).norm() / ref.norm()) < 1e-2  # probabilities and results in bf16: 2^-9 each
