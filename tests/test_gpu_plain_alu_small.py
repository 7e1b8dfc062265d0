"""The plain-ALU forms for launches that would leave the chip idle give the bits of the others: 8 x 16 tiles of the GEMM
(several chunks of a warp in flight) and one query per CTA of the attention."""
import numpy as np
import pytest

from paper_2506_06295_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    return torch, dllm


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("K", [31, 256, 257, 512, 688, 767, 769, 1537])     # 32-wide chunks by eight warps, up to three each in flight
@pytest.mark.parametrize("M,N", [(1, 15), (8, 17), (9, 256)])
def test_small_gemm_tiles_give_the_bits_of_large_ones(env, dtype, K, M, N):
    torch, dllm = env
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    A = torch.from_numpy(synth.random_normal((3000, K), seed=7)).cuda().to(td)
    W = torch.from_numpy(synth.random_normal((N, K), seed=8, std=0.05)).cuda().to(td)
    small, many = dllm.gemm_simt(A[:M].contiguous(), W), dllm.gemm_simt(A, W)
    assert torch.equal(small, many[:M])
    want = A[:M].double() @ W.double().T
    assert float((small.double() - want).norm() / want.norm()) < 2e-6       # fp32 sums of K products


@pytest.mark.parametrize("n,hd,Hkv", [(1, 32, 4), (33, 64, 4), (300, 64, 2), (96, 96, 4), (257, 128, 1)])
def test_one_query_per_cta_gives_the_bits_of_four(env, n, hd, Hkv):
    torch, dllm = env
    H, a, few = 4, 100, 30                                                  # 400 (query, head) pairs, and 120: one wave
    gen = torch.Generator(device="cuda").manual_seed(n)
    q = torch.randn(a, H * hd, device="cuda", generator=gen)
    k, v = (torch.randn(1, n, Hkv * hd, device="cuda", generator=gen) for _ in range(2))
    all_ = dllm.attention(q, k, v, 1, a, n, H, Hkv, hd)
    one = dllm.attention(q[:few].contiguous(), k, v, 1, few, n, H, Hkv, hd)
    assert torch.equal(one, all_[:few])
    kk, vv = (t.view(n, Hkv, hd).repeat_interleave(H // Hkv, 1).double() for t in (k, v))
    p = torch.softmax(torch.einsum("ahd,nhd->han", q.view(a, H, hd).double(), kk) / hd ** 0.5, -1)
    want = torch.einsum("han,nhd->ahd", p, vv).reshape(a, H * hd)
    assert float((all_.double() - want).norm() / want.norm()) < 1e-5       # fp32 sums of n products
