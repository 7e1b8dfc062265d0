"""Gate / up projection of few rows against weights whose rows lie a multiple of 8 KB apart: every other pair of weight tiles
walks the k range from its middle.  Against float64, and against the same product in two activation tiles, which walks every
tile from its start: the same bits in the tiles that are not turned, another order of the same sums in the others."""
import numpy as np
import pytest

from paper_2506_06295_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,tile", [(1, 32), (64, 64), (65, 128), (128, 128)])
@pytest.mark.parametrize("d_ffn,K,turned", [(1088, 4096, True),    # 17 weight tiles
                                            (576, 8192, True), (1088, 4160, False), (960, 4096, False)])   # (small weights)
def test_turned_walk(M, tile, d_ffn, K, turned):
    import torch
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    A = torch.from_numpy(synth.round_to_bf16(synth.random_normal((tile + 1, K), seed=M))).cuda().to(torch.bfloat16)
    W = torch.from_numpy(synth.round_to_bf16(synth.random_normal((2 * d_ffn, K), seed=d_ffn, std=0.05))).cuda().to(torch.bfloat16)
    # two large products that cancel: between them a sum keeps 2^-13 of an addend, so its order shows in the rounded result
    A[:, [0, K // 2]], W[:, 0], W[:, K // 2] = 1.0, 1024.0, -1024.0
    got = dllm.ffn_gate_up_bf16(A[:M].contiguous(), W).float().cpu().numpy()
    straight = dllm.ffn_gate_up_bf16(A, W, act_tile=tile).float().cpu().numpy()[:M]
    dllm.kernel_status()
    gate, up = (A[:M].double() @ W.double().T).cpu().numpy().reshape(M, d_ffn // 64, 2, 64).transpose(2, 0, 1, 3).reshape(2, M, d_ffn)
    want = gate / (1 + np.exp(-gate)) * up
    # one rounding to bf16, and at most 2^-13 per accumulation of 16 products in a gate or up sum
    bound = 2 ** -8 * np.abs(want).max() + K / 16 * 2 ** -13 * np.abs([gate, up]).max()
    assert np.abs(got - want).max() <= bound and np.abs(straight - want).max() <= bound
    other = (np.arange(d_ffn) // 64 >> 1) % 2 == 1                              # columns of every other pair of tiles
    assert np.array_equal(got[:, ~other], straight[:, ~other])
    assert np.array_equal(got[:, other], straight[:, other]) != turned
