"""V-verify in the epilogue of an unsplit V projection of many response rows, against the one-tile kernel and the kernel that
verifies its fp32 rows: the same V, scores that differ by the order of their sums only."""
import dataclasses

import numpy as np
import pytest

from paper_2506_06295_b200 import synth

pytestmark = pytest.mark.gpu

WIDE = dataclasses.replace(synth.LLADA_8B, n_layers=1, d_ffn=512, vocab=512, mask_id=511)
NARROW = synth.ModelConfig(n_layers=1, d_model=2048, n_heads=6, n_kv_heads=3, head_dim=64, d_ffn=512, vocab=512, mask_id=511,
                           dtype="bf16")          # 192 V columns: one and a half tiles


@pytest.fixture(scope="module")
def dllm():
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    yield dllm
    dllm._check(dllm.lib.dllm_debug_gemm_plan(0))


@pytest.mark.parametrize("metric", ["cosine", "l2"])
@pytest.mark.parametrize("v_update", ["whole", "selected"])
@pytest.mark.parametrize("cfg,B,P,R", [(WIDE, 3, 33, 401), (WIDE, 4, 20, 512), (WIDE, 2, 40, 1025), (NARROW, 19, 20, 999)],
                         ids=["ragged", "whole tiles", "one row more", "half a weight tile"])
def test_scores_and_rows(dllm, cfg, B, P, R, v_update, metric):
    m = dllm.Model(cfg, "cuda:0").random_init_on_device(4)
    rng = np.random.default_rng(1)
    prompt = rng.integers(0, cfg.vocab - 1, size=(B, P), dtype=np.int32)
    first = rng.integers(0, cfg.vocab - 1, size=(B, R), dtype=np.int32)
    then = np.where(rng.random((B, R)) < 0.4, rng.integers(0, cfg.vocab - 1, size=(B, R)), first).astype(np.int32)
    out = []
    for plan in (0, -1):
        dllm._check(dllm.lib.dllm_debug_gemm_plan(plan))
        ses = dllm.Session(m, B, P, R)
        ses.set_selection("v_verify", metric=metric, v_update=v_update)
        ses.set_prompt(prompt)
        ses.set_response_tokens(first)
        ses.step_full()
        before = ses.get_cache(0, dllm.CACHE_V)
        ses.set_response_tokens(then)
        ses.step_cached(False, False, 0.25)
        ses.sync()
        out.append((ses.selected(0), before, ses.get_cache(0, dllm.CACHE_V)))
        # which kernel verified: the merge reads 16 bytes per row and 128 columns, the other the fp32 row and the cached one
        ses.profile(True)
        ses.step_cached(False, False, 0.25)
        read = ses.profile_read(dllm.PROF_CLASSES.index("vverify"))
        assert read["bytes"] == B * R * (-(-cfg.dkv // 128) * 16 + 4 if plan == 0 else cfg.dkv * 8)
    ((idx0, sim0), b0, v0), ((idx1, sim1), b1, v1) = out
    assert np.array_equal(b0, b1)
    same = first == then
    exact = 1.0 if metric == "cosine" else 0.0
    assert (sim0[same] == exact).all() and (sim1[same] == exact).all()      # rows whose input did not change
    assert (sim0[~same] < (0.9 if metric == "cosine" else 0.0)).all()       # another token: another random row
    # sums of thousands of fp32 products in another order: a few ulp of each
    np.testing.assert_allclose(sim0, sim1, rtol=2e-6, atol=2e-6)
    if v_update == "whole":
        assert np.array_equal(v0, v1)
    else:   # rows whose scores differ in the last bits may change places at the threshold
        taken = np.zeros((2, B, R), bool)
        for i, idx in enumerate((idx0, idx1)):
            np.put_along_axis(taken[i], idx, True, 1)
        assert taken.sum() == 2 * B * (R // 4) and (taken[0] != taken[1]).sum() <= 4
        for v, t in zip((v0, v1), taken):
            assert np.array_equal(v[:, P:][~t], b0[:, P:][~t])
        assert np.array_equal(v0[:, P:][taken.all(0)], v1[:, P:][taken.all(0)])
        assert (v0[:, P:] != b0[:, P:]).any(2)[taken[0] & ~same].all()
