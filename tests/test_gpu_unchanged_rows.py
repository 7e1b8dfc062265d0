"""Rows whose inputs did not change reproduce their cached V bit for bit, whatever kind of step wrote it: on an adaptive
step over the same tokens they score exactly 1 (cosine) or 0 (L2 distance), and the ties go to the lowest indices."""
import dataclasses

import numpy as np
import pytest

from paper_2506_06295_b200 import synth

pytestmark = pytest.mark.gpu

WIDE = dataclasses.replace(synth.LLADA_8B, n_layers=3, d_ffn=4096, vocab=1024, mask_id=1023)
GROUPED = dataclasses.replace(synth.DREAM_7B, n_layers=3, d_ffn=3584, vocab=1024, mask_id=1023)


@pytest.fixture(scope="module")
def dllm():
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    return dllm


@pytest.mark.parametrize("metric", ["cosine", "l2"])
@pytest.mark.parametrize("cfg,B,P,R", [
    (WIDE, 1, 512, 256),       # V of the response is split over the k range in adaptive steps
    (GROUPED, 1, 256, 256),    # 512-wide V: many splits
    (WIDE, 2, 130, 150),       # ragged, two sequences
    (WIDE, 1, 1100, 300),      # more than 1024 rows in a full step, 300 in the others
    (WIDE, 4, 200, 512),       # the V product of 2048 rows is not split: it joins Q and K
], ids=["wide", "grouped", "ragged", "long", "batched"])
def test_unchanged_rows_score_exactly(dllm, cfg, B, P, R, metric):
    rng = np.random.default_rng(5)
    ses = dllm.Session(dllm.Model(cfg, "cuda:0").random_init_on_device(3), B, P, R)
    ses.set_selection("v_verify", metric=metric)
    ses.set_prompt(rng.integers(0, cfg.vocab - 1, size=(B, P), dtype=np.int32))
    tokens = np.full((B, R), cfg.mask_id, np.int32)
    tokens[:, :R // 2] = rng.integers(0, cfg.vocab - 1, size=(B, R // 2), dtype=np.int32)
    ses.set_response_tokens(tokens)
    k = R // 4
    exact = 1.0 if metric == "cosine" else 0.0
    layers = 1 if B * R >= 1024 else cfg.n_layers   # (deeper, batched steps that split their products sum a row's norm
    #                                                  in another kernel than those that do not)
    for kind, (rp, rr) in (("full", (True, True)), ("refresh", (False, True)), ("mixed", (True, False)),
                           ("partial", (False, False))):
        ses.step_cached(rp, rr, 0.25) if kind != "full" else ses.step_full()
        before = [ses.get_cache(l, dllm.CACHE_V)[:, P:] for l in range(layers)]
        ses.step_cached(False, False, 0.25)
        ses.sync()
        for l in range(layers):
            idx, sim = ses.selected(l)
            assert (idx == np.arange(k)).all(), f"after {kind}, layer {l}: {np.setdiff1d(idx, np.arange(k))}"
            assert (sim[:, k:] == exact).all(), f"after {kind}, layer {l}: {np.abs(sim[:, k:] - exact).max()}"
            assert np.array_equal(ses.get_cache(l, dllm.CACHE_V)[:, P + k:], before[l][:, k:]), f"after {kind}, layer {l}"


@pytest.mark.parametrize("metric", ["cosine", "l2"])
@pytest.mark.parametrize("cfg,B,P,R,rho", [(GROUPED, 1, 256, 256, 0.5), (GROUPED, 2, 90, 70, 0.3), (WIDE, 1, 130, 200, 0.25),
                                               (GROUPED, 1, 200, 400, 0.25), (WIDE, 1, 100, 300, 0.25), (WIDE, 4, 60, 300, 0.25)],
                         ids=["grouped", "two sequences", "wide", "grouped separate", "wide separate", "verified in the product"])
def test_rows_written_one_by_one_score_exactly(dllm, cfg, B, P, R, rho, metric):
    """The same where only the selected rows' V is written (another product in a mixed step): in the first layer, whose V
    depends on the tokens alone, every row keeps its bits."""
    rng = np.random.default_rng(5)
    ses = dllm.Session(dllm.Model(cfg, "cuda:0").random_init_on_device(3), B, P, R)
    ses.set_selection("v_verify", metric=metric, v_update="selected")
    ses.set_prompt(rng.integers(0, cfg.vocab - 1, size=(B, P), dtype=np.int32))
    ses.set_response_tokens(rng.integers(0, cfg.vocab - 1, size=(B, R), dtype=np.int32))
    exact = 1.0 if metric == "cosine" else 0.0
    ses.step_full()
    before = ses.get_cache(0, dllm.CACHE_V)[:, P:]
    for kind, (rp, rr) in (("refresh", (False, True)), ("mixed", (True, False)), ("partial", (False, False))):
        ses.step_cached(rp, rr, rho)
        assert np.array_equal(ses.get_cache(0, dllm.CACHE_V)[:, P:], before), kind
        ses.step_cached(False, False, rho)
        ses.sync()
        _, sim = ses.selected(0)
        assert (sim == exact).all(), f"after {kind}: {np.abs(sim - exact).max()}"
        assert np.array_equal(ses.get_cache(0, dllm.CACHE_V)[:, P:], before), f"after {kind}"
