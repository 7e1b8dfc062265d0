"""Projections that place their own rows (rounded, rotated, scattered: gemm_rows.cu) against the one-tile kernel and the
row-wise kernels behind it, bit for bit: same sums, same rounding, other launches.  Which path ran is asserted by the
launches a step takes."""
import dataclasses

import numpy as np
import pytest

from paper_2506_06295_b200 import synth

pytestmark = pytest.mark.gpu


def model(d, H, Hkv, hd, m):
    return synth.ModelConfig(n_layers=2, d_model=d, n_heads=H, n_kv_heads=Hkv, head_dim=hd, d_ffn=m, vocab=304,
                             mask_id=303, dtype="bf16")


# seven k-blocks are never split.  9472 or 4736 weight rows: 150 / 200 / 400 rows take tiles of 192 / 128 / 256
HEADS64, HEADS128 = model(448, 74, 74, 64, 448), model(448, 37, 37, 128, 448)
OUTS = model(4736, 7, 1, 64, 448)                                                   # O and down with seven k-blocks
BATCHED = dataclasses.replace(synth.LLADA_8B, n_layers=2, d_ffn=1024, vocab=1024, mask_id=1023)  # unsplit by tile count
VARIANTS = {"v_verify": {}, "k_verify": dict(strategy="k_verify"), "random": dict(strategy="random"),
            "selected_v": dict(v_update="selected")}


@pytest.fixture(scope="module")
def dllm():
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    yield dllm
    dllm._check(dllm.lib.dllm_debug_gemm_plan(0))


def steps(dllm, m, B, P, R, compact, variant, rho, plan, profiled=False, lists=False):
    """(launches, bytes of the O and down products if profiled, outputs) of a full, an adaptive, a refresh, a mixed and
    another adaptive step; lists: with what the steps selected."""
    dllm._check(dllm.lib.dllm_debug_gemm_plan(plan))
    cfg = m.cfg
    rng = np.random.default_rng(9)
    ses = dllm.Session(m, B, P, R, compact_cache=compact)
    ses.set_selection(**VARIANTS[variant])
    ses.set_prompt(rng.integers(0, cfg.vocab - 1, size=(B, P), dtype=np.int32))
    out = []
    for rp, rr in ((True, True), (False, False), (False, True), (True, False), (False, False)):
        ses.set_response_tokens(rng.integers(0, cfg.vocab, size=(B, R), dtype=np.int32))
        if variant == "random":
            for l in range(cfg.n_layers):
                ses.set_scores(l, rng.random((B, R), dtype=np.float32))
        ses.profile(profiled)
        before = ses.launch_count()
        ses.step_cached(rp, rr, rho)
        launches = ses.launch_count() - before
        ses.sync()
        nbytes = [ses.profile_read(dllm.PROF_CLASSES.index(c))["bytes"] for c in ("gemm_o", "gemm_down")]
        out.append((launches, nbytes, [ses.hidden(), ses.pred()[1]] + [ses.get_cache(l, w) for l in range(cfg.n_layers)
                                                               for w in range(4)]))
        for l in range(cfg.n_layers if lists else 0):
            idx, scores = ses.selected(l)
            out[-1][2].extend([idx] if rr else [idx, scores])   # (scores mean something after an adaptive step)
    return out


CASES = [
    # model, B, P, R, compact, rho, variant; of the five steps, those that take fewer launches with the row epilogue, and
    # those whose O and down products write bf16 rows (2 bytes per element instead of 4 in their profiled traffic)
    *[(HEADS64, 1, 200, 200, False, 0.75, v, "11111", ("00000", "00000")) for v in VARIANTS],
    (HEADS128, 1, 200, 200, False, 0.75, "v_verify", "11111", ("00000", "00000")),
    (HEADS128, 2, 150, 131, True, 0.55, "selected_v", "11111", ("00000", "00000")),  # 144 / 262 / 444 rows; response rows start inside a tile
    (OUTS, 1, 37, 131, False, 0.25, "v_verify", "00000", ("10100", "10100")),  # 168 and 131 rows; 32 and 69 in the other steps
    (OUTS, 1, 37, 131, True, 0.25, "v_verify", "00000", ("10100", "10100")),
    (BATCHED, 4, 100, 256, False, 0.5, "v_verify", "11111", ("10110", "11111")),  # O of 512 rows is split
]


@pytest.mark.parametrize("cfg,B,P,R,compact,rho,variant,fewer,placed", CASES,
                         ids=[f"{c[0].d_model}x{c[0].n_heads}h{c[0].head_dim}-{c[2]}-{c[6]}-{'c' if c[4] else 'f'}" for c in CASES])
def test_placed_rows_equal_the_row_kernels(dllm, cfg, B, P, R, compact, rho, variant, fewer, placed):
    m = dllm.Model(cfg, "cuda:0").random_init_on_device(4)
    got = steps(dllm, m, B, P, R, compact, variant, rho, 0)
    want = steps(dllm, m, B, P, R, compact, variant, rho, -1)
    prof = steps(dllm, m, B, P, R, compact, variant, rho, 0, profiled=True)
    prof_rows = steps(dllm, m, B, P, R, compact, variant, rho, -1, profiled=True)
    for k, ((n0, _, a), (n1, _, b), (_, p0, c), (_, p1, _)) in enumerate(zip(got, want, prof, prof_rows)):
        for j, (x, y, z) in enumerate(zip(a, b, c)):
            assert np.array_equal(x, y), f"step {k}: output {j} differs from the row kernels'"
            assert np.array_equal(x, z), f"step {k}: output {j} differs when profiled"
        assert (n0 < n1) == (fewer[k] == "1"), f"step {k}: {n0} launches, {n1} with the row kernels"
        assert [x < y for x, y in zip(p0, p1)] == [o[k] == "1" for o in placed], f"step {k}: bytes {p0}, {p1}"
