"""Sessions of not too many response rows take Q, K and V of all of them from one product and select behind it.  Against the
same session profiled, which runs V, selection and gather, Q / K and RoPE as launches of their own, and against the one-tile
kernel: the same sums, the same selection, bit for bit, at row counts around the edges of tiles and plans.  Which path ran is
asserted by the launches a step takes."""
import dataclasses

import numpy as np
import pytest

from paper_2506_06295_b200 import synth
from tests.test_gpu_row_epilogue import steps

pytestmark = pytest.mark.gpu

WIDE = dataclasses.replace(synth.LLADA_8B, n_layers=2, d_ffn=1024, vocab=1024, mask_id=1023)
GROUPED = dataclasses.replace(synth.DREAM_7B, n_layers=2, d_ffn=1024, vocab=1024, mask_id=1023)
FORTY = dataclasses.replace(WIDE, d_model=5120, n_heads=40, n_kv_heads=40)    # 60 weight tiles of a CTA pair
EIGHTY = dataclasses.replace(WIDE, d_model=8192, n_heads=64, n_kv_heads=8)    # 40 long ones
ODD = synth.small_bf16_model()                 # widths that are no multiples of 128, small weights

PLAIN = dataclasses.replace(synth.TINY, n_kv_heads=2)                    # plain ALUs
PLAIN96 = dataclasses.replace(PLAIN, n_heads=3, n_kv_heads=3, head_dim=96)   # heads that the streaming RoPE does not take


@pytest.fixture(scope="module")
def dllm():
    from paper_2506_06295_b200 import build as build_mod
    build_mod.build()
    from paper_2506_06295_b200 import dllm
    yield dllm
    dllm._check(dllm.lib.dllm_debug_gemm_plan(0))


@pytest.fixture(scope="module")
def models(dllm):
    made = {}

    def get(cfg):
        if id(cfg) not in made:
            made[id(cfg)] = dllm.Model(cfg, "cuda:0").random_init_on_device(4)
        return made[id(cfg)]
    return get


# model, B, P, R, rho, variant; launches per layer that the five steps (full, adaptive, refresh, mixed, adaptive) save against
# the same steps profiled, and against the one-tile kernel: V, V-verify, selection + gather, Q / K and RoPE become the product,
# V-verify and selection + RoPE in an adaptive step (with V of the selected rows alone, its product and scatter go too), the
# product and RoPE in a refresh or full step, where a full step had V and the scatter of the prompt rows as well, and the product
# alone where it places its rows (CTA pairs, unsplit)
CASES = [
    (WIDE, 1, 130, 1, 1.0, "v_verify", "52212", "00000"),
    (WIDE, 1, 40, 33, 0.3, "v_verify", "52212", "00000"),
    (WIDE, 2, 37, 64, 0.25, "v_verify", "52212", "00000"),
    (WIDE, 1, 100, 129, 0.5, "v_verify", "62322", "10110"),
    (WIDE, 1, 70, 193, 0.1, "selected_v", "64324", "10110"),
    (WIDE, 1, 900, 256, 0.25, "v_verify", "52322", "10120"),
    (WIDE, 1, 1200, 250, 0.25, "v_verify", "52322", "10120"),   # a mixed step of more than 1024 rows: V places its own
    (WIDE, 1, 64, 257, 0.25, "v_verify", "40100", "40100"),   # one row too many: separate products
    (FORTY, 1, 50, 200, 0.25, "v_verify", "62322", "10110"),
    (EIGHTY, 1, 50, 128, 0.25, "v_verify", "52212", "00000"),
    (EIGHTY, 1, 50, 224, 0.25, "v_verify", "40000", "40000"),   # the product would take 17 us more than its weights: separate
    (GROUPED, 1, 256, 256, 0.5, "v_verify", "52212", "00000"),
    (GROUPED, 4, 60, 65, 0.1, "v_verify", "00000", "00000"),   # one activation tile and four rows: separate
    (GROUPED, 3, 60, 259, 0.5, "v_verify", "40110", "40110"),   # separate
    (GROUPED, 3, 50, 85, 0.2, "selected_v", "54214", "00000"),
    (GROUPED, 1, 1500, 100, 0.3, "v_verify", "32212", "40010"),
    (ODD, 2, 150, 72, 0.25, "v_verify", "52212", "00000"),
    (ODD, 1, 90, 1023, 0.25, "selected_v", "54204", "00000"),
    (ODD, 16, 20, 16, 1.0, "v_verify", "52212", "00000"),
    (ODD, 2, 150, 72, 0.25, "k_verify", "50200", "00000"),
    (ODD, 2, 150, 72, 0.25, "random", "50200", "00000"),
    (PLAIN, 1, 60, 1030, 0.25, "v_verify", "50210", "00000"),
    (PLAIN, 3, 40, 350, 0.25, "v_verify", "50210", "00000"),
    (PLAIN96, 2, 40, 520, 0.25, "v_verify", "50210", "00000"),
]


@pytest.mark.parametrize("cfg,B,P,R,rho,variant,profiled_saves,one_tile_saves", CASES,
                         ids=[f"{c[0].d_model}-{c[1]}x{c[2]}+{c[3]}-{c[4]}-{c[5]}" for c in CASES])
def test_one_product_equals_separate_launches(dllm, models, cfg, B, P, R, rho, variant, profiled_saves, one_tile_saves):
    m = models(cfg)
    got = steps(dllm, m, B, P, R, False, variant, rho, 0, lists=True)
    for plan, profiled, saves in ((0, True, profiled_saves), (-1, False, one_tile_saves)):
        want = steps(dllm, m, B, P, R, False, variant, rho, plan, profiled, lists=True)
        for k, ((n0, _, a), (n1, _, b)) in enumerate(zip(got, want)):
            for j, (x, y) in enumerate(zip(a, b)):
                assert np.array_equal(x, y), f"plan {plan}, profiled {profiled}, step {k}: output {j} differs"
            assert n1 - n0 == cfg.n_layers * int(saves[k]), f"plan {plan}, profiled {profiled}, step {k}: {n0} launches, {n1}"
