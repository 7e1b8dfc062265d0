"""Sessions of not too many response rows take Q, K and V of all of them from one product and select behind it.  Against the
same session profiled, which runs V, selection and gather, Q / K and RoPE as launches of their own, and against the one-tile
kernel: the same sums, bit for bit, at row counts around the edges of tiles and plans."""
import dataclasses

import numpy as np
import pytest

from paper_2506_06295_b200 import synth
from tests.test_gpu_row_epilogue import steps

pytestmark = pytest.mark.gpu

WIDE = dataclasses.replace(synth.LLADA_8B, n_layers=2, d_ffn=1024, vocab=1024, mask_id=1023)
GROUPED = dataclasses.replace(synth.DREAM_7B, n_layers=2, d_ffn=1024, vocab=1024, mask_id=1023)
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


CASES = [(cfg, B, P, R, rho, variant) for cfg, B, P, R, rho, variant in [
    (WIDE, 1, 130, 1, 1.0, "v_verify"), (WIDE, 1, 40, 33, 0.3, "v_verify"), (WIDE, 2, 37, 64, 0.25, "v_verify"),
    (WIDE, 1, 100, 129, 0.5, "v_verify"), (WIDE, 1, 70, 193, 0.1, "selected_v"), (WIDE, 1, 900, 256, 0.25, "v_verify"),
    (WIDE, 1, 1200, 250, 0.25, "v_verify"),                     # a mixed step of more than 1024 rows: V places its own
    (WIDE, 1, 64, 257, 0.25, "v_verify"),                       # one row too many: separate products
    (GROUPED, 1, 256, 256, 0.5, "v_verify"), (GROUPED, 3, 60, 259, 0.5, "v_verify"), (GROUPED, 3, 50, 85, 0.2, "selected_v"), (GROUPED, 1, 1500, 100, 0.3, "v_verify"),
    (ODD, 2, 150, 72, 0.25, "v_verify"), (ODD, 1, 90, 1023, 0.25, "selected_v"), (ODD, 16, 20, 16, 1.0, "v_verify"), (ODD, 2, 150, 72, 0.25, "k_verify"),
    (ODD, 2, 150, 72, 0.25, "random"),
    (PLAIN, 1, 60, 1030, 0.25, "v_verify"), (PLAIN, 3, 40, 350, 0.25, "v_verify"), (PLAIN96, 2, 40, 520, 0.25, "v_verify")]]


@pytest.mark.parametrize("cfg,B,P,R,rho,variant", CASES,
                         ids=[f"{c[0].d_model}-{c[1]}x{c[2]}+{c[3]}-{c[4]}-{c[5]}" for c in CASES])
def test_one_product_equals_separate_launches(dllm, models, cfg, B, P, R, rho, variant):
    m = models(cfg)
    got = steps(dllm, m, B, P, R, False, variant, rho, 0)
    for plan, profiled in ((0, True), (-1, False)):
        want = steps(dllm, m, B, P, R, False, variant, rho, plan, profiled)
        for k, ((n0, _, a), (n1, _, b)) in enumerate(zip(got, want)):
            assert n0 <= n1, f"step {k}: {n0} launches against {n1}"
            for j, (x, y) in enumerate(zip(a, b)):
                assert np.array_equal(x, y), f"plan {plan}, profiled {profiled}, step {k}: output {j} differs"
