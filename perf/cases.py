"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one pass through the public API (`paper_2506_06295_b200.dllm`): one denoising step of a session in the
middle of a generation with the prediction read back, or a whole small generation.  The listed cases are the
repository's own configurations (`synth.WORKLOADS` and its small bf16 model) at the step kinds the caching schedule is
made of; `draw` gives others of the same ranges.

    partial   adaptive partial update: most steps of every schedule (211 of the 256 of the LLaDA-8B configuration)
    refresh   response refresh, every K_r steps
    mixed     prompt refresh on a step that updates the response adaptively
    full      everything recomputed: the first step, the joint refreshes, and the uncached decoder

Weights are i.i.d. N(0, 0.02^2) and prompts uniform ids, as everywhere in this repository.  For the steps of the bf16
models the branches that add to the residual stream are scaled by about 1 / sqrt(2 layers) and the embedding to unit
size, so that the stream changes slowly with depth as a trained model's does; without that a difference in the last
bit of one sum grows to 2 to 3 % over 32 layers and no two correct implementations agree.  The top two logits of a
position may still lie a few hundredths apart, so the greedy ids of bf16 models are no stable output, and a token
picked differently would change a whole row of every later pass.  The bf16 cases therefore return what a step leaves
behind -- the four caches of every layer and the confidences -- and no transition runs between their passes; the fp32
case generates to the end and returns the tokens.
"""
import math

import numpy as np
import torch

from paper_2506_06295_b200 import dllm, synth

MODELS = {
    "tiny": synth.TINY,                              # fp32
    "small": synth.small_bf16_model(),               # widths that are no multiples of 128
    "small_gqa": synth.small_bf16_model(gqa=True),   # the same with 7 query heads on one KV head
    "llada8b": synth.LLADA_8B,
    "dream7b": synth.DREAM_7B,                       # grouped heads
}
SCHEDULE = dict(K=256, Kp=100, Kr=6)                 # of the block-restricted steps
STEP_OF_KIND = {"partial": 129, "refresh": 126}      # a k of that schedule that is such a step
CHUNK = 1 << 30                                      # elements of one returned piece of the caches


def _step(name, model, kind, B, P, R, rho, block=0, compact=False):
    return {"name": name, "model": model, "kind": kind, "B": B, "P": P, "R": R, "rho": rho, "block": block,
            "compact": compact}


def listed():
    return [
        # a whole generation of the small fp32 configuration: launches and host calls, hardly any work
        {"name": "tiny_generate_fp32", "model": "tiny", "kind": "generate", "B": 1, "P": 64, "R": 32, "rho": 0.25,
         "block": 32, "steps": 8, "Kp": 4, "Kr": 2},
        # the smallest bf16 step, ragged in every dimension: launch latency
        _step("small_gqa_partial", "small_gqa", "partial", 2, 150, 72, 0.25),
        # the headline configuration: interactive decoding of one sequence, its three common step kinds
        _step("llada_partial", "llada8b", "partial", 1, 512, 256, 0.25),
        _step("llada_refresh", "llada8b", "refresh", 1, 512, 256, 0.25),
        _step("llada_full", "llada8b", "full", 1, 512, 256, 0.25),
        # a short answer to a ragged prompt, decoded in blocks of 32 with the prediction of that block only
        _step("llada_partial_block", "llada8b", "partial", 1, 389, 128, 0.25, block=32),
        # grouped heads, half of the response recomputed
        _step("dream_partial", "dream7b", "partial", 1, 256, 256, 0.5),
        _step("dream_refresh", "dream7b", "refresh", 1, 256, 256, 0.5),
        # question over a long document: three rows against 4128 keys, and the step that reads the document
        _step("long_partial", "llada8b", "partial", 1, 4096, 32, 0.1, compact=True),
        _step("long_full", "llada8b", "full", 1, 4096, 32, 0.1, compact=True),
        # batched serving
        _step("batch16_partial", "llada8b", "partial", 16, 1024, 512, 0.25),
        _step("batch16_full", "llada8b", "full", 16, 1024, 512, 0.25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    which = rng.random()
    if which < 0.12:
        block = rng.choice([8, 16, 24, 32])
        blocks = rng.randint(1, 3)
        return {"model": "tiny", "kind": "generate", "B": rng.randint(1, 3), "P": _log_int(rng, 17, 200),
                "R": block * blocks, "rho": round(rng.uniform(0.1, 0.5), 2), "block": block,
                "steps": blocks * rng.choice([2, 4, 8]), "Kp": rng.randint(3, 9), "Kr": rng.randint(2, 4)}
    if which < 0.24:
        return _draw_step(rng, rng.choice(["small", "small_gqa"]), 8, 2048)
    return _draw_step(rng, rng.choice(["llada8b", "llada8b", "dream7b"]), 16, 12288)


def _draw_step(rng, model, most_batch, most_rows):
    kind = rng.choice(["partial", "partial", "partial", "refresh", "refresh", "mixed", "full"])
    R = _log_int(rng, 24, 512)
    P = _log_int(rng, 40, min(4096, most_rows - R))
    B = min(_log_int(rng, 1, most_batch), max(1, most_rows // (P + R)))
    block = rng.choice([0, 0, 8, 16]) if kind in STEP_OF_KIND else 0
    case = _step("", model, kind, B, P, R, round(rng.uniform(0.05, 0.5), 2), block, rng.random() < 0.3)
    del case["name"]
    return case


# ---------------------------------------------------------------- what a user's program holds before the call
def prepare(case, seed):
    cfg = MODELS[case["model"]]
    B, P, R = case["B"], case["P"], case["R"]
    rng = np.random.default_rng(seed)
    prompt = rng.integers(0, cfg.vocab - 1, size=(B, P), dtype=np.int32)     # the mask id is vocab - 1
    model = dllm.Model(cfg, "cuda:0").random_init_on_device(seed)
    if case["kind"] != "generate":
        model.tensor_view("embed").mul_(1.0 / synth.WEIGHT_STD)
        for name, _ in synth.tensor_names(cfg):
            if name.endswith((".wo", ".wd")):        # a power of two: no rounding
                model.tensor_view(name).mul_(2.0 ** -round(math.log2(2 * cfg.n_layers) / 2))
    session = dllm.Session(model, B, P, R, compact_cache=bool(case.get("compact", False)))
    session.set_prompt(prompt)
    state = {"case": case, "prompt": prompt, "model": model, "session": session}
    if case["kind"] == "generate":
        return state
    # half of the response is decoded; then the transition before this step has set one more token per sequence
    # (left to right, as block-wise decoding does)
    done = max(1, R // 2)
    tokens = np.full((B, R), cfg.mask_id, np.int32)
    tokens[:, :done] = rng.integers(0, cfg.vocab - 1, size=(B, done), dtype=np.int32)
    session.set_response_tokens(tokens)
    session.step_full()
    tokens[:, done] = rng.integers(0, cfg.vocab - 1, size=B, dtype=np.int32)
    session.set_response_tokens(tokens)
    session.sync()
    state["caches"] = list(session.cache.view(torch.bfloat16).split(CHUNK))   # K, V, AttnOut, FFNOut, layer by layer
    return state


def _predicted(case):
    """First position and length of the part of the response whose prediction the step is asked for."""
    if not case["block"]:
        return 0, case["R"]
    start = case["R"] // 2 // case["block"] * case["block"]
    return start, min(case["block"], case["R"] - start)


def run(state):
    case, session = state["case"], state["session"]
    if case["kind"] == "generate":
        session.set_prompt(state["prompt"])
        session.generate(case["steps"], case["Kp"], case["Kr"], case["rho"], case["block"])
        return session.tokens()
    if case["block"]:
        start, length = _predicted(case)
        session.step_scheduled_block(STEP_OF_KIND[case["kind"]], **SCHEDULE, rho=case["rho"], block_start=start,
                                     block_len=length)
    elif case["kind"] == "full":
        session.step_full()
    else:
        session.step_cached(case["kind"] == "mixed", case["kind"] == "refresh", case["rho"])
    _, confidence = session.pred()
    return {"confidence": confidence, "caches": state["caches"]}


# ---------------------------------------------------------------- what a pass cannot do without
def _step_work(case, kind, head_rows):
    c = MODELS[case["model"]]
    B, P, R, n = case["B"], case["P"], case["R"], case["P"] + case["R"]
    d, dq, dkv, m, size = c.d_model, c.dq, c.dkv, c.d_ffn, 2 if c.dtype == "bf16" else 4
    prompt = B * P if kind in ("full", "mixed") else 0                        # prompt rows recomputed
    response = B * (R if kind in ("full", "refresh") else int(case["rho"] * R + 1e-6))
    active, values = prompt + response, prompt + (B * R if response else 0)  # V is projected for all response rows
    flops = 2.0 * d * (values * dkv + active * (dq + dkv)) + 2.0 * active * dq * d + 6.0 * active * d * m
    flops += 4.0 * active * n * dq
    weights = d * (dq + 2 * dkv) + dq * d + 3 * d * m
    old_k = B * n - active                                                    # cached rows read
    old_v = {"partial": B * n, "mixed": B * R, "refresh": B * P, "full": 0}[kind]
    outs_written = active if not case.get("compact") else response
    moved = (old_k + old_v + active + values) * dkv + 2 * (B * R - response) * d + 2 * outs_written * d
    embedded, head = (B * R + prompt) * d, c.vocab * d
    return (size * (c.n_layers * (weights + moved) + embedded + head) + 8.0 * B * R,
            c.n_layers * flops + 2.0 * head_rows * head)


def work(case):
    if case["kind"] != "generate":
        moved, flops = _step_work(case, case["kind"], case["B"] * _predicted(case)[1])
        return {"bytes": moved, "flops": flops}
    moved = flops = 0.0
    for k in range(case["steps"], 0, -1):
        full, p, r = k == case["steps"], k % case["Kp"] == 0, k % case["Kr"] == 0
        b, f = _step_work(case, "full" if full or (p and r) else "mixed" if p else "refresh" if r else "partial",
                          case["B"] * case["R"])
        moved, flops = moved + b, flops + f
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    if case["kind"] == "generate":
        return {"differ": 0.01}   # fp32: a tie of two confidences may fall either way
    # bf16 operands through up to 32 layers: each rounding is 2^-9 of its value, a confidence is the exponential of a
    # sum of them, and a row whose similarity lies at the selection's threshold may be recomputed by one
    # implementation and kept by another.  Splitting attention's keys otherwise moves the caches of the 8B model by
    # 6e-3 and its confidences by 1.1e-2; 2e-2 is the bound of this repository's tests for hidden states.
    return {"rel": 2e-2, "max": 0.3}
