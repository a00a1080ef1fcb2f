"""What a program that uses this framework has it do, as cases that can be timed and compared.

Model cases build a seeded synthetic model of one of the repository's shapes (kg_inputs) and go through
KangarooModel; operator cases call the single-operator entry points on tensors of the caller.
"""
from __future__ import annotations

import numpy as np
import torch

import kg_inputs as ki
from paper_2404_18911_b200 import binding, traffic

# A small bf16 decoder of the size the tests use: whole tiles, so that every tensor-core path is taken.
SMALL = ki.KgShape("small", 4, 512, 4, 128, 1408, 2048, 2, "bf16", logit_scale=10.0, page_size=16, gamma_max=10,
                   gain_std=0.1, deep_resid_scale=0.1, adapter_resid_scale=0.1)

# Of the 33B shape, 12 of the 60 layers: its widths (d 6656, 52 heads, F 17920) in a state of 13 GB.
LAYERS_33B = 12

# Nominal speculation statistics of the synthetic models (tokens a round, draft steps a round), from the benchmark job;
# they only enter the count of bytes that a generation cannot do without.
TOKENS_PER_ROUND, DRAFTS_PER_ROUND = 2.55, 2.36


def listed():
    return [
        # the smallest model, fp32: launches and latency; the repository's tiny configuration as it stands
        dict(name="tiny-f32-generate", kind="generate", model="tiny", prompt=32, new=64, eta=0.6, gamma=6),
        # a small bf16 model behind a service that hands tokens out round by round
        dict(name="small-bf16-rounds", kind="rounds", model="small", prompt=70, rounds=8, eta=0.6, gamma=6),
        # the headline job (prompt 512, eta 0.6, gamma 6); a shorter answer, so that two builds agree on every token
        dict(name="7b-generate-512", kind="generate", model="7b", prompt=512, new=64, eta=0.6, gamma=6),
        # plain greedy decoding after a question of one line (below the size where the prompt pass changes its method)
        dict(name="7b-greedy", kind="greedy", model="7b", prompt=21, new=24),
        # fixed-step drafting, the long end of gamma: verify passes of 11 rows
        dict(name="7b-rounds-gamma10", kind="rounds", model="7b", prompt=100, rounds=3, eta=0.0, gamma=10),
        # time to the first token: a short prompt, and a long one of no round size
        dict(name="7b-prefill-77", kind="prefill", model="7b", prompt=77),
        dict(name="7b-prefill-1999", kind="prefill", model="7b", prompt=1999),
        # the larger shapes with the prompts of their configurations: a long document, a short answer
        dict(name="13b-generate-2048", kind="generate", model="13b", prompt=2048, new=32, eta=0.6, gamma=6),
        dict(name="33b-layers-generate-4096", kind="generate", model="33b", prompt=4096, new=16, eta=0.6, gamma=8),
        # single operators under a caller's own loop: the allocation-free LM head of a verify pass, attention of a verify
        # pass over a long cache, the SwiGLU pair of one decode step
        dict(name="lm-head-noalloc-7", kind="lm_head", V=32000, K=4096, M=7),
        dict(name="attention-7-4090", kind="attention", H=32, hd=128, M=7, pos0=4090),
        dict(name="swiglu-1", kind="swiglu", N=11008, K=4096, M=1),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["generate", "generate", "greedy", "rounds", "prefill", "prefill", "lm_head", "attention", "swiglu"])
    if kind == "generate":
        model = rng.choice(["tiny", "small", "7b", "13b", "33b"])
        most = {"tiny": 120, "small": 1000, "7b": 3000, "13b": 2048, "33b": 3500}[model]
        new = {"tiny": 64, "small": 40, "7b": 48, "13b": 24, "33b": 16}[model]
        return dict(kind=kind, model=model, prompt=_log(rng, 8, most), new=rng.randint(4, new), eta=rng.choice([0.4, 0.6, 0.8]),
                    gamma=rng.randint(2, 8))
    if kind == "greedy":
        return dict(kind=kind, model=rng.choice(["tiny", "small", "7b", "13b"]), prompt=_log(rng, 1, 120), new=rng.randint(4, 20))
    if kind == "rounds":
        return dict(kind=kind, model=rng.choice(["tiny", "small", "7b"]), prompt=_log(rng, 8, 120), rounds=rng.randint(2, 4),
                    eta=rng.choice([0.0, 0.2, 0.6]), gamma=rng.randint(2, 10))
    if kind == "prefill":
        return dict(kind=kind, model=rng.choice(["small", "7b", "7b", "13b", "33b"]), prompt=_log(rng, 16, 2500))
    if kind == "lm_head":
        return dict(kind=kind, V=_log(rng, 2000, 64000), K=16 * rng.randint(32, 512), M=rng.randint(1, 16))
    if kind == "attention":
        return dict(kind=kind, H=rng.choice([8, 12, 32, 40, 52]), hd=rng.choice([64, 128]), M=rng.randint(1, 16), pos0=_log(rng, 60, 8000))
    return dict(kind=kind, N=_log(rng, 1000, 18000), K=16 * rng.randint(32, 512), M=rng.randint(1, 16))


def _shape(case, seed):
    if case["model"] == "small":
        s = SMALL
    elif case["model"] == "33b":
        s = ki.get_config("33b", n_layers=LAYERS_33B)
    else:
        s = ki.get_config(case["model"])
    new = case.get("new", case.get("rounds", 0) * (case.get("gamma", 0) + 1))
    return s.with_(seed=seed, max_seq=case["prompt"] + new + 2 * 16 + 2, gamma_max=10)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.kind = case, case["kind"]
    if "model" in case:
        # a program holds the model and the prompt's ids (host memory, as a tokenizer leaves them)
        shape = _shape(case, seed)
        s.model = binding.KangarooModel(shape, debug_logits=True)
        s.prompt = ki.make_prompt(shape, case["prompt"])
        return s
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*size, std=1.0, dtype=torch.float32):
        t = torch.empty(size, dtype=dtype, device="cuda")
        return t.normal_(0.0, std, generator=g)

    M = case["M"]
    s.scratch = binding.op_scratch(torch)
    if s.kind == "lm_head":
        s.W = normal(case["V"], case["K"], std=0.02, dtype=torch.bfloat16)
        s.x, s.gain = normal(M, case["K"]), 1.0 + normal(case["K"], std=0.1)
        s.tok = torch.empty(M, dtype=torch.int32, device="cuda")
        s.p = torch.empty(M, dtype=torch.float32, device="cuda")
        s.logits = torch.empty(M, case["V"], dtype=torch.float32, device="cuda")
    elif s.kind == "swiglu":
        s.W, s.W2 = (normal(case["N"], case["K"], std=0.02, dtype=torch.bfloat16) for _ in range(2))
        s.x, s.gain = normal(M, case["K"]), 1.0 + normal(case["K"], std=0.1)
    else:
        H, hd, pages = case["H"], case["hd"], (case["pos0"] + M + 15) // 16 + 2
        s.kc, s.vc = (normal(pages, H, 16, hd, dtype=torch.bfloat16) for _ in range(2))
        s.table = torch.randperm(pages, generator=g, device="cuda").to(torch.int32)
        s.qkv = normal(M, 3 * H * hd)
    return s


def _rounds(s):
    c, m = s.case, s.model
    emitted = np.full((c["rounds"], c["gamma"] + 1), -1, dtype=np.int32)
    conf = np.zeros((c["rounds"], c["gamma"]), dtype=np.float32)
    for r in range(c["rounds"]):
        d = m.draft(c["eta"], c["gamma"])
        v = m.verify()
        conf[r, :d["n_steps"]] = d["conf"]
        emitted[r, :v["k"] + 1] = v["emitted"]
    return emitted, conf


def run(s):
    c, k = s.case, s.kind
    if k == "generate":
        tokens, _ = s.model.generate(s.prompt, c["new"], c["eta"], c["gamma"])
        return {"tokens": np.asarray(tokens, dtype=np.int32), "logits": s.model.debug_logits(1, 0)}
    if k in ("greedy", "rounds", "prefill"):
        s.model.reset()
        x0 = s.model.prefill(s.prompt)
        if k == "greedy":
            tokens = s.model.decode_ar(c["new"])
            return {"tokens": np.asarray(tokens, dtype=np.int32), "logits": s.model.debug_logits(1, 0)}
        if k == "prefill":
            return {"token": x0, "logits": s.model.debug_logits(1, 0)}
        emitted, conf = _rounds(s)
        return {"token": x0, "emitted": emitted, "conf": conf, "logits": s.model.debug_logits(1, 0)}
    if k == "lm_head":
        binding.op_lm_head_noalloc(s.W, s.x, s.gain, 1e-6, 8.0, s.tok, s.p, s.logits)
        return {"tok": s.tok, "p": s.p, "logits": s.logits}
    if k == "swiglu":
        return binding.op_linear(s.W, s.x, gain=s.gain, W2=s.W2, scratch=s.scratch)
    out = binding.op_attention(s.qkv, c["pos0"], c["H"], c["hd"], 10000.0, s.kc, s.vc, s.table, 16, scratch=s.scratch)
    return {"out": out, "k": s.kc, "v": s.vc}


def _prompt_work(shape, n):
    """Weights once, the K / V rows written; one multiply-add per weight and row, causal attention."""
    L, d = shape.n_layers, shape.d_model
    layer = 4 * d * d + 3 * d * shape.d_ffn
    weights = L * traffic.layer_weight_bytes(shape) + traffic.adapter_weight_bytes(shape) * 3 // 4 + traffic.head_weight_bytes(shape)
    return (weights + (L + 1) * n * traffic.kv_bytes_per_token_layer(shape),
            2 * n * (L * layer + 3 * d * d) + 2 * shape.vocab * d + 2 * L * d * n * (n + 1))


def work(case):
    k = case["kind"]
    if "model" in case:
        shape, n = _shape(case, 0), case["prompt"]
        nbytes, flops = _prompt_work(shape, n)
        per_row = 2 * (traffic.ar_step_bytes(shape, 0) // traffic._es(shape))
        if k == "greedy":
            nbytes += sum(traffic.ar_step_bytes(shape, n + i) for i in range(case["new"] - 1))
            flops += (case["new"] - 1) * per_row
        elif k in ("generate", "rounds"):
            if k == "generate":
                rounds = max(1.0, (case["new"] - 1) / TOKENS_PER_ROUND)
                drafts = min(case["gamma"], DRAFTS_PER_ROUND)
            else:
                rounds, drafts = case["rounds"], (case["gamma"] if case["eta"] == 0.0 else min(case["gamma"], DRAFTS_PER_ROUND))
            nbytes += rounds * (drafts * traffic.draft_step_bytes(shape, n) + traffic.shallow_pass_bytes(shape, n) +
                                traffic.verify_bytes(shape, n, int(drafts) + 1))
            flops += rounds * (drafts + 1) * per_row
        return {"bytes": float(nbytes), "flops": float(flops)}
    M = case["M"]
    if k == "lm_head":
        V, K = case["V"], case["K"]
        return {"bytes": 2.0 * V * K + 4.0 * M * (K + V) + 4.0 * K, "flops": 2.0 * M * V * K}
    if k == "swiglu":
        N, K = case["N"], case["K"]
        return {"bytes": 4.0 * N * K + 4.0 * M * (K + N) + 4.0 * K, "flops": 4.0 * M * N * K}
    d, T = case["H"] * case["hd"], case["pos0"] + M
    return {"bytes": 4.0 * d * (T + M) + 16.0 * M * d, "flops": 4.0 * M * T * d}


# About four times what was measured.  Operators against float64: 3.5e-6 of the norm (9e-6 for the top-1 probability), at
# most 3e-5 of the root mean square; an entry of a K cache may round to the next bf16 value.  Models, between the two
# prompt passes (other order of every sum): logits 1.1e-4 to 3.2e-4 of the norm and 1.6e-3 of the root mean square,
# confidences 5.5e-4, because K and V pass through bf16; the fp32 model has no such step.  Tokens were the same.
def tolerance(case):
    if case["kind"] == "attention":
        return {"rel": 4e-5, "max": 8e-3}
    if case["kind"] in ("lm_head", "swiglu"):
        return {"rel": 4e-5, "max": 2e-4, "differ": 0.01}
    if case["model"] == "tiny":
        return {"rel": 1e-5, "differ": 0.01}
    if case["kind"] == "rounds":
        return {"rel": 2e-3, "max": 1e-2, "differ": 0.01}
    return {"rel": 1.2e-3, "max": 6e-3, "differ": 0.01}
