"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one engine and one pass over it, through the public calls of ``corun.Engine``:

  decode   requests are in the middle of their answers; a pass is ``steps`` decode iterations of the engine's one
           padded shape, and the logits of every running request at the end of it
  prompt   a request arrives at an idle engine; a pass is its isolated prefill, its first logits, ``steps`` more
           tokens, its last logits and its release
  chat     several short requests arrive together; a pass is their batched prefill, ``steps`` more tokens for all of
           them, their logits and their release

The decoders are the three that the benchmark serves (Qwen3-8B, Qwen3-30B-A3B and DeepSeek-V2-Lite shapes; all but
one case take a part of their layers, which are all alike, so that three engines fit one GPU) and one small
generic decoder of the kind that drafts tokens for a large one, where a step is bound by launches and latency.
"""
import math

import numpy as np
import torch

from paper_2608_14376_b200 import corun, synth

# The standard deviation of the embedding.  It is the LM head scaled up, as in decoders with tied embeddings: next-token
# distributions are then peaked, as a trained decoder's are, and a token does not hang on the last bits of a sum.
EMBED_STD = 3.0
W_STD = 0.02
KV_STD = 1.28          # cached keys and values: what the projections give for normalised activations at hidden 4096
LATENT_STD = 0.5

DRAFT = synth.ModelShape(12, 1024, 16, 8, 64, 3072, 32000, 1e-6, 1000000.0)


def _shape(case):
    full = {"qwen3_8b": synth.QWEN3_8B, "qwen3_30b_a3b": synth.QWEN3_30B_A3B, "deepseek_v2_lite": synth.DEEPSEEK_V2_LITE,
            "draft": DRAFT}[case["model"]]
    return synth.ModelShape(**dict(full.dict(), n_layers=case["layers"]))


def _moe(case):
    return {"qwen3_30b_a3b": synth.QWEN3_30B_A3B_MOE, "deepseek_v2_lite": synth.DEEPSEEK_V2_LITE_MOE}.get(case["model"])


def _mla(case):
    return synth.DEEPSEEK_V2_LITE_MLA if case["model"] == "deepseek_v2_lite" else None


def listed():
    def decode(name, model, layers, B, active, lo, hi, steps):
        return dict(name=name, kind="decode", model=model, layers=layers, B=B, active=active, lo=lo, hi=hi, steps=steps)

    def prompt(name, model, layers, n, kind="prompt", B=8, active=1, lo=None, steps=1):
        return dict(name=name, kind=kind, model=model, layers=layers, B=B, active=active, lo=lo or n, hi=n, steps=steps)

    return [
        # one user at a small decoder: a step is a chain of launches
        decode("draft_decode_b1", "draft", 12, 1, 1, 300, 300, 16),
        # a lightly loaded engine, long and short contexts side by side
        decode("dense_decode_b8", "qwen3_8b", 12, 8, 8, 256, 8192, 16),
        # the benchmark's own workload, all 36 layers: 64 slots, 40 of them in use
        decode("dense_decode_b64", "qwen3_8b", 36, 64, 40, 512, 4096, 16),
        # a large engine nearly full of short chats
        decode("dense_decode_b256", "qwen3_8b", 12, 256, 200, 64, 2048, 24),
        # time to the first tokens of a short, an ordinary and a long prompt (odd lengths)
        prompt("dense_prompt_77", "qwen3_8b", 12, 77),
        prompt("dense_prompt_1003", "qwen3_8b", 12, 1003),
        prompt("dense_prompt_6001", "qwen3_8b", 12, 6001),
        # a burst of short requests through batched prefill and their first 16 tokens
        prompt("dense_chat_12", "qwen3_8b", 12, 300, kind="chat", B=16, active=12, lo=20, steps=16),
        # decoder with expert layers: the benchmark's 64 slots with 40 in use, and a prompt
        decode("moe_decode_b64", "qwen3_30b_a3b", 12, 64, 40, 512, 4096, 16),
        prompt("moe_prompt_1003", "qwen3_30b_a3b", 12, 1003),
        # decoder with latent attention and expert layers: the benchmark's 128 slots in use, and a prompt
        decode("mla_decode_b128", "deepseek_v2_lite", 9, 128, 128, 512, 4096, 24),
        prompt("mla_prompt_2505", "deepseek_v2_lite", 9, 2505),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    model, layers = rng.choice([("draft", 12), ("qwen3_8b", 12), ("qwen3_8b", 12), ("qwen3_30b_a3b", 12), ("deepseek_v2_lite", 9)])
    kind = rng.choice(["decode", "decode", "prompt", "prompt", "chat"])
    if kind == "prompt":
        n = log_int(1, 5000)
        return dict(kind=kind, model=model, layers=layers, B=rng.choice([1, 8, 32]), active=1, lo=n, hi=n, steps=1)
    if kind == "chat":
        active = rng.randint(2, 16)
        lo = log_int(1, 200)
        return dict(kind=kind, model=model, layers=layers, B=rng.choice([16, 32, 64]), active=active, lo=lo, hi=lo + log_int(8, 300),
                    steps=rng.choice([4, 8, 16]))
    B = log_int(1, 256)
    active = max(1, int(round(B * rng.uniform(0.15, 1.0))))
    lo = log_int(16, 2048)
    hi = max(lo, min(8192, log_int(lo, 8 * lo), 2 * 200000 // active - lo))
    return dict(kind=kind, model=model, layers=layers, B=B, active=active, lo=lo, hi=hi, steps=rng.choice([8, 16]))


def _lengths(case, seed):
    """The running requests' cached tokens, or the prompts' lengths."""
    return [int(v) for v in synth.uniform_lengths(case["lo"], case["hi"], case["active"], seed=seed + 2)]


def prepare(case, seed):
    sh, moe, mla = _shape(case), _moe(case), _mla(case)
    B, n_active, steps = case["B"], case["active"], case["steps"]
    kw = {}
    if mla is not None:
        w, kw["mla"] = synth.make_mla_weights_torch(sh, mla, seed=seed, std=W_STD)
        kw["kv_block"] = 64
    else:
        w = synth.make_weights_torch(sh, seed=seed, std=W_STD, dense_ffn=moe is None)
    if moe is not None:
        kw["moe"] = synth.make_moe_torch(sh, seed=seed, std=W_STD, **moe)
    torch.mul(w["lm_head"], EMBED_STD / W_STD, out=w["embed"])
    lengths = _lengths(case, seed)
    more = 32 * steps if case["kind"] == "decode" else steps       # tokens that a request may still produce
    page = kw.get("kv_block", 16)
    reserve = [n + more + 1 for n in lengths]
    eng = corun.Engine(sh, w, B, max(reserve), kv_pool_blocks=sum(-(-r // page) for r in reserve), **kw)
    slots = [int(s) for s in synth.pick_slots(B, n_active, seed=seed + 7)]
    active, seeds = np.zeros(B, np.uint8), np.zeros(B, np.uint64)
    for i, s in enumerate(slots):
        active[s], seeds[s] = 1, synth.request_seed(seed + i)
    s = dict(eng=eng, kind=case["kind"], steps=steps, slots=slots, lengths=lengths, reserve=reserve, active=active, seeds=seeds,
             logits=np.empty((n_active, sh.vocab), np.float32))
    if case["kind"] == "decode":
        s["pending"] = [int(p[0]) for p in synth.make_prompts(sh.vocab, [1] * n_active, seed=seed + 5)]
        _admit(s)
        for i, slot in enumerate(slots):
            eng.kv_fill(slot, lengths[i], LATENT_STD if mla is not None else KV_STD, seed + 100 + i)
    else:
        s["prompts"] = synth.make_prompts(sh.vocab, lengths, seed=seed + 5)
    return s


def _admit(s):
    for slot, n, reserve, pending in zip(s["slots"], s["lengths"], s["reserve"], s["pending"]):
        s["eng"].adopt(slot, n, reserve, pending, temperature=0.7, top_p=0.95)


def run(s):
    eng, slots = s["eng"], s["slots"]
    out = {}
    if s["kind"] == "decode":
        if any(eng.context_len(slot) + s["steps"] > r for slot, r in zip(slots, s["reserve"])):
            for slot in slots:                # the requests have their last token: the next ones take their slots
                eng.release(slot)
            _admit(s)
    elif s["kind"] == "prompt":
        out["first"] = [eng.prefill(slots[0], s["prompts"][0], s["reserve"][0], 0.7, 0.95, int(s["seeds"][slots[0]]))]
        out["first_logits"] = eng.logits(slots[0])
    else:
        out["first"] = eng.prefill_batch(slots, s["prompts"], s["reserve"], 0.7, 0.95, [int(s["seeds"][x]) for x in slots])
    out["tokens"] = np.stack([eng.decode_step(s["active"], s["seeds"]) for _ in range(s["steps"])])
    for i, slot in enumerate(slots):
        s["logits"][i] = eng.logits(slot)
    out["logits"] = s["logits"]
    if s["kind"] != "decode":
        for slot in slots:
            eng.release(slot)
    return out


def _counts(case):
    """Per layer and in all: weights, weights that a token meets, cached values of a token, and the operations of one
    cached token in one row's attention."""
    sh, moe, mla = _shape(case), _moe(case), _mla(case)
    H, L, nh = sh.hidden, sh.n_layers, sh.n_q_heads
    if mla is not None:
        rank, nope, rope, vh = mla["kv_lora_rank"], mla["qk_nope"], mla["qk_rope"], mla["v_head"]
        attn = (nh * (nope + rope) + rank + rope) * H + nh * (nope + vh) * rank + H * nh * vh
        cached, ops, dense = rank + rope, 2 * nh * (nope + rope + vh), mla["first_dense"]
    else:
        attn = sh.qkv_dim * H + H * sh.q_dim
        cached, ops, dense = 2 * sh.kv_dim, 4 * sh.q_dim, (L if moe is None else 0)
    fixed = L * attn + dense * 3 * sh.ffn * H            # met by every token
    expert = n_exp = top = 0
    if moe is not None:
        expert, n_exp, top = 3 * moe["expert_ffn"] * H, moe["n_experts"], moe["top_k"]
        fixed += (L - dense) * (moe["n_experts"] * H + moe["n_shared"] * expert)
    return fixed, (L - dense) * expert, n_exp, top, L * cached, L * ops, sh.vocab * H


def work(case):
    fixed, expert, n_exp, top, cached, ops, head = _counts(case)
    n, m, steps = case["active"], (case["lo"] + case["hi"]) / 2, case["steps"]

    def weights(rows):                        # of experts: those that at least one of the rows selects
        return fixed + (expert * n_exp * (1 - (1 - top / n_exp) ** rows) if n_exp else 0)

    nbytes = steps * 2 * (weights(n) + head + n * cached * (m + steps / 2)) + steps * n * 2 * cached
    flops = steps * n * (2 * (fixed + top * expert + head) + ops * (m + steps / 2))
    logits = n * head / _shape(case).hidden * 4
    nbytes += logits
    if case["kind"] != "decode":
        nbytes += 2 * (weights(n * m) + head + n * m * cached) + logits
        flops += n * (2 * (m * (fixed + top * expert) + head) + ops * m * m / 2)
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    # Activations are pairs of bf16 and the cache is fp16: with the sums in another order (other tiles, other cuts of K, experts
    # in groups or not) the logits of these cases move by up to 1.6e-4 (a prompt of 77 tokens, dense; 1e-5 to 5e-5 elsewhere).
    return {"rel": 6e-4}
