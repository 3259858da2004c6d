"""The work that this library is measured on, as its users have it done through `paper_2211_17192_b200.binding`:

* `generate`: a prompt (or, for the encoder-decoder, a source) goes in, tokens come out: prompt pass of both models,
  then iterations of draft steps, verification pass, speculative sampling and commit (`Engine.generate`);
* `logits`: one teacher-forced pass of a model over a few rows per sequence on cached context, which is the verification
  pass by itself or, at one row, a plain decode or draft step (`Engine.truncate` + `Engine.forward_logits`);
* `verify`: the speculative-sampling rule on logits that a caller's own models produced (`spec_verify_sample`);
* `sample`: standardised sampling of a token per row of logits (`spec_sample`).

Models have the shapes of `workloads.model_config`.  Their block matrices are random; a trained model's next-token
distribution is peaked, though, and a draft agrees with its target more often than not, and both decide how decoding
runs.  So the embedding is large enough to be seen through the blocks and the head holds the embedding of token v at the
row of v's successor: either model predicts the successor of the last token with most of its probability, and the
target's table of successors is the draft's except for a quarter of the tokens.  Tokens then do not hang on the last bit
of a logit either, at T = 0 or within the 40 likeliest tokens at T = 1.
"""

import math

import numpy as np
import torch

from paper_2211_17192_b200 import binding, workloads

AGREE = 0.75  # share of the tokens after which draft and target predict the same successor
LOGIT_STD = 3.0

PAIRS = {
    "tiny": ("tiny_target", "tiny_draft"),
    "gpt97m": ("gpt97m_target", "gpt6m_draft"),
    "llama7b": ("llama7b_target", "llama160m_draft"),
    "t5xxl": ("t5xxl_target", "t5small_draft"),
}


# --------------------------------------------------------------------------- #
# the cases
# --------------------------------------------------------------------------- #
def listed():
    return [
        # one chat-sized decision: a lone sequence, the paper's small vocabulary; launches and host time are all there is
        dict(name="verify_b1_v8192", kind="verify", batch=1, gamma=3, vocab=8192, temperature=1.0, top_k=0, top_p=1.0,
             draft_noise=0.5),
        # a full serving batch on the whole vocabulary: every logit of both models is read once
        dict(name="verify_b64_v32000", kind="verify", batch=64, gamma=7, vocab=32000, temperature=1.0, top_k=0, top_p=1.0,
             draft_noise=1.0),
        # the usual serving options together (top-k, nucleus, T below 1) on a vocabulary that is not a multiple of four
        dict(name="verify_b24_v50003_k40_p90", kind="verify", batch=24, gamma=4, vocab=50003, temperature=0.8, top_k=40,
             top_p=0.9, draft_noise=1.0),
        # plain sampling with the nucleus alone, large vocabulary
        dict(name="sample_r200_v100000_p90", kind="sample", rows=200, vocab=100000, temperature=1.0, top_k=0, top_p=0.9),
        # the fp32 pair: the smallest models, exact arithmetic wanted
        dict(name="generate_tiny_fp32", kind="generate", pair="tiny", batch=1, prompt=16, ragged=0.0, n_new=64, gamma=3,
             temperature=0.0, top_k=0),
        # the paper's small bf16 pair, sampled at T = 1 within the 40 likeliest tokens
        dict(name="generate_gpt97m_k40", kind="generate", pair="gpt97m", batch=1, prompt=128, ragged=0.0, n_new=128, gamma=5,
             temperature=1.0, top_k=40),
        # one user of the 7B-shaped pair: long prompt, long answer
        dict(name="generate_llama7b_b1", kind="generate", pair="llama7b", batch=1, prompt=1024, ragged=0.0, n_new=256, gamma=2,
             temperature=0.0, top_k=0),
        # a serving batch of prompts of different lengths, short answers: mostly the prompt pass
        dict(name="generate_llama7b_b16", kind="generate", pair="llama7b", batch=16, prompt=1000, ragged=0.5, n_new=32,
             gamma=4, temperature=0.0, top_k=0),
        # translation: the encoder once over the source, then decoding with cross-attention
        dict(name="generate_t5xxl_b1", kind="generate", pair="t5xxl", batch=1, prompt=512, ragged=0.0, n_new=128, gamma=7,
             temperature=0.0, top_k=0),
        # one draft step for a few sequences
        dict(name="logits_llama160m_b4_m1", kind="logits", model="llama160m_draft", batch=4, rows=1, context=777),
        # the verification pass of one sequence, gamma = 2
        dict(name="logits_llama7b_b1_m3", kind="logits", model="llama7b_target", batch=1, rows=3, context=1023),
        # the verification pass of a large batch, gamma = 6
        dict(name="logits_llama7b_b32_m7", kind="logits", model="llama7b_target", batch=32, rows=7, context=509),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, none dearer than the dearest listed one."""
    kind = rng.choice(["verify", "verify", "sample", "generate", "generate", "logits", "logits"])
    if kind in ("verify", "sample"):
        vocab = _log_int(rng, 4000, 128000)
        if rng.random() < 0.6:
            vocab = vocab // 8 * 8
        top_k, top_p = rng.choice([(0, 1.0), (0, 1.0), (40, 1.0), (0, 0.9), (50, 0.95)])
        temperature = rng.choice([1.0, 1.0, 0.7])
        if kind == "sample":
            return dict(kind=kind, rows=_log_int(rng, 1, 256), vocab=vocab, temperature=temperature, top_k=top_k, top_p=top_p)
        return dict(kind=kind, batch=_log_int(rng, 1, 96), gamma=rng.randint(1, 8), vocab=vocab,
                    temperature=rng.choice([temperature, temperature, 0.0]), top_k=top_k, top_p=top_p,
                    draft_noise=rng.choice([0.5, 1.0, 2.0]))
    if kind == "generate":
        pair = rng.choice(["tiny", "gpt97m", "llama7b", "llama7b", "t5xxl"])
        gamma = rng.randint(1, 7)
        if pair == "tiny":
            return dict(kind=kind, pair=pair, batch=rng.randint(1, 4), prompt=rng.randint(1, 40), ragged=rng.choice([0.0, 0.5]),
                        n_new=rng.randint(16, 64), gamma=min(gamma, 5), temperature=0.0, top_k=0)
        if pair == "gpt97m":
            return dict(kind=kind, pair=pair, batch=_log_int(rng, 1, 8), prompt=_log_int(rng, 16, 700), ragged=rng.choice([0.0, 0.5]),
                        n_new=rng.randint(16, 128), gamma=gamma, temperature=0.0, top_k=0)
        if pair == "t5xxl":
            return dict(kind=kind, pair=pair, batch=rng.randint(1, 3), prompt=rng.randint(40, 512), ragged=rng.choice([0.0, 0.5]),
                        n_new=rng.randint(16, 64), gamma=gamma, temperature=0.0, top_k=0)
        batch = _log_int(rng, 1, 16)
        return dict(kind=kind, pair=pair, batch=batch, prompt=_log_int(rng, 30, min(1500, 12000 // batch)), ragged=rng.choice([0.0, 0.5]),
                    n_new=rng.randint(8, 32), gamma=min(gamma, 6), temperature=0.0, top_k=0)
    model = rng.choice(["gpt97m_target", "llama160m_draft", "llama7b_target"])
    batch = _log_int(rng, 1, 32)
    most = 500 if model == "gpt97m_target" else 1500 if batch <= 8 else 500
    return dict(kind=kind, model=model, batch=batch, rows=rng.randint(1, 7), context=_log_int(rng, 8, most))


# --------------------------------------------------------------------------- #
# what a user's program has in hand
# --------------------------------------------------------------------------- #
def _weights(cfg, gen, successor):
    """Random block matrices; the embedding and a head that predicts `successor`."""
    dtype = torch.bfloat16 if cfg["dtype"] == "bf16" else torch.float32
    emb_std = 2.0 if cfg["d_model"] >= 2048 else 1.0  # (wide blocks add more to the residual stream)
    out = {}
    for name, shape, kind in workloads.tensor_shapes(cfg):
        if kind == "gain":
            out[name] = torch.ones(shape, device="cuda")
        elif kind == "bias":
            out[name] = torch.randn(shape, device="cuda", generator=gen) * cfg["bias_std"]
        elif name == "head":
            out[name] = torch.empty(shape, device="cuda", dtype=dtype)
            out[name][successor] = out["tok_emb"] * (cfg["head_std"] / emb_std)
        else:
            std = emb_std if name == "tok_emb" else workloads.INIT_STD
            out[name] = torch.randn(shape, device="cuda", dtype=dtype, generator=gen).mul_(std)
    return out


def _pair(case):
    """The configs of both models; every head is a matrix of its own (a table of successors cannot be the embedding)."""
    return tuple(workloads.scaled_config(workloads.model_config(n), tied=False) for n in PAIRS[case["pair"]])


def _pair_weights(target, draft, gen):
    vocab = target["vocab"]
    drafts = torch.randperm(vocab, device="cuda", generator=gen)
    targets = drafts.clone()
    other = torch.randperm(vocab, device="cuda", generator=gen)[: int((1 - AGREE) * vocab)]
    targets[other] = drafts[other.roll(1)]
    return _weights(target, gen, targets), _weights(draft, gen, drafts)


def _draft_draws(logits, case, gen):
    """x ~ q for every row: Gumbel-max over what the cuts of the case leave."""
    l = logits / case["temperature"] if case["temperature"] > 0 else logits
    if case["temperature"] > 0 and case["top_k"]:
        l = l.masked_fill(l < l.topk(case["top_k"], dim=-1).values[..., -1:], -math.inf)
    if case["temperature"] > 0 and case["top_p"] < 1.0:
        ordered, index = l.sort(dim=-1, descending=True)
        mass = ordered.softmax(-1).cumsum(-1)
        ordered[..., 1:][mass[..., :-1] >= case["top_p"]] = -math.inf
        l = torch.empty_like(l).scatter_(-1, index, ordered)
    if case["temperature"] > 0:
        l = l - torch.empty_like(l).exponential_(generator=gen).log()
    return l.argmax(-1).to(torch.int32)


def _uniforms(shape, gen):
    return (2.0 * torch.randint(0, 1 << 23, shape, device="cuda", generator=gen).float() + 1.0) / (1 << 24)


def _lengths(case, rng):
    """Prompt lengths: all `prompt`, or spread below it by `ragged`."""
    low = max(1, int(case["prompt"] * (1.0 - case["ragged"])))
    lengths = rng.integers(low, case["prompt"] + 1, size=case["batch"])
    lengths[0] = case["prompt"]
    return [int(n) for n in lengths]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    kind = case["kind"]
    state = dict(case=case, kind=kind)
    if kind == "verify":
        b, g, v = case["batch"], case["gamma"], case["vocab"]
        target = torch.randn((b, g + 1, v), device="cuda", generator=gen) * LOGIT_STD
        draft = target[:, :g] + torch.randn((b, g, v), device="cuda", generator=gen) * case["draft_noise"]
        state.update(target=target, draft=draft, tokens=_draft_draws(draft, case, gen), uniforms=_uniforms((b, g + 1), gen),
                     out=torch.empty((2, b), dtype=torch.int32, device="cuda"),
                     workspace=torch.empty(binding.spec_verify_sample_workspace_bytes(b, g, v), dtype=torch.uint8, device="cuda"))
    elif kind == "sample":
        r, v = case["rows"], case["vocab"]
        state.update(logits=torch.randn((r, v), device="cuda", generator=gen) * LOGIT_STD, uniforms=_uniforms((r,), gen),
                     out=torch.empty(r, dtype=torch.int32, device="cuda"))
    elif kind == "generate":
        target, draft = _pair(case)
        tw, dw = _pair_weights(target, draft, gen)
        t5 = target["arch"] == "t5"
        lengths = _lengths(case, rng)
        engine = binding.Engine(target, tw, draft, dw, max_batch=case["batch"],
                                max_len=(1 if t5 else case["prompt"]) + case["n_new"] + case["gamma"] + 2,
                                max_gamma=case["gamma"], max_src_len=case["prompt"] if t5 else 0)
        engine.set_truncation(case["top_k"], 1.0)
        state.update(engine=engine, prompts=[rng.integers(0, target["vocab"], size=n).astype(np.int32) for n in lengths],
                     seed=int(rng.integers(1 << 40)))
    else:
        cfg = workloads.model_config(case["model"])
        b, m, ctx = case["batch"], case["rows"], case["context"]
        rows_at_once = max(m, 64 // b, 16)
        successor = torch.randperm(cfg["vocab"], device="cuda", generator=gen)
        engine = binding.Engine(cfg, _weights(cfg, gen, successor), max_batch=b, max_len=ctx + m + 1, max_gamma=rows_at_once - 1)
        tokens = rng.integers(0, cfg["vocab"], size=(b, ctx + m)).astype(np.int32)
        for c in range(0, ctx, rows_at_once):
            engine.forward_logits(0, tokens[:, c:min(c + rows_at_once, ctx)])
        state.update(engine=engine, cached=[ctx] * b, tokens=np.ascontiguousarray(tokens[:, ctx:]))
    torch.cuda.synchronize()
    return state


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "verify":
        out = state["out"]
        binding.spec_verify_sample(state["target"], state["draft"], state["tokens"], state["uniforms"], case["temperature"],
                                   n_accepted=out[0], next_token=out[1], workspace=state["workspace"], top_k=case["top_k"],
                                   top_p=case["top_p"])
        return out
    if kind == "sample":
        return binding.spec_sample(state["logits"], state["uniforms"], case["temperature"], tokens=state["out"],
                                   top_k=case["top_k"], top_p=case["top_p"])
    if kind == "generate":
        tokens, stats = state["engine"].generate(state["prompts"], case["n_new"], case["gamma"], case["temperature"], state["seed"])
        return {"tokens": tokens, "iterations": stats["iterations"], "tests_passed": stats["tests_passed"]}
    state["engine"].truncate(0, state["cached"])
    return state["engine"].forward_logits(0, state["tokens"])


# --------------------------------------------------------------------------- #
# what a pass cannot do without
# --------------------------------------------------------------------------- #
def _matrices(cfg):
    """(parameters that every decoder row meets, parameters that every source row meets)."""
    dec = enc = 0
    for name, shape, kind in workloads.tensor_shapes(cfg):
        if kind in ("gain", "bias") or name == "pos_emb" or (name == "tok_emb" and not cfg["tied"]):
            continue
        if name.startswith("enc.") or name.endswith("wkv_x"):
            enc += math.prod(shape)
        else:
            dec += math.prod(shape)
    return dec, enc


def _kv_row(cfg):
    """Bytes of one position's K and V rows over all blocks (16-bit rows for bf16 models)."""
    return 2 * cfg["n_layers"] * cfg["n_kv_heads"] * cfg["d_head"] * (2 if cfg["dtype"] == "bf16" else 4)


def _pass_work(cfg, batch, rows, context, cross):
    """Weights and cached rows once; multiply-adds of every row with every matrix and with the keys it sees."""
    elem = 2 if cfg["dtype"] == "bf16" else 4
    dec, _ = _matrices(cfg)
    keys = context + cross
    return (dec * elem + batch * keys * _kv_row(cfg),
            batch * rows * (2 * dec + 4 * keys * cfg["n_layers"] * cfg["n_heads"] * cfg["d_head"]))


def work(case):
    kind = case["kind"]
    if kind == "verify":
        b, g, v = case["batch"], case["gamma"], case["vocab"]
        logits = b * v * ((g + 1) if case["temperature"] == 0 else (2 * g + 1))
        return {"bytes": 4 * logits + 4 * b * (2 * g + 3), "flops": 3 * logits}
    if kind == "sample":
        return {"bytes": 4 * case["rows"] * (case["vocab"] + 2), "flops": 3 * case["rows"] * case["vocab"]}
    if kind == "logits":
        cfg = workloads.model_config(case["model"])
        nbytes, flops = _pass_work(cfg, case["batch"], case["rows"], case["context"] + case["rows"], 0)
        return {"bytes": nbytes + 4 * case["batch"] * case["rows"] * cfg["vocab"], "flops": flops}
    target, draft = _pair(case)
    t5 = target["arch"] == "t5"
    g, b = case["gamma"], case["batch"]
    source = case["prompt"] * (1 - case["ragged"] / 2)  # mean length
    per_iteration = (1 - AGREE ** (g + 1)) / (1 - AGREE)
    iterations = math.ceil(case["n_new"] / per_iteration)
    context = case["n_new"] / 2 + (0 if t5 else source)
    nbytes = flops = 0
    for cfg, passes, rows in ((target, iterations, g + 1), (draft, iterations * g, 1)):
        elem = 2 if cfg["dtype"] == "bf16" else 4
        dec, enc = _matrices(cfg)
        head = cfg["vocab"] * cfg["d_model"]
        # the prompt (the source) through the blocks once
        met = enc if t5 else dec - head
        layers = cfg["n_enc_layers"] if t5 else cfg["n_layers"]
        seen = source if t5 else source / 2
        nbytes += met * elem + b * source * _kv_row(cfg)
        flops += b * source * (2 * met + 4 * seen * layers * cfg["n_heads"] * cfg["d_head"])
        one = _pass_work(cfg, b, rows, context, source if t5 else 0)
        nbytes += passes * one[0]
        flops += passes * one[1]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "logits":
        # (the same rows through the library's two attention kernels, whose sums run in different orders: rel 4.5e-4, max 2.1e-3)
        return {"rel": 2e-3, "max": 1e-2}
    # a uniform on the edge between two tokens may fall either way when a sum over the vocabulary is taken in another order
    return {"rel": 0.0, "differ": 0.01}
