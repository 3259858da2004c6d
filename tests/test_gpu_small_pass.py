"""Passes of at most eight rows of a small decoder, which run as one kernel: widths of one to three 256-input steps, groups
of one to four query heads per KV head, FFNs of fewer columns than thread blocks and of more, 1 .. 8 rows of one to eight
sequences, and contexts around the edges of sixteen keys, of a page and of what one step of all warps covers."""
import numpy as np
import pytest
import torch

from oracle.decoder import Decoder
from oracle.encdec import START_TOKEN, EncoderDecoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

# Keys and values are cached in fp16 (2^-11 of each) and activations are two bf16 terms (2^-17): logits of size one, sums
# over a few blocks of such values, agree with the oracle's to a few 2^-11.
LOGIT_TOL = 2e-2


@pytest.mark.parametrize("base,d_model,heads,kv_heads,d_ff", [
    ("llama_test_target", 256, 4, 2, 704),
    ("llama_test_target", 256, 4, 1, 2064),  # 129 units of sixteen columns: a second round for a few blocks
    ("llama_test_target", 768, 9, 3, 4096),  # three rounds; shared memory for two units' weights only with few rows
    ("gpt6m_draft", 512, 8, 8, 1024),
])
def test_few_rows_against_the_oracle(base, d_model, heads, kv_heads, d_ff):
    cfg = workloads.scaled_config(workloads.model_config(base), d_model=d_model, n_heads=heads, n_kv_heads=kv_heads, d_head=64,
                                  d_ff=d_ff, n_layers=2, tied=False, vocab=512, max_positions=512)
    w = workloads.make_weights(cfg, 3)
    oracle = Decoder(cfg, w)
    contexts = [300, 0, 17, 33, 16, 129, 1, 15]
    total = max(contexts) + 8
    tokens = np.stack([workloads.make_prompt(60 + b, total, cfg["vocab"]) for b in range(len(contexts))])
    want = [oracle.forward_full(t) for t in tokens]
    eng = binding.Engine(cfg, w, max_batch=len(contexts), max_len=total, page_size=32, max_gamma=31)
    for order in (slice(None), slice(None, None, -1)):
        lengths = contexts[order]
        toks, refs = tokens[order], want[order]
        eng.reset()
        for c in range(0, max(contexts), 30):
            eng.forward_logits(0, np.ascontiguousarray(toks[:, c:c + 30]))
        for batch, rows in ((1, 8), (8, 1), (4, 2), (2, 3), (3, 1), (1, 1), (2, 1), (1, 5), (5, 1), (1, 2)):
            eng.truncate(0, lengths)
            step = np.stack([toks[b, lengths[b]:lengths[b] + rows] for b in range(batch)])
            got = eng.forward_logits(0, step).cpu().numpy()
            for b in range(batch):
                err = np.abs(got[b] - refs[b][lengths[b]:lengths[b] + rows]).max()
                assert err <= LOGIT_TOL, (batch, rows, b, err)
    eng.close()


def test_few_rows_with_cross_attention():
    cfg = workloads.scaled_config(workloads.model_config("t5_test_target"), d_model=256, n_heads=4, n_kv_heads=4, d_ff=528)
    w = workloads.make_weights(cfg, 5)
    lengths = [70, 16, 1, 33]
    sources = [workloads.make_prompt(80 + i, n, cfg["vocab"]) for i, n in enumerate(lengths)]
    eng = binding.Engine(cfg, w, max_batch=4, max_len=64, page_size=32, max_gamma=15, max_src_len=80)
    tokens = np.stack([np.concatenate([[START_TOKEN], workloads.make_prompt(90 + b, 20, cfg["vocab"])]) for b in range(4)]).astype(np.int32)
    oracles = []
    for s in sources:
        o = EncoderDecoder(cfg, w)
        o.encode(s)
        oracles.append(o)
    want = [o.forward_rows(t) for o, t in zip(oracles, tokens)]
    for batch, rows in ((1, 1), (4, 2), (1, 8), (3, 1), (2, 4)):
        eng.encode(sources[:batch])
        at = 0
        while at + rows <= 20:
            got = eng.forward_logits(0, np.ascontiguousarray(tokens[:batch, at:at + rows])).cpu().numpy()
            for b in range(batch):
                err = np.abs(got[b] - want[b][at:at + rows]).max()
                assert err <= LOGIT_TOL * max(1.0, np.abs(want[b]).max()), (batch, rows, at, b, err)
            at += rows
    eng.close()


def test_a_decoder_of_one_block():
    """Only a few clusters of thread blocks would have a head, and nothing in one block makes the pass wait for the others: such a
    model is left to the chain of kernels.  Passes back to back, each right after the last."""
    cfg = workloads.scaled_config(workloads.model_config("llama_test_target"), d_model=256, n_heads=4, n_kv_heads=1, n_layers=1,
                                  tied=False, vocab=512, max_positions=512)
    w = workloads.make_weights(cfg, 7)
    tokens = workloads.make_prompt(50, 320, cfg["vocab"])
    want = Decoder(cfg, w).forward_full(tokens)
    eng = binding.Engine(cfg, w, max_batch=1, max_len=330, page_size=32, max_gamma=7)
    got = [eng.forward_logits(0, tokens[None, i:i + 1])[0] for i in range(320)]
    eng.close()
    assert np.abs(torch.cat(got).cpu().numpy() - want).max() <= LOGIT_TOL
    # drawn by generation too, whose passes follow one another without the host in between
    draft = workloads.scaled_config(cfg, n_heads=2, n_kv_heads=2)
    eng = binding.Engine(cfg, w, draft, workloads.make_weights(draft, 8), max_batch=1, max_len=330, page_size=32, max_gamma=3)
    greedy, _ = eng.generate([tokens[:20]], 200, 0, 0.0, 1)
    guessed, _ = eng.generate([tokens[:20]], 200, 3, 0.0, 1)
    eng.close()
    full = Decoder(cfg, w).forward_full(np.concatenate([tokens[:20], greedy[0]]))[19:-1]
    for stream in (greedy[0], guessed[0]):
        n = next((i for i in range(200) if stream[i] != greedy[0][i]), 199)
        gap = full[:n + 1].max(axis=1) - full[np.arange(n + 1), stream[:n + 1]]
        assert (gap <= 2 * LOGIT_TOL).all()


def test_more_blocks_than_the_packing_takes():
    """The pointers of at most 1820 blocks of the narrowest model fit the memory in which they reach the packing kernel: a deeper
    model's passes are the chain's, not a kernel's on weights that were never packed."""
    layers = 1821
    cfg = workloads.scaled_config(workloads.model_config("llama_test_target"), d_model=256, n_heads=1, n_kv_heads=1, d_ff=16,
                                  n_layers=layers, tied=False, vocab=64, max_positions=64)
    drawn = workloads.make_weights(workloads.scaled_config(cfg, n_layers=2), 13)
    # (two blocks' weights in turn, on the device once)
    matrices = ("wqkv", "wo", "w_in", "w_out")
    cuda = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda().to(torch.bfloat16 if k.split(".")[-1] in matrices + ("tok_emb", "head")
                                                                     else torch.float32) for k, v in drawn.items()}
    repeat = lambda w: {k: v for k, v in w.items() if "." not in k} | {
        f"l{l}.{n}": w[f"l{l % 2}.{n}"] for l in range(layers) for n in ("ln1", "ln2") + matrices}
    tokens = workloads.make_prompt(51, 3, cfg["vocab"])
    want = Decoder(cfg, repeat(drawn)).forward_full(tokens)
    eng = binding.Engine(cfg, repeat(cuda), max_batch=1, max_len=32, page_size=32, max_gamma=3)
    got = torch.cat([eng.forward_logits(0, tokens[None, i:i + 1])[0] for i in range(3)]).cpu().numpy()
    eng.close()
    # (fp16 keys and values, 2^-11 of each, block after block: the errors add up like the blocks' outputs do)
    assert np.abs(got - want).max() <= LOGIT_TOL * np.abs(want).max()
