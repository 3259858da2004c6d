"""The packed prompt pass: rows of all prompts one after another, segments cut by chunk ends, queries that do not fill a
block, prompts of one row and of none (a one-token prompt leaves nothing to feed)."""
import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

LOGIT_TOL = 2e-2  # of bf16 models against the oracle on the same rounded weights


@pytest.mark.parametrize("heads,kv_heads,d_head,page,lengths", [
    (4, 2, 64, 32, [500, 1, 497, 2, 400, 129, 330, 64, 449]),  # 2363 rows: two chunks of 1280 and less, prompts cut in between
    (4, 1, 128, 128, [33, 290, 257]),                          # four query heads on one KV head of 128
    (3, 3, 64, 64, [470]),                                     # a lone prompt, one query per KV head and row
])
def test_ragged_prompts_against_the_oracle(heads, kv_heads, d_head, page, lengths):
    cfg = workloads.scaled_config(workloads.model_config("llama_test_target"), n_heads=heads, n_kv_heads=kv_heads, d_head=d_head)
    w = workloads.make_weights(cfg, 3)
    draft = workloads.model_config("llama_test_draft")
    n_new = 5
    prompts = [workloads.make_prompt(40 + i, n, cfg["vocab"]) for i, n in enumerate(lengths)]
    eng = binding.Engine(cfg, w, draft, workloads.make_weights(draft, 4), max_batch=len(lengths), max_len=max(lengths) + n_new + 4,
                         page_size=page, max_gamma=2)
    got, _ = eng.generate(prompts, n_new, 2, 0.0, 1)
    eng.close()
    oracle = Decoder(cfg, w)
    for prompt, tokens in zip(prompts, got):
        logits = oracle.forward_full(np.concatenate([prompt, tokens[:-1]]).astype(np.int32))[len(prompt) - 1:]
        # every greedy token is an argmax of the oracle's logits, up to the tolerance on either side
        assert (logits.max(axis=1) - logits[np.arange(n_new), tokens] <= 2 * LOGIT_TOL).all(), len(prompt)
