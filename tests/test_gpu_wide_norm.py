"""Rows of a wide bf16 decoder, normalised by a cluster of thread blocks each: widths from the first that takes a cluster to
the last, one that leaves a part of its threads without elements, and numbers of rows on either side of the limit."""
import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

# Keys and values are cached in fp16 (2^-11 of each) and activations are two bf16 terms (2^-17): sums over two blocks of such
# values agree with the oracle's to a few 2^-11 of the largest logit.
REL_TOL = 8e-3


@pytest.mark.parametrize("d_model", [2048, 2056, 3000, 4096])
def test_rows_against_the_oracle(d_model):
    cfg = workloads.scaled_config(workloads.model_config("llama_test_target"), d_model=d_model, n_heads=4, n_kv_heads=2, d_head=64,
                                  d_ff=520, n_layers=2, tied=False, vocab=512, max_positions=128)
    w = workloads.make_weights(cfg, 11)
    oracle = Decoder(cfg, w)
    batch = 5
    tokens = np.stack([workloads.make_prompt(40 + b, 60, cfg["vocab"]) for b in range(batch)])
    want = [oracle.forward_full(t) for t in tokens]
    eng = binding.Engine(cfg, w, max_batch=batch, max_len=64, max_gamma=31)
    at = 0
    for n, rows in ((5, 7), (1, 1), (1, 3), (4, 4), (3, 11), (4, 16), (5, 13), (4, 32), (5, 26)):  # 1 .. 130 rows in all
        eng.truncate(0, [at] * batch)
        got = eng.forward_logits(0, np.ascontiguousarray(tokens[:n, at:at + rows])).cpu().numpy()
        for b in range(n):
            ref = want[b][at:at + rows]
            assert np.abs(got[b] - ref).max() <= REL_TOL * np.abs(ref).max(), (n, rows, b)
        if n == batch:
            at += rows
    eng.close()
