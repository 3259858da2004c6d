"""Many rows of a wide block, against the oracle, on either side of the lines at which the small kernels between the GEMMs change:
four rows to a thread of the activation (from 111 rows of this shape on), a norm that leaves its factor to it and to the
projection's (up to 128), a cluster of four thread blocks to a row (up to 296) and one (beyond); row counts that are no multiple of four."""
import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

# Keys and values are cached in fp16 (2^-11 of each) and activations are two bf16 terms (2^-17): sums over a block of such
# values agree with the oracle's to a few 2^-11 of the largest logit.
REL_TOL = 8e-3


def test_rows_against_the_oracle():
    cfg = workloads.scaled_config(workloads.model_config("llama7b_target"), d_model=2056, n_layers=1, vocab=512, max_positions=320)
    w = workloads.make_weights(cfg, 13)
    oracle = Decoder(cfg, w, dtype=np.float32)
    batch = 7
    passes = ((2, 55), (3, 37), (2, 63), (2, 64), (3, 43), (7, 42), (7, 43), (7, 56), (7, 57), (7, 60))  # 110, 111, 126, 128, 129, 294, 301, 392, 399, 420
    tokens = np.stack([workloads.make_prompt(60 + b, 300, cfg["vocab"]) for b in range(batch)])
    want = [oracle.forward_full(t) for t in tokens]
    eng = binding.Engine(cfg, w, max_batch=batch, max_len=304, max_gamma=63)
    at = 0
    for n, rows in passes:
        eng.truncate(0, [at] * batch)
        got = eng.forward_logits(0, np.ascontiguousarray(tokens[:n, at:at + rows])).cpu().numpy()
        for b in range(n):
            ref = want[b][at:at + rows]
            assert np.abs(got[b] - ref).max() <= REL_TOL * np.abs(ref).max(), (n, rows, b)
        if n == batch:
            at += rows
    eng.close()
