"""fp32 models: the norm applied by the GEMM that follows and the FFN's function by its first GEMM, at every row tile and on
either side of the limits at which a launch changes (2, 4, 8, 64 rows; 2368 features to a warp each), with widths that fill
neither a lane's step nor a thread block."""
import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

# fp32 sums of a few thousand products in another order (2^-24 each, a few times over per block): relative to the largest logit
REL_TOL = 1e-4


@pytest.mark.parametrize("base,ffn,d_model,heads,kv_heads,d_ff", [
    ("llama_test_target", "swiglu", 200, 3, 1, 264),
    ("llama_test_target", "gated_gelu", 136, 2, 2, 2376),   # one feature more than a warp takes alone
    ("tiny_target", "gelu", 72, 1, 1, 2368),
    ("tiny_target", "gelu", 640, 4, 4, 96),                 # too wide for a fused norm beyond eight rows
])
def test_rows_against_the_oracle(base, ffn, d_model, heads, kv_heads, d_ff):
    cfg = workloads.scaled_config(workloads.model_config(base), ffn=ffn, d_model=d_model, n_heads=heads, n_kv_heads=kv_heads,
                                  d_head=64, d_ff=d_ff, n_layers=2, dtype="fp32", vocab=500, max_positions=256, tied=False)
    w = workloads.make_weights(cfg, 9)
    oracle = Decoder(cfg, w)
    batch = 5
    tokens = np.stack([workloads.make_prompt(30 + b, 120, cfg["vocab"]) for b in range(batch)])
    want = [oracle.forward_full(t) for t in tokens]
    eng = binding.Engine(cfg, w, max_batch=batch, max_len=128, max_gamma=31)
    at = 0
    for n, rows in ((5, 13), (1, 1), (2, 1), (3, 1), (4, 1), (5, 1), (4, 2), (3, 3), (5, 6), (4, 16), (5, 13)):  # 1 .. 65 rows in all
        eng.truncate(0, [at] * batch)
        got = eng.forward_logits(0, np.ascontiguousarray(tokens[:n, at:at + rows])).cpu().numpy()
        for b in range(n):
            ref = want[b][at:at + rows]
            assert np.abs(got[b] - ref).max() <= REL_TOL * np.abs(ref).max(), (n, rows, b)
        if n == batch:
            at += rows
    eng.close()
