"""Few-row passes of tiny fp32 decoders, which are one cluster of thread blocks: logits against the oracle for every number of
rows it takes (and one more, which the chain of kernels takes), over ragged caches from none to the most keys it serves."""
import numpy as np
import pytest
import torch

from oracle.decoder import Decoder
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

# fp32 sums of up to 1024 products in another order (2^-24 each, a few times over per block): relative to the largest logit
REL_TOL = 1e-4


@pytest.mark.parametrize("d_model,layers,max_len", [(128, 1, 256), (128, 2, 100), (256, 1, 64), (256, 4, 256)])
def test_cluster_pass_against_the_oracle(d_model, layers, max_len):
    cfg = workloads.scaled_config(workloads.model_config("tiny_target"), d_model=d_model, n_heads=d_model // 64, n_kv_heads=d_model // 64,
                                  d_ff=4 * d_model, n_layers=layers, vocab=500, max_positions=max_len)
    w = workloads.make_weights(cfg, 9)
    oracle = Decoder(cfg, w)
    batch, most = 9, max_len - 10
    tokens = np.stack([workloads.make_prompt(30 + b, most + 9, cfg["vocab"]) for b in range(batch)])
    want = [oracle.forward_full(t) for t in tokens]
    eng = binding.Engine(cfg, w, max_batch=batch, max_len=max_len, max_gamma=31, page_size=32)
    for at in range(0, most, 32):
        eng.forward_logits(0, np.ascontiguousarray(tokens[:, at:min(at + 32, most)]))
    for n, rows in ((1, 1), (2, 1), (3, 1), (4, 1), (5, 1), (7, 1), (8, 1), (9, 1), (1, 2), (1, 3), (1, 4), (1, 5), (1, 7), (1, 8), (1, 9),
                    (2, 2), (2, 3), (2, 4), (3, 2), (4, 2)):
        for lengths in ([0] * n, [(7 * b + 31) % most for b in range(n)], [most - (b % 5) for b in range(n)], [min(128, most) + b % 3 - 2 for b in range(n)]):
            eng.truncate(0, lengths + [most] * (batch - n))
            new = np.stack([tokens[b, lengths[b]:lengths[b] + rows] for b in range(n)])
            got = eng.forward_logits(0, new).cpu().numpy()
            for b in range(n):
                ref = want[b][lengths[b]:lengths[b] + rows]
                assert np.abs(got[b] - ref).max() <= REL_TOL * np.abs(ref).max(), (n, rows, lengths, b)
            # the cache whole again for the next case
            eng.truncate(0, [0] * batch)
            for at in range(0, most, 32):
                eng.forward_logits(0, np.ascontiguousarray(tokens[:, at:min(at + 32, most)]))
    eng.close()


def _tiny(layers, d_model):
    return workloads.scaled_config(workloads.model_config("tiny_target"), d_model=d_model, n_heads=d_model // 64, n_kv_heads=d_model // 64,
                                   d_ff=4 * d_model, n_layers=layers, vocab=500, max_positions=64)


@pytest.mark.parametrize("d_model", [128, 256])
@pytest.mark.parametrize("part", [0, 1, 2], ids=["q", "k", "v"])
def test_a_score_that_is_no_number_reaches_the_logits(d_model, part):
    """A NaN in the rows of Wqkv that make a head's q, k or v: every logit of a pass of one block is one, and generation reports it."""
    cfg = _tiny(1, d_model)
    w = dict(workloads.make_weights(cfg, 9))
    w["l0.wqkv"] = w["l0.wqkv"].copy()
    w["l0.wqkv"][part * d_model + 64 + 5] = np.nan
    tokens = workloads.make_prompt(3, 12, cfg["vocab"])
    eng = binding.Engine(cfg, w, max_batch=1, max_len=64, max_gamma=8, page_size=32)
    got = [eng.forward_logits(0, tokens[None, at:at + 3]) for at in (0, 3, 6)]
    assert all(g.isnan().all() for g in got)
    with pytest.raises(binding.SpecError) as e:
        eng.generate([tokens[:3]], 8, 0, 1.0, 1)
    assert e.value.status == -7
    eng.close()


@pytest.mark.parametrize("d_model", [128, 256])
def test_a_row_that_is_no_number_is_nothing_to_the_rows_in_front_of_it(d_model):
    cfg = _tiny(2, d_model)
    w = dict(workloads.make_weights(cfg, 9))
    w["tok_emb"] = w["tok_emb"].copy()
    w["tok_emb"][7] = np.nan
    tokens = np.array([[1, 2, 3, 4, 5, 7]], dtype=np.int32)
    eng = binding.Engine(cfg, w, max_batch=1, max_len=64, max_gamma=8, page_size=32)
    eng.forward_logits(0, tokens[:, :2])
    got = eng.forward_logits(0, tokens[:, 2:])
    assert got[0, 3].isnan().all() and got[0, :3].isfinite().all()
    eng.truncate(0, [2])
    assert torch.equal(eng.forward_logits(0, np.array([[3, 4, 5, 6]], dtype=np.int32))[0, :3], got[0, :3])
    eng.close()


@pytest.mark.parametrize("d_model", [128, 256])
def test_pages_of_any_size(d_model):
    cfg = _tiny(2, d_model)
    w = workloads.make_weights(cfg, 9)
    tokens = np.stack([workloads.make_prompt(b, 60, cfg["vocab"]) for b in range(2)])
    want = None
    for page_size in (32, 64, 256):
        eng = binding.Engine(cfg, w, max_batch=2, max_len=64, max_gamma=8, page_size=page_size)
        got = torch.cat([eng.forward_logits(0, np.ascontiguousarray(tokens[:, at:at + 2])) for at in range(0, 60, 2)], dim=1)
        eng.close()
        want = got if want is None else want
        assert torch.equal(got, want), page_size


def test_rows_beyond_what_the_context_holds():
    """One sequence takes more guesses than the other and is frozen early, at lengths whose guesses lie beyond the last position
    among others.  Each gets the tokens it gets alone."""
    cfg = _tiny(2, 128)
    w = workloads.make_weights(cfg, 9)
    d = dict(w)
    d["pos_emb"] = w["pos_emb"].copy()
    d["pos_emb"][:20] = np.random.default_rng(1).standard_normal((20, 128), dtype=np.float32)
    prompts = [workloads.make_prompt(1, 30, cfg["vocab"]), workloads.make_prompt(2, 3, cfg["vocab"])]
    gamma, frozen = 3, 0
    for n_new in range(8, 17):
        eng = binding.Engine(cfg, w, cfg, d, max_batch=2, max_len=30 + n_new + gamma + 1, max_gamma=gamma, page_size=32)
        alone = [eng.generate([p], n_new, gamma, 0.0, 1) for p in prompts]
        frozen += alone[0][1]["iterations"] < alone[1][1]["iterations"]
        both, _ = eng.generate(prompts, n_new, gamma, 0.0, 1)
        eng.close()
        for b in range(2):
            assert (both[b] == alone[b][0][0]).all(), n_new
    assert frozen
