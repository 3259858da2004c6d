"""Rows that start anywhere: vocabularies of every remainder mod 4, on either side of the width at which the selection
kernel takes its large CTAs, and logits that begin off a 16-byte boundary."""
import numpy as np
import pytest
import torch

from gpu_util import compare_verify, to_dev
from oracle import sampling as oracle_sampling
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab", [1, 2, 5, 1022, 1023, 49151, 49152, 49153, 49154])
@pytest.mark.parametrize("temperature,top_k,top_p", [(1.0, 0, 1.0), (0.0, 0, 1.0), (0.8, 40, 1.0), (1.0, 130, 1.0), (1.0, 0, 0.9), (0.7, 40, 0.9)])
def test_any_alignment_against_the_oracle(vocab, temperature, top_k, top_p):
    batch, gamma = 3, 2
    tl, ql = workloads.make_sampler_logits(vocab + gamma, batch, gamma, vocab, 1.0)
    us = workloads.make_uniform_grid(vocab, (batch, gamma + 1))
    draw = workloads.make_uniform_grid(vocab + 1, (batch, gamma))
    xs = np.array([[oracle_sampling.sample_token(ql[b, i], draw[b, i], 1.0)[0] for i in range(gamma)] for b in range(batch)],
                  dtype=np.int32)
    for offset in (0, 1):  # in floats: with 1 even a vocabulary that is a multiple of four has no aligned row
        def place(a):
            flat = torch.empty(a.size + offset, device="cuda")[offset:]
            return flat.view(a.shape).copy_(torch.from_numpy(a))
        n, t = binding.spec_verify_sample(place(tl), place(ql), to_dev(xs), to_dev(us), temperature, top_k=top_k, top_p=top_p)
        flagged, _ = compare_verify(n, t, tl, ql, xs, us, temperature, top_k=top_k, top_p=top_p)
        assert flagged <= 1
        rows = tl.reshape(-1, vocab)
        tokens = binding.spec_sample(place(rows), to_dev(us.reshape(-1)), temperature, top_k=top_k, top_p=top_p).cpu().numpy()
        for r in range(rows.shape[0]):
            token, margin = oracle_sampling.sample_token(rows[r], us.reshape(-1)[r], temperature, top_k, top_p)[:2]
            assert tokens[r] == token or margin < 1e-5 or top_p < 1.0 and oracle_sampling.nucleus_floor(rows[r], temperature, top_k, top_p)[1] < 5e-5


def test_numbers_of_any_kind_as_options():
    vocab, batch, gamma = 300, 2, 2
    tl, ql = workloads.make_sampler_logits(1, batch, gamma, vocab, 1.0)
    us = workloads.make_uniform_grid(2, (batch, gamma + 1))
    xs = ql.argmax(axis=2).astype(np.int32)
    t, q, x, u = to_dev(tl), to_dev(ql), to_dev(xs), to_dev(us)
    want = binding.spec_verify_sample(t, q, x, u, 0.75, lenience=0.5, top_k=40, top_p=0.875)
    for kind in (np.float32, np.float64, torch.tensor):
        got = binding.spec_verify_sample(t, q, x, u, kind(0.75), lenience=kind(0.5), top_k=kind(40.0), top_p=kind(0.875))
        assert all(torch.equal(a, b) for a, b in zip(got, want))
