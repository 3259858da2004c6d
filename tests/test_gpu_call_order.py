"""Tokens drawn by one call and verified by the next, with nothing between the two launches: the decision must see the drawn
tokens although its kernels may start early."""
import pytest
import torch

from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("temperature,top_k", [(1.0, 0), (0.0, 0), (1.0, 20)])
@pytest.mark.parametrize("batch,gamma", [(9, 1), (12, 3)])
def test_verification_right_behind_the_draws(batch, gamma, temperature, top_k):
    vocab = 8192
    tl, ql = workloads.make_sampler_logits(5, batch, gamma, vocab, 1.0)
    target, draft = torch.from_numpy(tl).cuda(), torch.from_numpy(ql).cuda()
    us = torch.from_numpy(workloads.make_uniform_grid(6, (batch, gamma + 1))).cuda()
    draws = torch.from_numpy(workloads.make_uniform_grid(7, (batch * gamma,))).cuda()
    tokens = torch.empty(batch * gamma, dtype=torch.int32, device="cuda")
    out = torch.empty((2, batch), dtype=torch.int32, device="cuda")
    ws = torch.empty(binding.spec_verify_sample_workspace_bytes(batch, gamma, vocab), dtype=torch.uint8, device="cuda")

    def sample():
        binding.spec_sample(draft.view(batch * gamma, vocab), draws, temperature, tokens=tokens, top_k=top_k)

    def verify():
        binding.spec_verify_sample(target, draft, tokens.view(batch, gamma), us, temperature, n_accepted=out[0], next_token=out[1],
                                   workspace=ws, top_k=top_k)

    sample()
    torch.cuda.synchronize()
    verify()
    torch.cuda.synchronize()
    want = out.clone()
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        sample()
        verify()
    for _ in range(20):
        tokens.fill_(-1)
        out.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
