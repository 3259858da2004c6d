"""Few logits are decided by one kernel, more by two: the same decision on either side of the line (eight sequences; 32768
logits per eight rows, 131072 at T = 0), with rows that start anywhere."""
import pytest
import torch

from gpu_util import compare_verify
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("temperature", [1.0, 0.0])
@pytest.mark.parametrize("gamma,vocab", [(1, 3), (3, 8191), (3, 32768), (3, 32769), (4, 16384), (4, 16386), (1, 131072), (1, 131073)])
def test_one_kernel_decides_as_two_do(gamma, vocab, temperature):
    tl, ql = workloads.make_sampler_logits(vocab + gamma, 3, gamma, vocab, 1.0)
    us = workloads.make_uniform_grid(vocab, (3, gamma + 1))
    place = lambda a: torch.from_numpy(a).to("cuda")
    t, q, u = place(tl), place(ql), place(us)
    xs = ql.argmax(axis=2).astype("int32")
    x = place(xs)
    got = binding.spec_verify_sample(t, q, x, u, temperature)  # three sequences
    flagged, _ = compare_verify(*got, tl, ql, xs, us, temperature)
    assert flagged == 0
    many = [a.repeat(3, *[1] * (a.dim() - 1)).contiguous() for a in (t, q, x, u)]  # nine
    n, token = binding.spec_verify_sample(*many, temperature)
    assert torch.equal(n, got[0].repeat(3)) and torch.equal(token, got[1].repeat(3))
    alone = binding.spec_verify_sample(t[1:2].contiguous(), q[1:2].contiguous(), x[1:2].contiguous(), u[1:2].contiguous(), temperature)
    assert int(alone[0][0]) == int(got[0][1]) and int(alone[1][0]) == int(got[1][1])
