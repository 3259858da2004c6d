"""Teacher-forced passes of one shape over and over: plain launches first, a captured pass from the third on."""
import numpy as np
import pytest
import torch

from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["llama_test_target", "tiny_draft"])  # bf16: captured; fp32: never
def test_repeated_passes_are_the_same_pass(model):
    cfg = workloads.model_config(model)
    eng = binding.Engine(cfg, workloads.make_weights(cfg, 1), max_batch=3, max_len=96, max_gamma=15)
    prefix = np.stack([workloads.make_prompt(i, 20, cfg["vocab"]) for i in range(3)])
    eng.forward_logits(0, prefix[:, :10])
    eng.forward_logits(0, prefix[:, 10:])
    for batch, rows in ((3, 4), (1, 1), (3, 1), (2, 4), (1, 3), (1, 4), (2, 1), (2, 2), (2, 3), (3, 4)):  # (more shapes than are kept)
        step = prefix[:batch, 3:3 + rows]
        other = prefix[:batch, 7:7 + rows]
        first = eng.forward_logits(0, step)
        for k in range(5):  # other tokens, other lengths and other output buffers in between change nothing
            eng.truncate(0, [20 - k] * batch)
            eng.forward_logits(0, other)
            if k:  # back to 20 cached rows, by passes of the length that wrote them
                eng.truncate(0, [0] * batch)
                eng.forward_logits(0, prefix[:batch, :10])
                eng.forward_logits(0, prefix[:batch, 10:])
            else:
                eng.truncate(0, [20] * batch)
            again = eng.forward_logits(0, step)
            assert torch.equal(first, again), (batch, rows, k)
            eng.truncate(0, [20] * batch)
    unaligned = torch.empty(3 * cfg["vocab"] + 1, device="cuda")[1:]
    tokens = np.ascontiguousarray(prefix[:3, :1], dtype=np.int32)
    want = eng.forward_logits(0, tokens)
    eng.truncate(0, [20] * 3)
    for _ in range(4):
        binding._check(binding.lib().spec_forward_logits(eng._ctx, 0, tokens.ctypes.data, 3, 1, unaligned.data_ptr()))
        eng.truncate(0, [20] * 3)
        assert torch.equal(unaligned.view(3, 1, -1), want)
    eng.close()
