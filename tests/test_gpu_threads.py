"""Contexts beside other work.  Of several threads on one device, set up and used at the same time in a process that has
launched nothing yet: one thread at a time opts a kernel into its shared memory, and the others wait for it.  And made of weights
that a stream is still writing."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

SCRIPT = """
import threading
import numpy as np, torch
from paper_2211_17192_b200 import binding, workloads

cfg = workloads.model_config("llama_test_target")
draft = workloads.scaled_config(cfg, n_layers=2)
weights, draft_weights = workloads.make_weights(cfg, 1), workloads.make_weights(draft, 2)
prompts = [workloads.make_prompt(3, 200, cfg["vocab"]), workloads.make_prompt(4, 150, cfg["vocab"])]
torch.zeros(1, device="cuda")
start = threading.Barrier(6)
results = [None] * 6

def work(i):
    torch.cuda.set_device(0)
    try:
        start.wait()
        eng = binding.Engine(cfg, weights, draft, draft_weights, max_batch=2, max_len=256, max_gamma=3)
        results[i] = [eng.generate(prompts, 24, 3, 1.0, 5)[0] for _ in range(3)]
        eng.close()
    except Exception as e:
        results[i] = e

threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
for t in threads: t.start()
for t in threads: t.join()
for r in results:
    if isinstance(r, Exception): raise r
    for tokens in r: assert np.array_equal(tokens, results[0][0])
print("same")
"""


def test_contexts_of_six_threads_in_a_fresh_process():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    done = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=240)
    assert done.returncode == 0 and done.stdout.strip() == "same", done.stderr[-2000:]


@pytest.mark.parametrize("model", ["gpt6m_draft", "llama_test_target", "tiny_draft"])
def test_weights_that_a_stream_is_still_writing(model):
    """A context is made while the stream that is current has yet to write the weights (behind a kernel that takes a while)."""
    cfg = workloads.model_config(model)
    dtype = torch.bfloat16 if cfg["dtype"] == "bf16" else torch.float32
    weights = {}
    for name, shape, kind in workloads.tensor_shapes(cfg):
        gen = torch.Generator(device="cuda").manual_seed(len(weights))
        weights[name] = torch.ones(shape, device="cuda") if kind == "gain" else (torch.randn(shape, device="cuda", generator=gen) * 0.05).to(dtype)
    tokens = workloads.make_prompt(2, 6, cfg["vocab"])[None]
    eng = binding.Engine(cfg, weights, max_len=32, max_gamma=7)
    want = eng.forward_logits(0, tokens)
    eng.close()
    late = {name: torch.zeros_like(t) for name, t in weights.items()}
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)  # (a fifth of a second)
        for name, t in weights.items():
            late[name].copy_(t)
        eng = binding.Engine(cfg, late, max_len=32, max_gamma=7)
    got = eng.forward_logits(0, tokens)
    eng.close()
    assert torch.equal(got, want)
