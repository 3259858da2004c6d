"""Contexts of several threads on one device, set up and used at the same time in a process that has launched nothing yet: one
thread at a time opts a kernel into its shared memory, and the others wait for it."""
import os
import subprocess
import sys

import pytest

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
