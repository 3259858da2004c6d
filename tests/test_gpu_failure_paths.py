"""Failure paths of the library, exercised without faulting the GPU: non-finite logits are
reported (not sampled from in silence), and a bounded device-side wait that runs out
comes back as a status while the context stays usable."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import sampling as oracle_sampling
from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu


def _pair():
    tcfg, dcfg = workloads.model_config("llama_test_target"), workloads.model_config("llama_test_draft")
    return tcfg, workloads.make_weights(tcfg, 1), dcfg, workloads.make_weights(dcfg, 2)


@pytest.mark.parametrize("which,value,temperature,gamma", [
    ("target", np.nan, 1.0, 3), ("target", np.inf, 1.0, 3), ("target", np.nan, 0.0, 2),
    ("draft", np.nan, 1.0, 3), ("draft", np.nan, 0.0, 2), ("target", np.nan, 1.0, 0),
])
def test_non_finite_logits_are_reported(which, value, temperature, gamma):
    """A NaN (or +inf) planted in one row of an LM head makes one logit of every row non-finite:
    the generation call returns SPEC_ERR_NONFINITE; the same pair without it generates."""
    tcfg, tw, dcfg, dw = _pair()
    prompt = workloads.make_prompt(3, 8, tcfg["vocab"])
    good = binding.Engine(tcfg, tw, dcfg, dw, max_batch=1, max_len=64, page_size=32, max_gamma=3)
    out, stats = good.generate([prompt], 12, gamma, temperature, 1)
    assert out.shape == (1, 12)
    good.close()
    bad_t, bad_d = dict(tw), dict(dw)
    victim = bad_t if which == "target" else bad_d
    head = victim["head"].copy()
    head[7, :] = value
    victim["head"] = head
    eng = binding.Engine(tcfg, bad_t, dcfg, bad_d, max_batch=1, max_len=64, page_size=32, max_gamma=3)
    try:
        with pytest.raises(binding.SpecError) as e:
            eng.generate([prompt], 12, gamma, temperature, 1)
        assert e.value.status == -7
    finally:
        eng.close()


@pytest.mark.parametrize("part", [0, 1, 2], ids=["q", "k", "v"])
@pytest.mark.parametrize("base,rows", [("tiny_target", 9), ("tiny_target", 40), ("t5_tiny_target", 5)])
def test_a_score_that_is_no_number_reaches_the_logits_of_fp32_models(base, rows, part):
    """A NaN in the rows of Wqkv that make a head's q, k or v: no row of the pass (a chain of kernels at these sizes) has a finite logit
    of it, whether a row's key slices are merged in a cluster or by a kernel of their own."""
    cfg = workloads.scaled_config(workloads.model_config(base), n_layers=1)
    w = dict(workloads.make_weights(cfg, 9))
    w["l0.wqkv"] = w["l0.wqkv"].copy()
    w["l0.wqkv"][part * cfg["n_heads"] * 64 + 64 + 5] = np.nan
    t5 = cfg["arch"] == "t5"
    for max_len in (64, 128):
        eng = binding.Engine(cfg, w, max_batch=1, max_len=max_len, max_gamma=rows, page_size=32, max_src_len=40 if t5 else 0)
        if t5:
            eng.encode([workloads.make_prompt(5, 40, cfg["vocab"])])
        assert eng.forward_logits(0, workloads.make_prompt(3, rows, cfg["vocab"])[None]).isnan().all()
        eng.close()


def test_a_bounded_wait_that_runs_out_is_reported_and_leaves_the_library_usable():
    h = binding.lib()
    h.spec_timeout_drill.restype = ctypes.c_int
    h.spec_timeout_drill.argtypes = [ctypes.c_void_p]
    torch.cuda.synchronize()
    assert binding.spec_device_error() == 0
    status = h.spec_timeout_drill(torch.cuda.current_stream().cuda_stream)
    assert status == -6, h.spec_last_error().decode()      # SPEC_ERR_DEVICE_TIMEOUT, as the drill intends
    assert b"gave up on a bounded wait" in h.spec_last_error()
    assert binding.spec_device_error() == 0                  # the drill consumed the flag it raised
    # the same kernel does its work right afterwards
    rng = np.random.default_rng(0)
    x = rng.standard_normal((3, 256)).astype(np.float32)
    w = workloads.round_to_bf16(rng.standard_normal((384, 256)).astype(np.float32) * 0.05)
    got = binding.spec_linear(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda().to(torch.bfloat16), "tensor").cpu().numpy()
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    assert binding.spec_device_error() == 0


@pytest.mark.parametrize("base", ["llama_test_target", "t5_test_target", "tiny_target", "tiny_draft"])
def test_a_one_kernel_pass_whose_exchange_never_comes(base):
    """No CTA of the pass publishes its share: all of them give up and go on, the next call reports it, and the pass after it is
    what it was before."""
    cfg = workloads.scaled_config(workloads.model_config(base), n_layers=3)
    eng = binding.Engine(cfg, workloads.make_weights(cfg, 4), max_batch=1, max_len=64, page_size=32, max_gamma=7,
                         max_src_len=40 if cfg["arch"] == "t5" else 0)
    h = binding.lib()
    h.spec_timeout_drill_pass.restype = ctypes.c_int
    h.spec_timeout_drill_pass.argtypes = [ctypes.c_void_p, ctypes.c_int]
    try:
        if cfg["arch"] == "t5":
            eng.encode([workloads.make_prompt(5, 40, cfg["vocab"])])
        tokens = workloads.make_prompt(3, 12, cfg["vocab"])[None]
        eng.forward_logits(0, tokens[:, :8])
        want = [eng.forward_logits(0, tokens[:, i:i + 1]) for i in range(8, 12)]
        for _ in range(3):
            eng.truncate(0, [8])
            assert h.spec_timeout_drill_pass(eng._ctx, 0) == -6, h.spec_last_error().decode()
            assert b"gave up on a bounded wait" in h.spec_last_error()
            assert binding.spec_device_error() == 0
            for i in range(8, 12):
                assert torch.equal(eng.forward_logits(0, tokens[:, i:i + 1]), want[i - 8])
    finally:
        eng.close()
    chain = workloads.scaled_config(cfg, n_layers=17 if cfg["dtype"] == "fp32" else 1)  # (one block of bf16, more than sixteen of fp32)
    eng = binding.Engine(chain, workloads.make_weights(chain, 4), max_batch=1, max_len=64, page_size=32, max_src_len=40 if cfg["arch"] == "t5" else 0)
    assert h.spec_timeout_drill_pass(eng._ctx, 0) == -2
    eng.close()



    """T = 0 with a drafted token that is not the draft's own maximum (x ~ q cannot produce it,
    so Algorithm 1's test decides nothing): library and oracle accept it iff it is the
    target's maximum."""
    vocab, gamma = 64, 2
    tl, ql = workloads.make_sampler_logits(5, 3, gamma, vocab, 1.0)
    xs = np.zeros((3, gamma), dtype=np.int32)
    top = tl.argmax(axis=-1)                     # [3, gamma + 1]
    draft_top = ql.argmax(axis=-1)
    xs[0] = [top[0, 0], top[0, 1]]               # the target's maxima (whatever the draft prefers): both accepted
    xs[1] = [top[1, 0], (top[1, 1] + 1) % vocab]  # second guess is not the target's maximum: rejected there
    xs[2] = [(draft_top[2, 0] + 3) % vocab if (draft_top[2, 0] + 3) % vocab != top[2, 0] else (draft_top[2, 0] + 4) % vocab, top[2, 1]]
    us = workloads.make_uniform_grid(6, (3, gamma + 1))
    n, t = binding.spec_verify_sample(torch.from_numpy(tl).cuda(), torch.from_numpy(ql).cuda(), torch.from_numpy(xs).cuda(),
                                      torch.from_numpy(us).cuda(), 0.0)
    n, t = n.cpu().numpy(), t.cpu().numpy()
    assert n.tolist() == [2, 1, 0]
    for b in range(3):
        ref = oracle_sampling.verify_step(tl[b], ql[b], xs[b], us[b], 0.0)
        assert (int(n[b]), int(t[b])) == (ref.n_accepted, ref.next_token)
        assert t[b] == top[b, n[b]]
