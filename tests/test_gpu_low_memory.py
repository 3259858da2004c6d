"""Contexts on a GPU with little memory left: what only makes passes faster is left out, and what remains gives the same
results.  The memory is taken by one untouched block beside the context."""
import numpy as np
import pytest
import torch

from paper_2211_17192_b200 import binding, workloads

pytestmark = pytest.mark.gpu

MB = 1 << 20
LOGIT_TOL = 2e-2  # of bf16 models, on either side (see the parity tests)


class Fixture:
    """A decoder of the 160M shape whose weights are on the device already; contexts of it beside a block that leaves `free` bytes."""

    def __init__(self):
        self.cfg = workloads.model_config("llama160m_draft")
        self.weights = {}
        for name, shape, kind in workloads.tensor_shapes(self.cfg):
            gen = torch.Generator(device="cuda").manual_seed(len(self.weights))
            t = torch.ones(shape, device="cuda") if kind == "gain" else (torch.randn(shape, device="cuda", generator=gen) * 0.02).bfloat16()
            self.weights[name] = t
        self.tokens = np.stack([workloads.make_prompt(70 + b, 48, self.cfg["vocab"]) for b in range(2)])
        self.block = None

    def free(self):
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def leave(self, bytes):
        self.release()
        self.block = torch.empty(max(0, self.free() - bytes), dtype=torch.uint8, device="cuda")

    def release(self):
        self.block = None
        torch.cuda.empty_cache()

    def run(self):
        """Logits of a few few-row passes, tokens of a prompt, and what the context takes."""
        before = self.free()
        eng = binding.Engine(self.cfg, self.weights, max_batch=2, max_len=1100, max_gamma=15)
        took = before - self.free()
        try:
            eng.forward_logits(0, self.tokens[:, :16])
            logits = [eng.forward_logits(0, self.tokens[:, 16 + 2 * i:18 + 2 * i]).cpu() for i in range(6)]
            prompts = [workloads.make_prompt(80, 1000, self.cfg["vocab"]), workloads.make_prompt(81, 700, self.cfg["vocab"])]
            tokens, _ = eng.generate(prompts, 1, 0, 0.0, 0)
        finally:
            eng.close()
        return torch.cat(logits, 1), tokens, took


@pytest.fixture(scope="module")
def fixture():
    f = Fixture()
    f.run()  # (modules and the library's own memory)
    yield f
    f.release()


def test_a_context_without_room_for_the_packed_copy(fixture):
    roomy, tokens, most = fixture.run()
    try:
        fixture.leave(most + 256 * MB)  # it would fit, and leave nothing for graphs and the caller
        logits, _, took = fixture.run()
        assert took < most - 128 * MB
        assert (logits - roomy).abs().max() <= LOGIT_TOL
        fixture.leave(took + 64 * MB)  # now only the rest fits
        logits, same, _ = fixture.run()
        assert (logits - roomy).abs().max() <= LOGIT_TOL
        assert np.array_equal(same, tokens)
    finally:
        fixture.release()


def test_a_context_without_room_for_long_prompt_chunks(fixture):
    """Prompts go in chunks of 2048 rows, or of 256 where the partial sums of more would not leave room enough."""
    _, tokens, most = fixture.run()
    try:
        fixture.leave(most + 256 * MB)
        _, same, least = fixture.run()
        assert np.array_equal(same, tokens)
        # a context that packs no second copy takes less than this by what 1792 rows of partial sums need
        cfg = fixture.cfg
        rows = 1792 * 2 * cfg["d_ff"] * 4
        packed = 2 * sum(t.numel() for n, t in fixture.weights.items() if n.split(".")[-1] in ("wqkv", "wo", "w_in", "w_out"))
        assert least < most - packed - rows
        # and fits where it always has
        fixture.leave(least + 16 * MB)
        _, same, _ = fixture.run()
        assert np.array_equal(same, tokens)
    finally:
        fixture.release()


def test_repeated_passes_with_no_memory_left(fixture):
    """From the third pass of a shape on a context replays a captured one, if there is memory for it."""
    cfg = fixture.cfg
    eng = binding.Engine(cfg, fixture.weights, max_batch=2, max_len=96, max_gamma=15)
    outs = [torch.empty(2, rows, cfg["vocab"], device="cuda") for rows in (3, 1)]
    steps = [np.ascontiguousarray(fixture.tokens[:, 16:16 + rows]) for rows in (3, 1)]
    blocks = []

    def passes():
        for out, step in zip(outs, steps):
            eng.truncate(0, [16, 16])
            out.fill_(-1.0)
            torch.cuda.synchronize()
            binding._check(binding.lib().spec_forward_logits(eng._ctx, 0, step.ctypes.data, 2, step.shape[1], out.data_ptr()))

    try:
        eng.forward_logits(0, fixture.tokens[:, :16])
        passes()
        want = [out.cpu() for out in outs]
        passes()
        fixture.leave(8 * MB)
        for size in (2 * MB, MB // 2):
            try:
                while True:
                    blocks.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                pass
        for _ in range(4):
            passes()
            assert all(torch.equal(out.cpu(), w) for out, w in zip(outs, want))
    finally:
        blocks.clear()
        fixture.release()
        eng.close()
