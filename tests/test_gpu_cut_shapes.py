"""A row's cut is the same however the rows are shared out: alone, where a cluster of thread blocks takes it, among few, among
as many as fit on the GPU at once and among more (the number of rows at which the launch changes, and one more)."""
import numpy as np
import pytest
import torch

from paper_2211_17192_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top_k,top_p", [(0, 0.9), (40, 1.0), (50, 0.95), (129, 0.9), (300, 1.0)])
@pytest.mark.parametrize("vocab", [4099, 12288, 49152, 50003])
def test_floors_and_draws_do_not_depend_on_the_number_of_rows(vocab, top_k, top_p):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(vocab + top_k)
    few = torch.randn(5, vocab, device="cuda", generator=gen) * torch.tensor([0.5, 1.0, 2.0, 4.0, 8.0], device="cuda")[:, None]
    few[1, ::3] = 0.25  # heavy ties, where the cut may fall
    few[2, 7] = -torch.inf
    u = torch.rand(5, device="cuda", generator=gen)
    floors = torch.cat([binding.spec_truncation_floors(few[i:i + 1].contiguous(), 0.8, top_k=top_k, top_p=top_p) for i in range(5)])
    tokens = torch.cat([binding.spec_sample(few[i:i + 1].contiguous(), u[i:i + 1].contiguous(), 0.8, top_k=top_k, top_p=top_p) for i in range(5)])
    # by hand, in double precision: what a floor keeps is at least k logits, or at least top_p of the mass of what top-k keeps
    for i in range(5):
        row = np.sort(few[i].double().cpu().numpy())[::-1]
        kept = row >= float(floors[i])
        allowed = row >= row[top_k - 1] if top_k else np.ones_like(kept)
        mass = np.where(allowed, np.exp((row - row[0]) / 0.8), 0.0)
        if top_p < 1.0:
            # (masses are summed in units of 2^-32 of the largest, rounded down, and a weight is good to 2^-21)
            slack = vocab * 2.0 ** -31 + mass.sum() * 2.0 ** -20
            assert mass[kept].sum() >= top_p * mass.sum() - slack
            # and no less would do
            assert mass[row > float(floors[i])].sum() < top_p * mass.sum() + slack
        else:
            assert float(floors[i]) == row[top_k - 1]
        assert float(few[i, int(tokens[i])]) >= float(floors[i])
    for rows in (5, 74, 75, 148, 149, 296, 297, 592, 593):
        many = few.repeat((rows + 4) // 5, 1)[:rows].contiguous()
        us = u.repeat((rows + 4) // 5)[:rows].contiguous()
        got = binding.spec_truncation_floors(many, 0.8, top_k=top_k, top_p=top_p)
        assert torch.equal(got, floors.repeat((rows + 4) // 5)[:rows]), rows
        drawn = binding.spec_sample(many, us, 0.8, top_k=top_k, top_p=top_p)
        # (weights are added in another order: 2^-20 of their sum at most, so a uniform number next to a step may fall on
        # the other side; of five, none is)
        assert torch.equal(drawn, tokens.repeat((rows + 4) // 5)[:rows]), rows


@pytest.mark.parametrize("rows,vocab", [(1, 12288), (3, 12289), (2, 49152), (149, 50003), (150, 110000), (300, 12291), (600, 4099)])
@pytest.mark.parametrize("top_p", [0.1, 0.9, 0.999])
def test_nucleus_of_rows_whose_sample_misleads(rows, vocab, top_p):
    """The nucleus is looked for among the logits that a sample of the row says to list.  Rows where that is wrong or no use: flat
    ones, mass in a stretch that the sample misses, weight where it looks, more candidates in one stretch than a warp's list
    holds, masked logits, few finite ones, ties."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(vocab)
    base = torch.randn(10, vocab, device="cuda", generator=gen)
    base[0] *= 3
    base[1] *= 0.01
    base[2] = 1.0
    base[3, vocab // 2 + 300: vocab // 2 + 900] += 9
    base[4, :128] += 5
    base[5, vocab // 3: vocab // 3 + vocab // 8] += 6
    base[6, 1::2] = -torch.inf
    base[7, 17:] = -torch.inf
    base[8] = base[8].mul(2).round()
    base[9, : vocab // 2] -= 40
    many = base.repeat((rows + 9) // 10, 1)[:rows].contiguous()
    got = binding.spec_truncation_floors(many, 0.8, top_p=top_p)
    again = binding.spec_truncation_floors(many, 0.8, top_p=top_p)
    assert torch.equal(got, again)
    u = torch.rand(rows, device="cuda", generator=gen)
    tokens = binding.spec_sample(many, u, 0.8, top_p=top_p)
    for i in range(min(rows, 10)):
        row = np.sort(many[i].double().cpu().numpy())[::-1]
        floor = float(got[i])
        weight = np.exp((row - row[0]) / 0.8)
        # (as above: 2^-32 of the largest per logit, a weight good to 2^-21, sums in fp32)
        slack = vocab * 2.0 ** -31 + weight.sum() * 2.0 ** -20
        assert weight[row >= floor].sum() >= top_p * weight.sum() - slack, i
        assert weight[row > floor].sum() < top_p * weight.sum() + slack, i
        assert float(many[i, int(tokens[i])]) >= floor, i
    for i in range(10, rows):
        assert float(got[i]) == float(got[i % 10]), i


@pytest.mark.parametrize("vocab,many,few", [(8192, 1184, (148,)), (4099, 1184, (148,)), (12289, 1184, (296, 61)), (50003, 600, (200, 100, 40))])
@pytest.mark.parametrize("temperature,shift,top_p", [(1.0, 0.0, 0.9), (0.05, 100.0, 0.9), (0.7, -3000.0, 0.5)])
def test_a_nucleus_is_the_same_from_bins_and_from_a_list(vocab, many, few, temperature, shift, top_p):
    """Floors to the last bit over hundreds of random rows: many in one call against the same rows a few at a time, which other
    launches take (short rows: bins, not lists).  Also at a temperature and a shift that leave few bits of the weights' exponents."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(vocab)
    rows = torch.randn(many, vocab, device="cuda", generator=gen) * (3.0 * temperature) + shift
    want = binding.spec_truncation_floors(rows, temperature, top_p=top_p)
    assert len(torch.unique(want)) > many // 2
    for n in few:
        got = torch.cat([binding.spec_truncation_floors(rows[i:i + n].contiguous(), temperature, top_p=top_p) for i in range(0, many, n)])
        differ = int((got != want).sum())
        assert differ == 0, (n, differ)


@pytest.mark.parametrize("rows,vocab", [(1, 50003), (40, 100000), (130, 60001), (200, 100000), (310, 8192), (600, 20000)])
@pytest.mark.parametrize("top_p", [0.5, 0.9, 0.95])
def test_a_nucleus_is_the_same_wherever_its_logits_lie(rows, vocab, top_p):
    """A row shuffled, sorted, sorted the other way, and with its large logits in one stretch: one floor, and not much more time."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(vocab)
    shuffled = torch.randn(rows, vocab, device="cuda", generator=gen) * 3
    falling = shuffled.sort(dim=-1, descending=True).values
    tenth = vocab // 10
    inside = torch.cat([falling[:, tenth:4 * tenth], falling[:, torch.randperm(tenth, device="cuda", generator=gen)], falling[:, 4 * tenth:]], dim=1)
    want = binding.spec_truncation_floors(shuffled, 1.0, top_p=top_p)
    u = torch.rand(rows, device="cuda", generator=gen)
    tokens = torch.empty(rows, dtype=torch.int32, device="cuda")

    def microseconds(logits):
        times = []
        for _ in range(15):
            start, stop = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(4):
                binding.spec_sample(logits, u, 1.0, tokens=tokens, top_p=top_p)
            stop.record()
            stop.synchronize()
            times.append(start.elapsed_time(stop) * 250)
        return sorted(times)[len(times) // 2]

    usual = microseconds(shuffled)
    for other in (falling, falling.flip(1).contiguous(), inside.contiguous()):
        assert torch.equal(binding.spec_truncation_floors(other, 1.0, top_p=top_p), want)
        # (up to 1.45 times as long, and 2 to 3 times where a list that one warp overflows leaves the row to the bins; a nucleus
        # of 0.95 is at the edge of what is listed, so that chance decides which rows are)
        if top_p < 0.95:
            assert microseconds(other) <= 1.7 * usual + 2.0
