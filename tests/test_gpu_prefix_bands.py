"""The prefix join's signatures over relations of many keys: a warp takes its keys in
bands over the whole relation.  Every row's match is found for sizes around whole
bands, on either side, and a run of long keys takes no longer than the same keys
shuffled."""
import pytest
import torch

pytestmark = pytest.mark.gpu

WARPS, BAND = 16, 256                                      # per SM; keys of a warp in a band


def fixed(ag, rows):
    n, w = rows.shape
    return ag.DeviceRelation(torch.cat([rows.reshape(-1), torch.zeros(16, dtype=torch.uint8, device="cuda")]),
                             torch.arange(n + 1, dtype=torch.int64, device="cuda") * w)


def numbered(numbers, width, gen):
    """Keys of `width` bytes: the number in the first 8, the rest random."""
    rows = torch.randint(0, 256, (numbers.numel(), width), dtype=torch.uint8, device="cuda", generator=gen)
    rows[:, :8] = numbers.view(-1, 1).contiguous().view(torch.uint8)
    return rows


@pytest.mark.parametrize("bands,more", [(1, 5), (2, -1), (2, 0), (2, 1), (2, 33), (3, -32), (3, 7000)])
@pytest.mark.parametrize("side", ["S", "R"])
def test_every_row_signed(cuda, side, bands, more):
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(100 * bands + more + 50)
    n = torch.cuda.get_device_properties(0).multi_processor_count * WARPS * BAND * bands + more
    few = torch.arange(997, dtype=torch.int64, device="cuda") * 0x9E3779B97F4A7C1
    if side == "S":                                        # every S row has one partner among few R rows
        src = torch.randint(0, few.numel(), (n,), device="cuda", generator=gen)
        dR, dS = fixed(ag, numbered(few, 24, gen)), fixed(ag, numbered(few[src], 17, gen))
        want_r, want_s = src, torch.arange(n, device="cuda")
    else:                                                  # distinct R rows, some of them looked up
        every = torch.arange(n, dtype=torch.int64, device="cuda")
        look = torch.cat([every[:3000], every[-3000:], torch.randint(0, n, (100_000,), device="cuda", generator=gen)])
        dR, dS = fixed(ag, numbered(every, 17, gen)), fixed(ag, numbered(look, 24, gen))
        want_r, want_s = look, torch.arange(look.numel(), device="cuda")
    pairs = ag.join_prefix(dR, dS, 8)
    assert pairs.shape[0] == want_s.numel()
    got = torch.empty(want_s.numel(), dtype=torch.int32, device="cuda").fill_(-1)
    got[pairs[:, 1].long()] = pairs[:, 0]
    assert torch.equal(got.long(), want_r)


def test_order_of_lengths_costs_nothing(cuda):
    """1.3M keys of 64 bytes and 60k of 8 KB under a cap above all of them."""
    ag = cuda
    lens = torch.cat([torch.full((1_300_000,), 64, device="cuda"), torch.full((60_000,), 8192, device="cuda")])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    times = []
    for order in (torch.arange(lens.numel(), device="cuda"), torch.randperm(lens.numel(), device="cuda", generator=gen)):
        off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(lens[order], 0, out=off[1:])
        arena = torch.empty(int(off[-1]) + 16, dtype=torch.uint8, device="cuda")
        arena.random_(0, 256, generator=gen)
        dS = ag.DeviceRelation(arena, off)
        dR = ag.DeviceRelation(arena, off[:1001])
        ws = ag.alloc_ws(ag.join_prefix_ws_bytes(dR.n, dS.n))
        pairs = torch.empty(2 * 2000, dtype=torch.int32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        best = float("inf")
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            ag.join_prefix_into(dR, dS, 1 << 20, ws, pairs, count, sync=False)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        assert int(count) == 1000
        times.append(best)
    assert times[0] < 1.8 * times[1], times
