"""Cumulative signatures of relations whose items (keys' blocks) differ in length: the
warps take equal shares of the items' bytes.  Every key's last entry is its
signature whatever the order of the lengths, whole keys' entries are the oracle's
where shares meet, and a run of long keys takes no longer than the same keys
shuffled."""
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def relation(ag, lens, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    arena = torch.empty((int(off[-1]) + 15) // 16 * 16 + 16, dtype=torch.uint8, device="cuda")
    return ag.DeviceRelation(arena.random_(0, 256, generator=gen), off)


def lengths(name):
    full = lambda n, x: torch.full((n,), x, dtype=torch.int64, device="cuda")
    return {"short_first": lambda: torch.cat([full(90_000, 40), full(9_000, 6000)]),
            "long_first": lambda: torch.cat([full(9_000, 6001), full(90_000, 39)]),
            "one_giant": lambda: torch.cat([full(70_000, 100), full(1, 30_000_000), full(40_000, 300)]),
            "giant_last": lambda: torch.cat([full(100_000, 129), full(1, 20_000_001)]),
            "empties": lambda: torch.cat([full(80_000, 0), full(20_000, 2000), full(50_000, 0), full(3, 500_000)]),
            "even": lambda: full(160_000, 200)}[name]()


@pytest.mark.parametrize("name", ["short_first", "long_first", "one_giant", "giant_last", "empties", "even"])
@pytest.mark.parametrize("block", [64, 256, 4096, 65536])
def test_every_item_signed(cuda, name, block):
    ag = cuda
    rel = relation(ag, lengths(name), block)
    pref, out = ag.sig_prefixes(rel, block)
    assert torch.equal(pref[1:] - pref[:-1], ((rel.off[1:] - rel.off[:-1] + block - 1) // block).clamp_(min=1))
    assert torch.equal(out[pref[1:] - 1], ag.sig_compute(rel))
    off, host = rel.off.cpu().tolist(), pref.cpu().tolist()
    for i in range(1, rel.n, rel.n // 37):
        key = rel.arena[off[i]:off[i + 1]].cpu().numpy().tobytes()
        if len(key) < 10_000:
            got = [x & (2 ** 64 - 1) for x in out[host[i]:host[i + 1]].cpu().tolist()]
            assert got == oracle.sig_prefixes(key, block), i


def test_order_of_lengths_costs_nothing(cuda):
    """1M keys of 64 bytes and 40k of 8 KB, at blocks of 4 KB and of 1 MB (an item per key)."""
    ag = cuda
    lens = torch.cat([torch.full((1_000_000,), 64, device="cuda"), torch.full((40_000,), 8192, device="cuda")])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    shuffled = lens[torch.randperm(lens.numel(), device="cuda", generator=gen)]
    for block in (4096, 1 << 20):
        times = []
        for x in (lens, shuffled):
            rel = relation(ag, x, 5)
            best = float("inf")
            for _ in range(6):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record()
                ag.sig_prefixes(rel, block)
                e1.record()
                e1.synchronize()
                best = min(best, e0.elapsed_time(e1))
            times.append(best)
        assert times[0] < 1.8 * times[1], (block, times)
