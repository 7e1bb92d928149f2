"""The rule that picks how cumulative signatures are computed looks at the longest of
neighbouring keys: entries on both sides of its lines, in keys' lengths and in their
number, and for relations smaller than what it looks at; and a relation of short keys
with long ones among them takes the way that does not wait for the longest."""
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def relation(ag, lens, gen):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    arena = torch.empty((int(off[-1]) + 15) // 16 * 16 + 16, dtype=torch.uint8, device="cuda")
    return ag.DeviceRelation(arena.random_(0, 256, generator=gen), off)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 33, 63, 65, 20_000, 20_001, 32_767, 32_768, 163_840, 163_841])
@pytest.mark.parametrize("mean", [1, 176, 184, 192, 272, 288])
def test_both_sides_of_the_lines(cuda, n, mean):
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + mean)
    some = torch.randint(0, n, (20,), generator=torch.Generator().manual_seed(n)).tolist()
    for lens in (torch.full((n,), mean, dtype=torch.int64, device="cuda"),
                 torch.randint(0, 2 * mean + 1, (n,), device="cuda", generator=gen)):
        rel = relation(ag, lens, gen)
        off = rel.off.cpu().tolist()
        for block in (16, 32, 64, 256):
            pref, out = ag.sig_prefixes(rel, block)
            assert torch.equal(pref[1:] - pref[:-1], ((lens + block - 1) // block).clamp_(min=1))
            assert torch.equal(out[pref[1:] - 1], ag.sig_compute(rel))
            for i in set(some[:20 if n < 1000 else 3]):
                key = rel.arena[off[i]:off[i + 1]].cpu().numpy().tobytes()
                a, b = int(pref[i]), int(pref[i + 1])
                assert [x & (2 ** 64 - 1) for x in out[a:b].cpu().tolist()] == oracle.sig_prefixes(key, block), (i, block)


def test_long_keys_among_short_ones(cuda):
    """500k keys of 48 bytes, a tenth of them 520 long, against as many equal ones of as many bytes."""
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    n, block = 500_000, 256
    mixed = torch.where(torch.rand(n, device="cuda", generator=gen) < 0.9, 48, 520)
    lib, times = ag.load(), []
    for lens in (mixed, torch.full((n,), int(mixed.sum()) // n, dtype=torch.int64, device="cuda")):
        rel = relation(ag, lens, gen)
        pref, out = ag.sig_prefixes(rel, block)
        stream = torch.cuda.current_stream().cuda_stream
        best = float("inf")
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(5):
                assert lib.as_sig_prefixes(rel.arena.data_ptr(), rel.off.data_ptr(), n, block, pref.data_ptr(),
                                           out.data_ptr(), stream) == 0
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[0] < 2.8 * times[1], times
