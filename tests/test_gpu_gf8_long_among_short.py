"""Byte-symbol signatures of relations of many short keys with some long ones where
nothing is looked at: pieces of a long key by the warp, at every start and around the
lengths where the pieces change, against the oracle; a key of megabytes among them
takes no longer than alone, and a run of long keys no longer than the same keys
shuffled."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(1000, 1100), (2000, 2100), (8000, 8300), (16370, 16400)])
def test_pieces(cuda, lo, hi):
    ag = cuda
    rng = np.random.default_rng(lo)
    n = 150_000
    lens = rng.integers(0, 9, n)
    at = rng.choice(n, hi - lo, replace=False)             # every length once, none where the relation is looked at
    at = at[np.all([abs(at - n * k // 16) > 64 for k in range(1, 16, 2)], axis=0)]
    lens[at] = np.arange(lo, hi)[:at.size]
    lens[at[1]] = 70_001
    lens[-1] = hi + 1
    off = np.zeros(n + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    arena = rng.integers(0, 256, (int(off[-1]) + 15) // 16 * 16 + 16, dtype=np.uint8)
    got = ag.sig_compute_gf8(ag.DeviceRelation.from_host(arena, off)).cpu().numpy().view(np.uint64)
    assert np.array_equal(got, oracle.sig8_batch(arena, off, nthreads=8))


def timed(ag, lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    rel = ag.DeviceRelation(torch.randint(0, 256, (int(off[-1]) // 16 * 16 + 32,), dtype=torch.uint8, device="cuda"), off)
    out = torch.empty(lens.numel(), dtype=torch.int64, device="cuda")
    best = float("inf")
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        ag.sig_compute_gf8(rel, out)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def full(n, x):
    return torch.full((n,), x, dtype=torch.int64, device="cuda")


def test_one_key_of_megabytes(cuda):
    alone = timed(cuda, full(1, 4 << 20))
    assert timed(cuda, torch.cat([full(700_000, 16), full(1, 4 << 20), full(400_000, 16)])) < 1.3 * alone


def test_a_run_of_long_keys(cuda):
    lens = torch.cat([full(1_000_000, 16), full(30_000, 8192)])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    shuffled = lens[torch.randperm(lens.numel(), device="cuda", generator=gen)]
    assert timed(cuda, lens) < 2.0 * timed(cuda, shuffled)


def test_a_tenth_of_long_keys(cuda):
    """24 bytes and a tenth of 264, of which no long one is near an odd eighth of the relation: not one key per
    thread, which would take three times as long as the two components that share the staged kernel."""
    ag = cuda
    n = 500_000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    long = torch.rand(n, device="cuda", generator=gen) < 0.1
    for k in (1, 3, 5, 7):
        long[n * k // 8 - 64:n * k // 8 + 64] = False
    lens = torch.where(long, 264, 24)
    bytes_ = timed(ag, lens)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    rel = ag.DeviceRelation(torch.randint(0, 256, (int(off[-1]) // 16 * 16 + 32,), dtype=torch.uint8, device="cuda"), off)
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    best = float("inf")
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        ag.sig_compute(rel, out, n_components=2)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    assert bytes_ < 1.6 * best, (bytes_, best)
