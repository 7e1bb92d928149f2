"""Byte-symbol signatures of many short keys, which are computed one key per thread,
against the oracle: every length and every start within 16 bytes, empty keys, long
keys among them, both sides of the lines in number and length; and against the
time that the four components over GF(2^16) take."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def check(ag, lens, seed, shift=0):
    rng = np.random.default_rng(seed)
    off = np.zeros(lens.size + 1, np.uint64)
    off[0] = shift
    off[1:] = np.cumsum(lens) + shift
    arena = rng.integers(0, 256, (int(off[-1]) + 15) // 16 * 16 + 16, dtype=np.uint8)
    got = ag.sig_compute_gf8(ag.DeviceRelation.from_host(arena, off)).cpu().numpy().view(np.uint64)
    assert np.array_equal(got, oracle.sig8_batch(arena, off, nthreads=8))


@pytest.mark.parametrize("length", [0, 1, 2, 3, 4, 5, 7, 8, 15, 16, 17, 31, 32, 33, 47, 48, 49, 50, 51, 64])
def test_equal_lengths(cuda, length):
    for n, shift in ((100_001, 0), (150_000, 7)):
        check(cuda, np.full(n, length, np.int64), length + n, shift)


@pytest.mark.parametrize("n", [99_999, 100_000, 100_001, 200_003, 700_000])
@pytest.mark.parametrize("hi", [3, 20, 50, 56])
def test_mixed_lengths(cuda, n, hi):
    check(cuda, np.random.default_rng(n + hi).integers(0, hi + 1, n), n * hi, hi % 16)


def test_long_keys_among_short_ones(cuda):
    rng = np.random.default_rng(1)
    lens = rng.integers(0, 24, 300_000)
    lens[rng.integers(0, lens.size, 40)] = rng.integers(255, 5000, 40)
    lens[-1] = 3001
    lens[0] = 1500
    check(cuda, lens, 2)


def test_short_keys_cost_less_than_double_bytes(cuda):
    ag = cuda
    n, times = 1_000_000, []
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * 16
    rel = ag.DeviceRelation(torch.randint(0, 256, (16 * n + 16,), dtype=torch.uint8, device="cuda"), off)
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    for f in (ag.sig_compute_gf8, ag.sig_compute):
        best = float("inf")
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                f(rel, out)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[0] < 0.75 * times[1], times
