"""Windows of keys that are all short are not sorted by length: windows on either side
of that line within one relation, the line crossed by single keys, every start
within 32 bytes, for each signature; and the time that empty keys take."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pattern", ["short", "line", "one_long", "windows", "empty_and_long"])
@pytest.mark.parametrize("n", [33, 255, 256, 257, 5000, 100_000, 700_000])
def test_either_side(cuda, pattern, n):
    ag = cuda
    rng = np.random.default_rng(n)
    i = np.arange(n)
    lens = {"short": rng.integers(0, 65, n), "line": rng.integers(60, 100, n),
            "one_long": np.where(i % 256 == 77, 700, rng.integers(0, 40, n)),
            "windows": np.where(i // 256 % 2, rng.integers(0, 40, n), rng.integers(0, 300, n)),
            "empty_and_long": np.where(rng.random(n) < 0.001, 400, 0)}[pattern]
    off = np.zeros(n + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    arena = rng.integers(0, 256, (int(off[-1]) + 15) // 16 * 16 + 16, dtype=np.uint8)
    D = ag.DeviceRelation.from_host(arena, off)
    want = oracle.sig_batch(arena, off, nthreads=8)
    assert np.array_equal(ag.sig_compute(D).cpu().numpy().view(np.uint64), want)
    assert np.array_equal(ag.sig_compute(D, n_components=2).cpu().numpy().view(np.uint64), want & np.uint64(0xFFFFFFFF))
    assert np.array_equal(ag.sig_compute_gf8(D).cpu().numpy().view(np.uint64), oracle.sig8_batch(arena, off, nthreads=8))


def test_empty_keys_cost_no_sort(cuda):
    """Two components of 4M empty keys against 4M keys of 32-96 bytes, which are sorted."""
    ag = cuda
    n, times = 4_000_000, []
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    for lens in (torch.zeros(n, dtype=torch.int64, device="cuda"), torch.randint(32, 97, (n,), device="cuda", generator=gen)):
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(lens, 0, out=off[1:])
        rel = ag.DeviceRelation(torch.randint(0, 256, (int(off[-1]) // 16 * 16 + 32,), dtype=torch.uint8, device="cuda"), off)
        best = float("inf")
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                ag.sig_compute(rel, out, n_components=2)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[0] < 0.76 * times[1], times
