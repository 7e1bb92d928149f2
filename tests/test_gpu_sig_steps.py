"""The signature kernel's step loop against the oracle where it can go wrong:
key lengths around a block (32 bytes), a step (128), the unrolled loop (384),
the change of arithmetic (3 blocks) and the windows (31 to 257 keys), groups
whose lengths differ by many steps, and arenas whose first chunk lies on an
odd 16-byte boundary with no readable byte before it or after the last chunk."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 2, 15, 16, 17, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 255, 256, 257, 383, 384, 385, 511, 512,
         513, 767, 768, 769, 1535, 1537]


@pytest.mark.parametrize("first", [0, 1, 15, 16, 17, 31])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 5000])
def test_step_edges(cuda, first, n):
    ag = cuda
    rng = np.random.default_rng(100 * n + first)
    lens = rng.choice(EDGES, n).astype(np.uint64)
    off = np.zeros(n + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    off += np.uint64(first)
    end = (int(off[-1]) + 15) // 16 * 16
    host = rng.integers(0, 256, max(16, end), dtype=np.uint8)
    want = oracle.sig_batch(host, off, nthreads=4)
    want8 = oracle.sig8_batch(host, off, nthreads=4)
    for shift in (0, 16):                                  # the arena at an even and an odd 16-byte boundary
        buf = torch.empty(host.size + shift, dtype=torch.uint8, device="cuda")
        arena = buf[shift:]
        arena.copy_(torch.as_tensor(host))
        R = ag.DeviceRelation(arena, torch.as_tensor(off.view(np.int64)).cuda())
        for shape in range(len(ag.sig_shapes())):
            for nc in (4, 2):
                got = ag.sig_compute(R, n_components=nc, shape=shape).cpu().numpy().view(np.uint64)
                assert np.array_equal(got, want & np.uint64(oracle.component_mask(nc))), (shift, shape, nc)
        assert np.array_equal(ag.sig_compute_gf8(R).cpu().numpy().view(np.uint64), want8), shift


@pytest.mark.parametrize("lo,hi", [(1, 3000), (200, 280), (0, 12)])
def test_ranges_cut_by_work(cuda, lo, hi):
    """From 2^19 keys the warps' ranges are cut by secant steps, or by a search where those do not
    settle (here a long run of short keys before long ones): every key is signed exactly once."""
    ag = cuda
    n = (1 << 19) + 77
    rng = np.random.default_rng(lo + hi)
    lens = rng.integers(lo, hi + 1, n).astype(np.uint64)
    lens[: n // 2] = np.minimum(lens[: n // 2], 3)
    off = np.zeros(n + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    host = rng.integers(0, 256, workloads.padded_size(int(off[-1])), dtype=np.uint8)
    R = ag.DeviceRelation.from_host(host, off)
    out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    got = ag.sig_compute(R, out).cpu().numpy().view(np.uint64)
    assert np.array_equal(got, oracle.sig_batch(host, off, nthreads=8))


@pytest.mark.parametrize("groups,rest", [(1, -1), (1, 0), (1, 1), (2, 31), (3, 0), (6, 17)])
def test_ranges_of_whole_groups(cuda, groups, rest):
    """Below 2^19 keys the warps get whole groups of 32 keys: around one, two, three and six groups per
    warp of each block shape, every key is signed exactly once."""
    ag = cuda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for shape, (warps, _) in enumerate(ag.sig_shapes()):
        n = 32 * sms * warps * groups + rest
        rng = np.random.default_rng(n)
        off = np.zeros(n + 1, np.uint64)
        off[1:] = np.cumsum(rng.integers(0, 70, n).astype(np.uint64))
        host = rng.integers(0, 256, workloads.padded_size(int(off[-1])), dtype=np.uint8)
        R = ag.DeviceRelation.from_host(host, off)
        out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        got = ag.sig_compute(R, out, shape=shape).cpu().numpy().view(np.uint64)
        assert np.array_equal(got, oracle.sig_batch(host, off, nthreads=8)), shape
