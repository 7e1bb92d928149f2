"""Cumulative signatures by blocks (items) against the oracle's definition, on
both sides of the rule that picks the kernels (mean key length): keys of many
blocks (more than a warp scans at once, more than a window holds), empty keys
between them, windows that start and end inside a key, ranges of one item."""
import numpy as np
import pytest

import oracle
from workloads import relation_from_keys

pytestmark = pytest.mark.gpu

RELATIONS = {
    "mixed": [0, 1, 15, 16, 17, 255, 256, 257, 700, 0, 0, 31, 512, 513, 1024, 300] * 20,
    "long": [0, 70_000, 3, 0, 0, 9_000, 256, 40_001, 0],
    "short": list(range(0, 24)) * 30,
    "one": [5000],
    "equal": [512] * 1000,
}


@pytest.mark.parametrize("name", sorted(RELATIONS))
@pytest.mark.parametrize("block", [16, 32, 64, 128, 256, 1024])
def test_blocks_sum_up(cuda, name, block):
    ag = cuda
    rng = np.random.default_rng(block)
    keys = [rng.integers(0, 256, n, dtype=np.uint8).tobytes() for n in RELATIONS[name]]
    rel = relation_from_keys(keys)
    D = ag.DeviceRelation.from_host(rel.arena, rel.off)
    pref, out = ag.sig_prefixes(D, block)
    pref, out = pref.cpu().numpy(), out.cpu().numpy().view(np.uint64)
    sig = oracle.sig_batch(rel.arena, rel.off, nthreads=4)
    assert pref[0] == 0 and np.array_equal(np.diff(pref), [max(1, -(-len(k) // block)) for k in keys])
    assert np.array_equal(out[pref[1:] - 1], sig)              # the last entry is the whole key's
    for i, k in enumerate(keys):
        if len(k) <= 3000 or i == 1:
            assert out[pref[i]:pref[i + 1]].tolist() == oracle.sig_prefixes(k, block), (i, len(k))


@pytest.mark.parametrize("block", [256, 512, 1024])
def test_many_windows_per_warp(cuda, block):
    """More than a million blocks, so that every warp walks several windows, most of which end inside
    a key: each key's last entry is the signature of the whole key."""
    ag = cuda
    rng = np.random.default_rng(block)
    lens = rng.integers(block, 5 * block, 420_000).astype(np.uint64)
    off = np.zeros(lens.size + 1, np.uint64)
    off[1:] = np.cumsum(lens)
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(block)
    arena = torch.empty((int(off[-1]) + 15) // 16 * 16 + 16, dtype=torch.uint8, device="cuda").random_(0, 256, generator=gen)
    D = ag.DeviceRelation(arena, torch.as_tensor(off.view(np.int64)).cuda())
    pref, out = ag.sig_prefixes(D, block)
    assert torch.equal(out[pref[1:] - 1], ag.sig_compute(D))
    some = rng.integers(0, lens.size, 40)
    pref, host = pref.cpu().numpy(), out.cpu().numpy().view(np.uint64)
    for i in some:
        key = arena[int(off[i]):int(off[i + 1])].cpu().numpy().tobytes()
        assert host[pref[i]:pref[i + 1]].tolist() == oracle.sig_prefixes(key, block), i


@pytest.mark.parametrize("block", [32, 80, 256])
def test_blocks_around_the_scan_factors(cuda, block):
    """Block counts around the factors that the scan splits a block's place into (16), the keys that
    one thread sums (32) and the tables' end (512)."""
    ag = cuda
    rng = np.random.default_rng(block)
    counts = [2, 3, 4, 5, 6, 15, 16, 17, 18, 31, 32, 33, 34, 47, 48, 49, 63, 64, 65, 511, 512, 513, 545]
    keys = [rng.integers(0, 256, c * block - int(rng.integers(0, block)), dtype=np.uint8).tobytes() for c in counts]
    rel = relation_from_keys(keys)
    D = ag.DeviceRelation.from_host(rel.arena, rel.off)
    pref, out = ag.sig_prefixes(D, block)
    pref, out = pref.cpu().numpy(), out.cpu().numpy().view(np.uint64)
    assert np.array_equal(np.diff(pref), counts)
    for i, k in enumerate(keys):
        assert out[pref[i]:pref[i + 1]].tolist() == oracle.sig_prefixes(k, block), counts[i]


@pytest.mark.parametrize("block", [131056, 131072, 262128])
def test_blocks_whose_factors_wrap(cuda, block):
    """Blocks of nearly, exactly one more than and nearly twice the order of x in symbols."""
    ag = cuda
    rng = np.random.default_rng(block)
    keys = [rng.integers(0, 256, n, dtype=np.uint8).tobytes() for n in (block + 1, 2 * block + 77, 4 * block, 9)]
    rel = relation_from_keys(keys)
    pref, out = ag.sig_prefixes(ag.DeviceRelation.from_host(rel.arena, rel.off), block)
    pref, out = pref.cpu().numpy(), out.cpu().numpy().view(np.uint64)
    want = [k[:(j + 1) * block] for k in keys for j in range(max(1, -(-len(k) // block)))]
    ref = relation_from_keys(want)
    assert np.array_equal(out, oracle.sig_batch(ref.arena, ref.off, nthreads=4))
