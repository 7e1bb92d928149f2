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
