"""The byte comparison of candidates that differ: it ends soon after the first
difference, whatever the keys' length, and only where no candidate compared beside it
is still equal.  Rows get signatures of the test's own choice, so that every S row
meets exactly the R row of its number."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def relation(ag, keys, n, width):
    return ag.DeviceRelation.from_host(np.concatenate([keys.ravel(), np.zeros(16, np.uint8)]),
                                       np.arange(n + 1, dtype=np.uint64) * np.uint64(width))


def probe(ag, dR, dS, n):
    sig = torch.arange(n, dtype=torch.int64, device="cuda")
    ws = ag.alloc_ws(ag.join_table_bytes(n))
    table = ag.join_build(dR, ws, sigR=sig)
    pairs = torch.empty(2 * n, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    table.keep = (ws, sig)

    def run(sync=True):
        return ag.join_probe_sigs(table, dS, sig, pairs, count, sync=sync)
    return run, pairs


@pytest.mark.parametrize("width", [1008, 1023, 1024, 1025, 1041, 2047, 2048, 2049, 3072, 4097, 6000])
def test_candidates_side_by_side(cuda, width):
    """Equal keys beside keys that differ at bytes around every multiple of 1 KB."""
    ag = cuda
    rng = np.random.default_rng(width)
    n = 3000
    r = rng.integers(0, 256, (n, width), dtype=np.uint8)
    s = r.copy()
    places = sorted({p for k in range(0, width + 1024, 512) for p in (k - 17, k - 1, k, k + 16) if 0 <= p < width}
                    | {width - 1})
    what = rng.integers(-1, len(places), n)                 # -1: equal
    hit = what >= 0
    s[np.nonzero(hit)[0], np.array(places)[what[hit]]] ^= 1
    run, pairs = probe(ag, relation(ag, r, n, width), relation(ag, s, n, width), n)
    cnt = run()
    got = np.sort(pairs[:2 * cnt].cpu().numpy().reshape(-1, 2), axis=0)
    assert np.array_equal(got[:, 0], np.nonzero(~hit)[0]) and np.array_equal(got[:, 1], got[:, 0])


def test_a_difference_ends_the_comparison(cuda):
    """20k pairs of 32 KB: those that differ in their first byte take a fraction of the
    time of equal ones (they read 1 KB of 32)."""
    ag = cuda
    n, width = 20_000, 32768
    a = torch.randint(0, 256, (n, width), dtype=torch.uint8, device="cuda")
    b = a.clone()
    b[:, 0] ^= 255
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * width
    pad = torch.zeros(16, dtype=torch.uint8, device="cuda")
    dR, dE, dD = (ag.DeviceRelation(torch.cat([x.view(-1), pad]), off) for x in (a, a.clone(), b))
    times = []
    for dS, want in ((dE, n), (dD, 0)):
        run, _ = probe(ag, dR, dS, n)
        assert run() == want
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            run(sync=False)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
    assert times[1] < 0.4 * times[0], times
