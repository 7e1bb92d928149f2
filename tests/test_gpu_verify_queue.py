"""The probe's candidate queue and byte comparison where they can go wrong: every
key is given the same signature, so that each pair of equally long keys is a
candidate and only the comparison decides; lengths around a 16-byte chunk, the
pieces of eight lanes (128, 256 bytes) and of a warp (512, 1024) and the change
between them (2048); copies of an R key, and keys that differ from one in their
first, last or some other byte; groups that overflow the queue."""
import numpy as np
import pytest
import torch

from workloads import relation_from_keys

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 2, 15, 16, 17, 31, 32, 33, 47, 127, 128, 129, 143, 255, 256, 257, 272, 511, 512, 513, 1023, 1024, 1040,
           2047, 2048]
LONG = [2049, 2064, 4096, 5001]
NO_ROW = 0xFFFFFFFF


def relations(lengths, copies, per_s, seed):
    rng = np.random.default_rng(seed)
    r_keys, s_keys = [], []
    for n in lengths:
        base = rng.integers(0, 256, n, dtype=np.uint8)
        r_keys += [base.tobytes()] * copies
        for _ in range(per_s):
            k = base.copy()
            what = rng.integers(0, 5)
            if n and what:                                 # 0: a copy
                k[[0, n - 1, rng.integers(0, n), rng.integers(0, n)][what - 1]] ^= 1 << rng.integers(0, 8)
            s_keys.append(k.tobytes())
    order = rng.permutation(len(s_keys))
    s_keys = [s_keys[i] for i in order]
    return relation_from_keys(r_keys), relation_from_keys(s_keys), r_keys, s_keys


def expected(r_keys, s_keys, mode):
    by = {}
    for i, k in enumerate(r_keys):
        by.setdefault(k, []).append(i)
    pairs = [(r, s) for s, k in enumerate(s_keys) for r in by.get(k, ())]
    hit_s, hit_r = {s for _, s in pairs}, {r for r, _ in pairs}
    lost_s = [(NO_ROW, s) for s in range(len(s_keys)) if s not in hit_s]
    lost_r = [(r, NO_ROW) for r in range(len(r_keys)) if r not in hit_r]
    return sorted({"inner": pairs, "outer_s": pairs + lost_s, "semi": [(NO_ROW, s) for s in hit_s], "anti": lost_s,
                   "outer_r": pairs + lost_r, "semi_r": [(r, NO_ROW) for r in hit_r], "anti_r": lost_r}[mode])


@pytest.mark.parametrize("lengths,copies,per_s", [(LENGTHS, 1, 40), (LENGTHS, 3, 9), (LENGTHS + LONG, 2, 9),
                                                  ([64], 70, 100), ([0], 5, 33), ([300], 1, 1)])
@pytest.mark.parametrize("mode", ["inner", "outer_s", "semi", "anti", "outer_r", "semi_r", "anti_r"])
def test_comparison_decides(cuda, lengths, copies, per_s, mode):
    ag = cuda
    for seed in range(2):
        R, S, r_keys, s_keys = relations(lengths, copies, per_s, seed)
        dR = ag.DeviceRelation.from_host(R.arena, R.off, R.ids if seed else None)
        dS = ag.DeviceRelation.from_host(S.arena, S.off, S.ids if seed else None)
        sig = 0x0123456789ABCDEF
        sR = torch.full((R.n,), sig, dtype=torch.int64, device="cuda")
        sS = torch.full((S.n,), sig, dtype=torch.int64, device="cuda")
        want = expected(r_keys, s_keys, mode)
        ws = ag.alloc_ws(ag.join_table_bytes(R.n))
        table = ag.join_build(dR, ws, sigR=sR)
        pairs = torch.zeros(2 * (len(want) + 1), dtype=torch.int32, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        cnt = ag.join_probe_mode(table, dS, sS, pairs, count, mode=mode)
        got = pairs[:2 * cnt].cpu().numpy().view(np.uint32).reshape(-1, 2)
        assert sorted(map(tuple, got.tolist())) == want


@pytest.mark.parametrize("mode", ["inner", "outer_s", "semi", "anti"])
def test_many_groups_per_warp(cuda, mode):
    """300k S rows of 24 bytes, half of them copies: every warp fills its queue across groups, and
    S rows' records are put out between the pairs."""
    ag = cuda
    rng = np.random.default_rng(5)
    m, n, w = 1000, 300_000, 24
    r = rng.integers(0, 256, (m, w), dtype=np.uint8)
    src = rng.integers(0, m, n)
    s = r[src].copy()
    miss = rng.random(n) < 0.5
    s[miss, 0] ^= 255
    mk = lambda a, k: ag.DeviceRelation.from_host(np.concatenate([a.ravel(), np.zeros(16, np.uint8)]),
                                                  np.arange(k + 1, dtype=np.uint64) * np.uint64(w))
    dR, dS = mk(r, m), mk(s, n)
    ws = ag.alloc_ws(ag.join_table_bytes(m))
    table = ag.join_build(dR, ws)
    pairs = torch.empty(2 * n, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    cnt = ag.join_probe_mode(table, dS, ag.sig_compute(dS), pairs, count, mode=mode)
    got = pairs[:2 * cnt].cpu().numpy().view(np.uint32).reshape(-1, 2).astype(np.int64)
    got = got[np.argsort(got[:, 1], kind="stable")]
    rows = {"inner": ~miss, "semi": ~miss, "anti": miss, "outer_s": np.ones(n, bool)}[mode]
    assert np.array_equal(got[:, 1], np.nonzero(rows)[0])
    want_r = np.where(miss | (mode in ("semi", "anti")), NO_ROW, src)[rows]
    assert np.array_equal(got[:, 0], want_r)


@pytest.mark.parametrize("per_warp,rest", [(1, 1), (4, 0), (4, 33), (5, 5), (9, 31)])
@pytest.mark.parametrize("mode", ["outer_s", "semi", "anti"])
def test_open_groups(cuda, mode, per_warp, rest):
    """S rows' records are put out for a few groups of 32 rows at a time: around those groups, with
    one or several equal R keys (so that the queue also drains, or is left full, between them)."""
    ag = cuda
    rng = np.random.default_rng(10 * per_warp + rest)
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 16
    m, n, w = 400, 32 * warps * per_warp + rest, 8
    r = rng.integers(0, 256, (m, w), dtype=np.uint8)
    r[m // 2:m // 2 + 9] = r[0]                            # ten equal R keys
    src = rng.integers(0, m, n)
    src[n // 3:n // 3 + 64] = 0                            # two groups that overfill the queue
    s = r[src].copy()
    miss = rng.random(n) < 0.6
    miss[n // 3:n // 3 + 64] = False
    s[miss] ^= 255
    mk = lambda a, k: ag.DeviceRelation.from_host(np.concatenate([a.ravel(), np.zeros(16, np.uint8)]),
                                                  np.arange(k + 1, dtype=np.uint64) * np.uint64(w))
    dR, dS = mk(r, m), mk(s, n)
    ws = ag.alloc_ws(ag.join_table_bytes(m))
    table = ag.join_build(dR, ws)
    keys = {}
    for i, k in enumerate(r):
        keys.setdefault(k.tobytes(), []).append(i)
    hits = [keys.get(k.tobytes(), []) for k in s]
    want = {"semi": [(NO_ROW, j) for j in range(n) if hits[j]], "anti": [(NO_ROW, j) for j in range(n) if not hits[j]],
            "outer_s": [(i, j) for j in range(n) for i in (hits[j] or [NO_ROW])]}[mode]
    pairs = torch.empty(2 * (len(want) + 1), dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    cnt = ag.join_probe_mode(table, dS, ag.sig_compute(dS), pairs, count, mode=mode)
    got = pairs[:2 * cnt].cpu().numpy().view(np.uint32).reshape(-1, 2)
    assert sorted(map(tuple, got.tolist())) == sorted(want)
