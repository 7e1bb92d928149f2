"""The probe's groups of 32 S rows per warp, by the warps that it really runs (32 per SM):
whole sets of the groups whose records are put out together, one set and several, and
one group more; and a queue that fills and drains across many groups of a warp."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

WARPS = 32                                                 # per SM
NO_ROW = 0xFFFFFFFF


def keys(ag, rows):
    n, w = rows.shape
    return ag.DeviceRelation.from_host(np.concatenate([rows.ravel(), np.zeros(16, np.uint8)]),
                                       np.arange(n + 1, dtype=np.uint64) * np.uint64(w))


def check(ag, mode, m, n, same, missing, seed):
    """m R keys of which `same` are equal (the first and those from m // 2 on); n S rows with a partner or,
    a share `missing` of them, none; 64 rows in a row look up the equal keys."""
    rng = np.random.default_rng(seed)
    r = np.zeros((m, 8), np.uint8)
    r[:, :4] = np.arange(m, dtype=np.uint32).view(np.uint8).reshape(m, 4)
    r[:, 4:] = rng.integers(0, 255, (m, 4), dtype=np.uint8)
    dup = np.concatenate([[0], np.arange(m // 2, m // 2 + same - 1)]).astype(np.int64)
    r[dup] = r[0]
    src = rng.integers(0, m, n)
    src[n // 3:n // 3 + 64] = 0
    miss = rng.random(n) < missing
    miss[n // 3:n // 3 + 64] = False
    s = r[src]
    s[miss, 7] = 255
    dR, dS = keys(ag, r), keys(ag, s)
    row = np.arange(n, dtype=np.uint64)
    hit = ~miss
    many = hit & np.isin(src, dup)
    one = hit & ~many
    inner = np.concatenate([src[one].astype(np.uint64) << np.uint64(32) | row[one],
                            (dup.astype(np.uint64)[None, :] << np.uint64(32) | row[many][:, None]).ravel()])
    alone = np.uint64(NO_ROW << 32) | row
    want = {"inner": inner, "outer_s": np.concatenate([inner, alone[miss]]), "semi": alone[hit], "anti": alone[miss]}[mode]
    ws = ag.alloc_ws(ag.join_table_bytes(m))
    table = ag.join_build(dR, ws)
    pairs = torch.empty(2 * (want.size + 1), dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    cnt = ag.join_probe_mode(table, dS, ag.sig_compute(dS), pairs, count, mode=mode)
    got = pairs[:2 * cnt].cpu().numpy().view(np.uint32).reshape(-1, 2).astype(np.uint64)
    assert np.array_equal(np.sort(got[:, 0] << np.uint64(32) | got[:, 1]), np.sort(want))


@pytest.mark.parametrize("per_warp,rest", [(1, 0), (3, 31), (4, 0), (4, 1), (5, 0), (8, 0), (8, 33), (9, 0), (13, 7)])
@pytest.mark.parametrize("mode", ["outer_s", "semi", "anti"])
def test_sets_of_open_groups(cuda, mode, per_warp, rest):
    n = 32 * WARPS * torch.cuda.get_device_properties(0).multi_processor_count * per_warp + rest
    check(cuda, mode, 400, n, 10, 0.6, 10 * per_warp + rest)


@pytest.mark.parametrize("mode", ["inner", "outer_s", "semi"])
@pytest.mark.parametrize("same,missing", [(1, 0.0), (1, 0.5), (1, 0.97), (40, 0.9)])
def test_queue_across_many_groups(cuda, mode, same, missing):
    n = 32 * WARPS * torch.cuda.get_device_properties(0).multi_processor_count * 20 + 5
    check(cuda, mode, 5000, n, same, missing, 100 * same + int(100 * missing))
