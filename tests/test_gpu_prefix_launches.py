"""Cumulative signatures are two launches whatever the keys: the signature kernel over
the keys' blocks, and one kernel for the rest, which may begin while the first still
runs.  Counted in a captured graph; and calls that take the one route or the other
follow each other on a stream, directly and in a replayed graph whose keys' lengths
change."""
import ctypes

import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def relation(ag, lens, gen):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    arena = torch.empty((int(off[-1]) + 15) // 16 * 16 + 16, dtype=torch.uint8, device="cuda")
    return ag.DeviceRelation(arena.random_(0, 256, generator=gen), off)


def call(ag, rel, block, pref, out, stream):
    st = ag.load().as_sig_prefixes(rel.arena.data_ptr(), rel.off.data_ptr(), rel.n, block, pref.data_ptr(),
                                   out.data_ptr(), stream.cuda_stream)
    assert st == ag.AS_OK


@pytest.mark.parametrize("n,length,block", [(1000, 40, 64), (1000, 40, 16), (1000, 900, 16), (1000, 900, 256), (1, 5000, 32)])
def test_two_launches(cuda, n, length, block):
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    rel = relation(ag, torch.full((n,), length, dtype=torch.int64, device="cuda"), gen)
    pref, out = ag.sig_prefixes(rel, block)
    want = out.clone()
    out.fill_(-1)
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, count = ctypes.c_void_p(), ctypes.c_size_t(0)
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 2) == 0
    call(ag, rel, block, pref, out, stream)
    assert cu.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    assert cu.cuGraphDestroy(graph) == 0
    assert count.value == 2
    call(ag, rel, block, pref, out, stream)
    stream.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("block", [16, 64, 256])
def test_routes_follow_each_other(cuda, block):
    """Both routes, many keys and few, into one buffer, each result read by the next kernel of the stream."""
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(block)
    rels, want = [], []
    for n, lo, hi in ((30_000, 10, 60), (30_000, 300, 900), (40, 1, 20), (40, 2000, 9000), (200_000, 1, 30)):
        rel = relation(ag, torch.randint(lo, hi, (n,), device="cuda", generator=gen), gen)
        pref, out = ag.sig_prefixes(rel, block)
        assert torch.equal(out[pref[1:] - 1], ag.sig_compute(rel))
        rels.append((rel, pref))
        want.append(out)
    buf = torch.empty(max(w.numel() for w in want), dtype=torch.int64, device="cuda")
    stream = torch.cuda.current_stream()
    got = []
    for turn in range(40):
        i = (turn * 7 + turn // 5) % len(rels)
        rel, pref = rels[i]
        call(ag, rel, block, pref, buf, stream)
        got.append((i, buf[:want[i].numel()].clone()))
        buf.fill_(0)
    for i, g in got:
        assert torch.equal(g, want[i]), i


def test_a_replay_picks_by_the_lengths_it_finds(cuda):
    ag = cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    n, block = 5000, 64
    most = relation(ag, torch.full((n,), 2000, dtype=torch.int64, device="cuda"), gen)
    off = most.off.clone()
    rel = ag.DeviceRelation(most.arena, off)
    pref = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    out = torch.empty(n * 40, dtype=torch.int64, device="cuda")
    ag.sig_prefixes(rel, block)                             # the tables are set up before the capture
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(ag, rel, block, pref, out, torch.cuda.current_stream())
    for length in (2000, 20, 700, 0, 129):
        off[1:] = torch.arange(1, n + 1, device="cuda") * length
        p, want = ag.sig_prefixes(rel, block)
        pref.copy_(p)
        out.fill_(-1)
        g.replay()
        assert torch.equal(out[:want.numel()], want), length
        key = rel.arena[7 * length:8 * length].cpu().numpy().tobytes()
        a, b = int(p[7]), int(p[8])
        assert [x & (2 ** 64 - 1) for x in want[a:b].cpu().tolist()] == oracle.sig_prefixes(key, block)
