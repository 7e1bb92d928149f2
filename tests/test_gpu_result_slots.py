"""Calls that wait for their result from many host threads at once: more of them than
there are page-locked result slots (64), each with its own sizes, so that each has a
count of its own to receive."""
import threading

import numpy as np
import pytest
import torch

from workloads import relation_from_keys

pytestmark = pytest.mark.gpu


def test_more_threads_than_slots(cuda):
    ag = cuda
    threads = 96
    rng = np.random.default_rng(3)
    jobs = []
    for t in range(threads):
        m, n = 50 + t, 120 + 3 * t
        r = [bytes(rng.integers(0, 256, 12, dtype=np.uint8)) for _ in range(m)]
        src = rng.integers(-t - 1, m, n)
        s = [r[i] if i >= 0 else bytes(rng.integers(0, 256, 13, dtype=np.uint8)) for i in src]
        R, S = relation_from_keys(r), relation_from_keys(s)
        jobs.append((ag.DeviceRelation.from_host(R.arena, R.off), ag.DeviceRelation.from_host(S.arena, S.off), src))
    ag.join(jobs[0][0], jobs[0][1])
    torch.cuda.synchronize()
    start, failed = threading.Barrier(threads), []

    def work(t):
        try:
            R, S, src = jobs[t]
            want = sorted((int(i), j) for j, i in enumerate(src) if i >= 0)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for turn in range(3):
                    start.wait(timeout=60)
                    torch.cuda._sleep(4_000_000)            # so that the calls wait side by side
                    if (t + turn) % 3 == 2:
                        got = ag.join_prefix(R, S, 100, stream=stream)
                    elif (t + turn) % 3:
                        got = ag.join_partitioned(R, S, stream=stream)
                    else:
                        got = ag.join(R, S, stream=stream)
                    if sorted(map(tuple, got.cpu().tolist())) != want:
                        failed.append((t, turn))
        except Exception as e:                              # noqa: BLE001 - reported below
            failed.append((t, repr(e)))

    pool = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
    for p in pool:
        p.start()
    for p in pool:
        p.join(timeout=120)
    assert not failed and not any(p.is_alive() for p in pool), failed[:5]
