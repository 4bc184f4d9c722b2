"""Calls from several threads at once."""
import threading

import numpy as np
import pytest
import torch

import paper_2601_19178_b200 as ckv
from ckv_testlib import random_session

pytestmark = pytest.mark.gpu


def _together(n, work):
    """work(k) in n threads that start at once, each on a stream of its own."""
    start, failed = threading.Barrier(n), []

    def run(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait(60)
                work(k)
        except Exception as e:  # noqa: BLE001
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=run, args=(k,)) for k in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not failed and not any(t.is_alive() for t in threads)


@pytest.mark.parametrize("threads", [4, 70])  # the router's calls share 64 pairs of words that a kernel reports through
def test_router_calls_from_several_threads(threads):
    n, G, d, m = 200, 2, 64, 1024
    g = torch.Generator(device="cuda").manual_seed(3)
    W = torch.randn((G, m, d), generator=g, device="cuda").bfloat16()
    x = torch.randn((threads, n, d), generator=g, device="cuda").bfloat16()
    want = torch.empty((threads, n, G), dtype=torch.int32, device="cuda")
    for k in range(threads):
        ckv.ckv_route(0, n, G, d, m, x[k], W, None, want[k])
    got = torch.full((threads, 10, n, G), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def work(k):
        for i in range(10):
            ckv.ckv_route(0, n, G, d, m, x[k], W, None, got[k, i])

    _together(threads, work)
    torch.cuda.synchronize()
    assert torch.equal(got, want[:, None].expand_as(got))


def test_contexts_of_several_threads():
    """Each thread has a context of its own; what their kernels report goes through words of one block."""
    n = 12
    made = [random_session(torch.bfloat16, 6, 50 + k, seed=k) for k in range(n)]
    q_off = np.arange(7, dtype=np.int32) * 4
    queries = [rnd(24, 2, 32) for _, _, rnd in made]
    new = [[torch.full((3, 2), k + i, dtype=torch.int32, device="cuda") for i in range(2)] + [rnd(3, 2, 2), rnd(3, 2, 2)]
           for k, (_, _, rnd) in enumerate(made)]
    bad = torch.full((3, 2), 300, dtype=torch.int32, device="cuda")  # as many entries as the pool has
    outs = [None] * n
    torch.cuda.synchronize()

    def work(k):
        s, ids, _ = made[k]
        for r in range(20):
            if k % 3 == 2:  # a refused append in one context is not seen by another
                with pytest.raises(ckv.CkvError) as e:
                    s.cache_append(int(ids[r % 6]), bad, *new[k][1:])
                assert e.value.status == ckv.CKV_ERR_INDEX_RANGE
            s.cache_append(int(ids[r % 6]), *new[k])
        outs[k] = s.attend(ids, q_off, queries[k])
        torch.cuda.current_stream().synchronize()

    _together(n, work)
    for k in range(n):
        s, ids, rnd = random_session(torch.bfloat16, 6, 50 + k, seed=k)
        for r in range(20):
            s.cache_append(int(ids[r % 6]), *new[k])
        assert torch.equal(s.attend(ids, q_off, queries[k]), outs[k])
        s.close()
        made[k][0].close()
