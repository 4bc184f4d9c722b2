"""Order between calls that are set up ahead of each other."""
import numpy as np
import pytest
import torch

from ckv_testlib import random_session

pytestmark = pytest.mark.gpu

# fp32: CUDA-core kernel; 16 bit: warp-level tensor-core kernel; 225 users: through a plan
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("users,length,queries", [(1, 40, 3), (8, 700, 5), (200, 33, 1), (225, 33, 1)])
def test_calls_whose_queries_are_the_outputs_before(dtype, users, length, queries):
    """A call's blocks are set up while the kernel before it runs.  Six calls in a row, each attending with what the one
    before it wrote, give the bits of six calls that are waited for."""
    s, ids, rnd = random_session(dtype, users, length)
    q_off = np.arange(users + 1, dtype=np.int32) * queries
    for _ in range(10):
        first = rnd(users * queries, 2, 32)
        want = [first]
        for _ in range(6):
            want.append(s.attend(ids, q_off, want[-1]))
            torch.cuda.synchronize()
        assert not any(torch.equal(a, b) for a, b in zip(want, want[1:]))  # (they settle in the end)
        got = [first] + [torch.full_like(first, float("nan")) for _ in range(6)]  # read too early they spread
        torch.cuda.synchronize()
        for a, b in zip(got, got[1:]):
            s.attend(ids, q_off, a, b)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        # two buffers in turn: a call writes what the call before it reads
        a, b = first.clone(), torch.empty_like(first)
        torch.cuda.synchronize()
        for _ in range(3):
            s.attend(ids, q_off, a, b)
            s.attend(ids, q_off, b, a)
        torch.cuda.synchronize()
        assert torch.equal(a, want[6]) and torch.equal(b, want[5])
    s.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("other_stream", [False, True])
def test_puts_and_appends_between_attends(dtype, other_stream):
    """Puts and appends wait for their kernel: an attend behind one finds the new history, in stream order (its blocks are set
    up while the kernel before it runs) and on another stream alike, and finds the bits that it finds after a synchronise."""
    s, ids, rnd = random_session(dtype, 6, 1500)
    t, _, _ = random_session(dtype, 6, 1500)
    q_off = np.arange(7, dtype=np.int32) * 3
    q = rnd(18, 2, 32)
    streams = [torch.cuda.current_stream(), torch.cuda.Stream() if other_stream else torch.cuda.current_stream()]
    rng = np.random.default_rng(1)
    steps = []
    for k in range(40):  # appends in place, appends that move the user, a put of the user anew
        n = int(rng.choice([1, 5, 33, 700]))
        steps.append((int(ids[k % 6]), k % 5 == 4, n, torch.full((n, 2), k, dtype=torch.int32, device="cuda"),
                      torch.full((n, 2), k + 1, dtype=torch.int32, device="cuda"), rnd(n, 2, 2), rnd(n, 2, 2)))
    torch.cuda.synchronize()

    def go(session, wait):
        outs = []
        for user, anew, n, *parts in steps:
            if anew:
                session.cache_put_batch(np.array([user]), np.array([0, n]), *parts)
            else:
                session.cache_append(user, *parts)
            if wait:
                torch.cuda.synchronize()
            with torch.cuda.stream(streams[1]):
                outs.append(session.attend(ids, q_off, q))
                if wait or other_stream:  # (the next call may give the storage of this one's users to others)
                    streams[1].synchronize()
        torch.cuda.synchronize()
        return outs

    want = go(t, True)
    assert not any(torch.equal(a, b) for a, b in zip(want, want[1:]))
    assert all(torch.equal(a, b) for a, b in zip(go(s, False), want))
    s.close()
    t.close()
