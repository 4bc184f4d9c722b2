"""The named barriers by which the tcgen05 router's read-out warps hand an accumulator back (csrc/kernels_route_umma.cu), on the CPU:
every order in which a block's five warps can come, and give up after a wait that ran out."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_19178_b200", "csrc", "kernels_route_umma.cu")
READERS, TILES = 4, 4
RUN, BLOCKED, END = 0, 1, 2


def barrier_of():
    code = open(SOURCE).read()
    expr = re.search(r"int read_barrier\(int acc, int tile\)\s*\{\s*return ([^;]+);", code).group(1)
    # what the roles name: the read-out the tile it has read, the issuing warp the tile before its own
    assert set(re.findall(r"\bacc_(?:arrive|sync)\(([^;]*)\);", code.split("__launch_bounds__", 1)[1])) == {
        "acc, t", "ACCS * blk + h, t - 1"}
    return eval("lambda acc, tile: " + expr)


def stuck(barrier, accs):
    """A state no warp gets out of, or an accumulator written before it was read although nobody gave up; None if there is none.

    Step t of a block is accumulator t % accs of tile t // accs.  A warp is (state, step, still ok); the issuing warp has issued the
    products of `issued` steps, and each barrier has counted some arrivals."""
    steps = TILES * accs
    name = [barrier(t % accs, t // accs) for t in range(steps)]
    ids = sorted(set(name))
    start = (((RUN, 0, True),) * READERS, (RUN, 0, True), 0, (0,) * len(ids))
    seen, todo = {start}, [start]
    while todo:
        state = todo.pop()
        readers, issuer, issued, counts = state
        after = []

        def arrive(readers, issuer, issued, counts, step):
            b = ids.index(name[step])
            counts = list(counts)
            counts[b] += 1
            if counts[b] == READERS + 1:  # all who are blocked there go on
                counts[b] = 0
                readers = tuple((RUN, t + 1, ok) if s == BLOCKED and name[t] == ids[b] else (s, t, ok) for s, t, ok in readers)
                s, t, ok = issuer
                if s == BLOCKED and name[t - accs] == ids[b]:
                    issuer, issued = go_on(t, ok, issued)
            return tuple(sorted(readers)), issuer, issued, tuple(counts)

        def go_on(t, ok, issued):  # the issuing warp behind the barrier of step t - accs
            return ((RUN, t + 1, ok) if t + 1 < steps else (END, 0, ok)), issued + ok

        for i, (s, t, ok) in enumerate(readers):
            if s != RUN:
                continue
            others = readers[:i] + readers[i + 1:]
            for here in ([True, False] if ok and issued > t else [False]):  # a wait that has its tile, or runs out
                last = t + accs >= steps  # (nobody waits for an accumulator's last tile)
                now = (RUN, t + 1, here) if here or last else (BLOCKED, t, False)
                if now[1] == steps:
                    now = (END, 0, here)
                step = (tuple(sorted(others + (now,))), issuer, issued, counts)
                after.append(step if last else arrive(*step, t))
        s, t, ok = issuer
        if s == RUN:
            for here in ([True, False] if ok else [False]):
                if t < accs:
                    now, n = go_on(t, here, issued)
                    after.append((readers, now, n, counts))
                else:
                    after.append(arrive(readers, (BLOCKED, t, here), issued, counts, t - accs))
        if not after and any(w[0] != END for w in readers + (issuer,)):
            return "stuck", state
        for a in after:
            if all(w[2] for w in a[0] + (a[1],)) and any(w[0] == RUN and w[1] < a[2] - accs for w in a[0]):
                return "written before it was read", a
            if a not in seen:
                seen.add(a)
                todo.append(a)
    return None


@pytest.mark.parametrize("accs", [1, 2])
def test_no_order_of_giving_up_leaves_a_warp_behind(accs):
    assert stuck(barrier_of(), accs) is None


@pytest.mark.parametrize("accs", [1, 2])
def test_one_barrier_per_accumulator_would_not_do(accs):
    """A warp that gives up has already arrived for the tile before, and a second time counts for the issuing warp."""
    assert stuck(lambda acc, tile: 1 + acc, accs)[0] == "stuck"


@pytest.mark.parametrize("accumulators", [3, 6])
def test_every_accumulator_has_barriers_of_its_own(accumulators):
    barrier = barrier_of()
    ids = [{barrier(acc, t) for t in range(TILES)} for acc in range(accumulators)]
    assert sum(map(len, ids)) == len(set().union(*ids)) and set().union(*ids) <= set(range(1, 15))  # 0 and 15 are the whole block's
