"""Edges of the kernels' tiles and of the rules that choose among them, against the CPU oracle through the C ABI."""
import numpy as np
import pytest
import torch

import synth
from ckv_testlib import assert_close, gpu_attend, make_session, oracle_attend, to_dev
from oracle import ckv_oracle as O
from test_route import _bf16, _check, _gpu_route

pytestmark = pytest.mark.gpu


def _workload(mode="softmax", dtype="bf16", head=(30, 2), groups=2, pool=500, users=4, hist=(1, 300), queries=5,
              zipf=1.1, seed=7):
    return synth.Workload("edge", groups, head[0], head[1], pool, users, hist, queries, mode, dtype, zipf, 1 / 32,
                          1 / 32, seed)


def _attend_matches(w, d, want_kernel=None, scale=0.0, **options):
    s = make_session(w, d, scale=scale, **options)
    got = gpu_attend(w, d, session=s)
    kernel, split = s.stat("kernel"), s.stat("split_items")
    assert s.stat("device_errors") == 0
    s.close()
    if want_kernel is not None:
        assert kernel == want_kernel
    assert_close(got, oracle_attend(w, d, scale=scale if scale else None), w.dtype, repr(w))
    return split


@pytest.mark.parametrize("users", [1, 224, 225])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_request_list_as_kernel_argument_and_as_table(users, dtype):
    """Up to 224 requests travel as a kernel argument, and so does the table of a put of as many users."""
    w = _workload(dtype=dtype, users=users, hist=(1, 70), queries=3)
    _attend_matches(w, synth.generate(w), want_kernel=1 if dtype == "f32" else 2)


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("head", [(30, 2), (60, 4)], ids=["d32", "d64"])
@pytest.mark.parametrize("length", [1, 31, 33, 64, 65, 129, 512, 1025, 4097])
def test_warps_sharing_one_unit(mode, head, length):
    """One user: 1 to 32 warps (in up to eight blocks of a cluster) share a unit and merge their results."""
    w = _workload(mode=mode, head=head, users=1, hist=(length, length), queries=17)
    _attend_matches(w, synth.generate(w), want_kernel=2)


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("head,queries", [((31, 1), 17), ((31, 1), 32), ((31, 1), 33), ((31, 1), 47), ((60, 4), 17), ((60, 4), 40)])
def test_several_query_tiles_per_warp(mode, head, queries):
    """Enough work for every resident warp: a warp holds 32 or 48 queries (32-wide heads) or 32 (64-wide)."""
    w = _workload(mode=mode, head=head, groups=4, users=450, hist=(400, 430), queries=queries)
    d = synth.generate(w)
    sel = np.arange(0, w.n_users, 37)
    s = make_session(w, d, kernel=2)
    got = gpu_attend(w, d, session=s)
    s.close()
    rows = np.concatenate([np.arange(d["q_off"][u], d["q_off"][u + 1]) for u in sel])
    assert_close(got[rows], oracle_attend(w, d, sel=sel), "bf16", f"{head} {queries}")


@pytest.mark.parametrize("dtype,length", [("f32", 1), ("f32", 65), ("f32", 1000), ("f32", 4097), ("bf16", 4097)])
@pytest.mark.parametrize("queries", [1, 5])
def test_wide_blocks_of_the_cuda_core_kernel(dtype, length, queries):
    """Fewer blocks than SMs: 16 (8 with several queries) warps on one history, beyond 4096 positions chunks."""
    w = _workload(dtype=dtype, users=2, hist=(length, length), queries=queries)
    split = _attend_matches(w, synth.generate(w), want_kernel=1, kernel=1)
    assert (split > 0) == (length > 4096)


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("head", [(14, 2), (30, 2), (60, 4), (120, 8)], ids=["d16", "d32", "d64", "d128"])
@pytest.mark.parametrize("users,hist,queries", [(149, (17, 130), 1), (80, (17, 700), 9), (230, (63, 65), 4), (20, (17, 2500), 3)])
def test_cuda_core_kernel_between_one_block_per_sm_and_many(mode, head, users, hist, queries):
    """Wide blocks beyond one per SM, chunks from 64 positions on and whole histories, as the estimate chooses."""
    w = _workload(mode=mode, dtype="f32", head=head, users=users, hist=hist, queries=queries)
    _attend_matches(w, synth.generate(w), want_kernel=1)


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("head", [(14, 2), (30, 2), (60, 4), (120, 8)], ids=["d16", "d32", "d64", "d128"])
@pytest.mark.parametrize("chunks", [2, 8, 9, 40])
def test_merge_of_chunks(mode, head, chunks):
    """The merge kernel requests eight chunks at a time."""
    w = _workload(mode=mode, head=head, users=2, hist=(64 * chunks - 5, 64 * chunks - 5), queries=9)
    assert _attend_matches(w, synth.generate(w), split_len=64) > 0


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("queries", [1, 127, 128, 129])
@pytest.mark.parametrize("length", [1, 63, 64, 65, 127, 449, 513])
def test_tcgen05_kernel_tile_edges(mode, queries, length):
    """Tiles of 64 positions and 128 queries; a ring of seven tiles."""
    w = _workload(mode=mode, head=(28, 4), groups=3, users=3, hist=(length, length), queries=queries)
    _attend_matches(w, synth.generate(w), want_kernel=3, kernel=3)


@pytest.mark.parametrize("queries,hist", [(47, (500, 500)), (48, (60, 60)), (96, (1500, 1500)), (97, (1500, 1500)),
                                          (200, (1, 4096)), (60, (4096, 9000))])
def test_short_lists_of_many_queries(queries, hist):
    """From 48 queries on: warp-level kernel, tcgen05 kernel, or that in chunks, as the list's size decides."""
    w = _workload(users=3, hist=hist, queries=queries, groups=4)
    _attend_matches(w, synth.generate(w))


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("head", [(30, 2), (60, 4)], ids=["d32", "d64"])
@pytest.mark.parametrize("pool", [1, 33, 9000, 9500, 19000, 19600, 28000])
def test_factorisation_table_sizes(mode, head, pool):
    """Two CTAs per SM, two table buffers, or one, as the pool's size leaves shared memory."""
    w = _workload(mode=mode, head=head, pool=pool, users=5, hist=(1, 3000), queries=1, zipf=None)
    _attend_matches(w, synth.generate(w), want_kernel=4, kernel=4)


@pytest.mark.parametrize("scale", [2e-3, 1.0, 400.0])
@pytest.mark.parametrize("pool,zipf", [(4, None), (3000, 1.6)])
def test_factorisation_of_large_scores_and_crowded_entries(scale, pool, zipf):
    """Weights are first taken relative to 2^0 and again if the top score is far from it; many positions of one entry."""
    w = _workload(head=(60, 4), pool=pool, users=6, hist=(200, 2500), queries=1, zipf=zipf)
    d = synth.generate(w)
    # (histories of few distinct rows: at the largest scale one position takes all the weight)
    _attend_matches(w, d, want_kernel=4, scale=scale, kernel=4)


@pytest.mark.parametrize("n_new", [1, 12, 13, 40])
def test_append_inside_and_beyond_the_padding(n_new):
    """A history of 20 has room for 12 more positions in place; a refused append leaves everything as it was."""
    import paper_2601_19178_b200 as ckv
    w = _workload(users=2, hist=(20 + n_new, 20 + n_new), queries=4, pool=64)
    d = synth.generate(w)
    L = 20 + n_new
    part = dict(d, hist_off=np.array([0, 20, 20 + L], dtype=np.int64))
    keep = np.r_[0:20, L:2 * L]
    for k in ("idx_K", "idx_V", "user_K", "user_V"):
        part[k] = d[k][keep]
    s = make_session(w, part)
    tail = lambda k, t: to_dev(np.ascontiguousarray(d[k][20:L]), t)
    new = [tail("idx_K", "i"), tail("idx_V", "i"), tail("user_K", "bf16"), tail("user_V", "bf16")]
    before = gpu_attend(w, d, session=s)
    bad = new[1].clone()
    bad[-1, -1] = 64
    with pytest.raises(ckv.CkvError) as e:
        s.cache_append(int(d["users"][0]), new[0], bad, new[2], new[3])
    assert e.value.status == ckv.CKV_ERR_INDEX_RANGE
    assert np.array_equal(gpu_attend(w, d, session=s), before)
    s.cache_append(int(d["users"][0]), *new)
    got = gpu_attend(w, d, session=s)
    s.close()
    assert_close(got, oracle_attend(w, d), "bf16", "appended")


@pytest.mark.parametrize("d_in", [32, 64, 128])
@pytest.mark.parametrize("n,m", [(1, 1), (1, 127), (128, 129), (129, 1000), (256, 128), (257, 3001), (3, 16384)])
def test_router_block_edges(d_in, n, m):
    """Blocks of 256 positions, tiles of 128 entries, entries shared by up to eight CTAs for few positions."""
    rng = np.random.default_rng(n * 7 + m)
    x, W = _bf16(rng.standard_normal((n, d_in))), _bf16(rng.standard_normal((3, m, d_in)) / np.sqrt(d_in))
    _check(x, W, None, f"{n} {m} {d_in}", 2)
    _check(x, W, rng.standard_normal((3, m)).astype(np.float32), f"{n} {m} {d_in} bias", 2)


def test_router_bias_keeps_its_32_bits():
    """The bias enters as three bf16 parts: entries that differ in its last bit only are told apart."""
    m, d_in = 300, 64
    bias = np.full((1, m), np.float32(1.2345678), dtype=np.float32)
    bias[0, 217] = np.nextafter(bias[0, 0], np.float32(2), dtype=np.float32)
    x, W = _bf16(np.zeros((5, d_in))), _bf16(np.zeros((1, m, d_in)))
    assert (_gpu_route(x, W, bias, 2) == 217).all()


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("hist,users", [((48, 52), 1), ((17, 300), 5), ((129, 129), 9), ((700, 700), 2)])
def test_causal_self_attention_of_few_users(mode, hist, users):
    """As many queries as positions, each seeing those up to its own: the warp-level kernel, whatever the number."""
    w = _workload(mode=mode, users=users, hist=hist, queries=1)
    d = synth.generate(w)
    lens = np.diff(d["hist_off"])
    vis = np.concatenate([np.arange(1, n + 1) for n in lens]).astype(np.int32)
    d["q_off"] = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    rng = np.random.default_rng(3)
    d["queries"] = synth.f32_to_bf16_bits(rng.standard_normal((int(lens.sum()), w.n_groups, w.head_dim)).astype(np.float32))
    s = make_session(w, d)
    out = s.attend_visible(d["users"], d["q_off"], vis, to_dev(d["queries"], "bf16"))
    got = out.float().cpu().numpy().astype(np.float64)
    assert s.stat("kernel") == 2 and s.stat("device_errors") == 0
    s.close()
    want = O.attend_variants("bf16", mode, w.default_scale, w.head_dim, d["pool_K"], d["pool_V"], d["hist_off"], d["idx_K"],
                             d["idx_V"], d["user_K"], d["user_V"], d["q_off"], d["queries"], vis=vis)
    # (a SiLU row that sees a few positions is a sum of a few terms: its small values are compared with the largest of all)
    if mode == "softmax":
        assert_close(got, want, "bf16", f"{hist} {users}")
    else:
        assert np.abs(got - want).max() <= 1e-2 * np.abs(want).max()


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("queries", [1, 31, 33, 64, 65, 96, 97, 129, 161, 225])
def test_tcgen05_kernel_with_warps_without_a_row(mode, queries):
    """Blocks of 1 to 128 query rows, several units per worker (rows turn by 32 from unit to unit), histories that end in
    the first or the second half of a tile."""
    w = _workload(mode=mode, groups=8, users=150, hist=(17, 200), queries=queries)
    _attend_matches(w, synth.generate(w), want_kernel=3, kernel=3)


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("queries", [40, 97, 260])
def test_tcgen05_kernel_rows_that_see_parts_of_a_tile(mode, queries):
    """Visible lengths around the 32-position chunks of a tile, whole warps and single rows that see nothing of one."""
    w = _workload(mode=mode, groups=4, users=60, hist=(60, 300), queries=queries)
    d = synth.generate(w)
    rng = np.random.default_rng(queries)
    lens = np.diff(d["hist_off"])
    vis = np.concatenate([np.clip(32 * rng.integers(0, 11, queries) + rng.integers(-1, 2, queries), 0, L) if u % 2 else
                          np.full(queries, min(32 * (u % 9), L)) for u, L in enumerate(lens)]).astype(np.int32)
    vis[vis == 1] = 0
    s = make_session(w, d, kernel=3)
    out = s.attend_visible(d["users"], d["q_off"], torch.from_numpy(vis).cuda(), to_dev(d["queries"], w.dtype))
    torch.cuda.synchronize()
    assert s.stat("kernel") == 3 and s.stat("device_errors") == 0
    s.close()
    want = O.attend_variants(w.dtype, w.mode, w.default_scale, w.head_dim, d["pool_K"], d["pool_V"], d["hist_off"], d["idx_K"],
                             d["idx_V"], d["user_K"], d["user_V"], d["q_off"], d["queries"], vis=vis)
    assert_close(out.float().cpu().numpy().astype(np.float64), want, "bf16", f"{mode} {queries}")


@pytest.mark.parametrize("users", [1, 900])
@pytest.mark.parametrize("head,queries", [((30, 2), 7), ((30, 2), 16), ((30, 2), 33), ((60, 4), 5), ((60, 4), 20)])
@pytest.mark.parametrize("ramp", [(-60, 60), (60, -60), (0, 95)])
def test_warp_level_kernel_reference_far_from_later_scores(users, head, queries, ramp):
    """Scores that climb or fall by 130 to 170 octaves along a history: a row's reference, the maximum of its first tile, is left
    and moved, or stays far above everything behind it.  One user: warps share a unit and merge references apart."""
    w = _workload(head=head, users=users, hist=(200, 400), queries=queries)
    d = synth.generate(w)
    for a, b in zip(d["hist_off"][:-1], d["hist_off"][1:]):
        d["user_K"][a:b, :, 0] = synth.f32_to_bf16_bits(np.linspace(*ramp, b - a, dtype=np.float32))[:, None]
    d["queries"][:, :, 0] = synth.f32_to_bf16_bits(np.full(d["queries"].shape[:2], 1.0, np.float32))
    sel = np.arange(0, users, 90)
    s = make_session(w, d, scale=1.0, kernel=2)
    got = gpu_attend(w, d, session=s)
    s.close()
    rows = np.concatenate([np.arange(d["q_off"][u], d["q_off"][u + 1]) for u in sel])
    assert_close(got[rows], oracle_attend(w, d, scale=1.0, sel=sel), "bf16", f"{users} {head} {queries} {ramp}")


@pytest.mark.parametrize("mode", ["softmax", "silu_over_l"])
@pytest.mark.parametrize("users,hist,queries,groups,pool", [(220, (1000, 1000), 3, 2, 500), (700, (1, 300), 16, 3, 500),
                                                            (700, (1, 300), 20, 3, 500), (225, (31, 65), 1, 9, 66000)])
def test_more_resident_warps_at_64_wide_heads(mode, users, hist, queries, groups, pool):
    """Lists that fill the SMs run with rings of two slots and twelve warps per SM: warps that share a unit and whole units, 16-
    and 32-bit indices, histories from one position on."""
    w = _workload(mode=mode, head=(60, 4), groups=groups, users=users, hist=hist, queries=queries, pool=pool)
    if mode != "softmax":
        w = synth.scaled(w, hist_len=(max(hist[0], 17), hist[1]))
    d = synth.generate(w)
    sel = np.arange(0, users, 23)
    s = make_session(w, d, kernel=2)
    got = gpu_attend(w, d, session=s)
    s.close()
    rows = np.concatenate([np.arange(d["q_off"][u], d["q_off"][u + 1]) for u in sel])
    assert_close(got[rows], oracle_attend(w, d, sel=sel), "bf16", f"{users} {hist} {queries}")


@pytest.mark.parametrize("queries", [5, 24, 47])
def test_short_lists_under_stream_capture(queries):
    """A list that travels as a kernel argument is captured as it is: replays do not depend on plans of other lists."""
    w = _workload(groups=8, users=200, hist=(100, 900), queries=queries)
    d = synth.generate(w)
    s = make_session(w, d)
    q = to_dev(d["queries"], w.dtype)
    want = s.attend(d["users"], d["q_off"], q).clone()
    out = torch.zeros_like(want)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        s.attend(d["users"], d["q_off"], q, out)
    torch.cuda.current_stream().wait_stream(stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.attend(d["users"], d["q_off"], q, out)
    for k in range(6):  # other lists, planned ones
        users = np.concatenate([np.roll(d["users"], k), d["users"][:30]])
        q_off = (np.arange(len(users) + 1) * queries).astype(np.int32)
        s.attend(users, q_off, torch.cat([q, q[:30 * queries]]))
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del graph
    s.close()


_WIDE_LISTS = [(2, head, users, queries) for head, queries in (((30, 2), 7), ((30, 2), 33), ((60, 4), 16), ((60, 4), 20))
               for users in (1, 900)] + [(3, (30, 2), users, queries) for queries in (20, 120) for users in (1, 300)]


@pytest.mark.parametrize("kernel,head,users,queries", _WIDE_LISTS)
@pytest.mark.parametrize("ramp", [(-60, 60), (60, -60), (0, 20)])
def test_values_near_the_largest_behind_scores_above_the_first(kernel, head, users, queries, ramp):
    """Values of 2^112 and scores that climb by up to 170 octaves along a history: weights and sums stay in fp32's range, as they
    do with weights relative to the running maximum (at most 400 of them, each at most one: 2^121)."""
    w = _workload(head=head, users=users, hist=(200, 400), queries=queries)
    d = synth.generate(w)
    for a, b in zip(d["hist_off"][:-1], d["hist_off"][1:]):
        d["user_K"][a:b, :, 0] = synth.f32_to_bf16_bits(np.linspace(*ramp, b - a, dtype=np.float32))[:, None]
    d["queries"][:, :, 0] = synth.f32_to_bf16_bits(np.full(d["queries"].shape[:2], 1.0, np.float32))
    sel = np.arange(0, users, 90)
    want = oracle_attend(w, d, scale=1.0, sel=sel)
    for k in ("pool_V", "user_V"):  # times a power of two: exact
        d[k] = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(d[k]) * np.float32(2.0 ** 112))
    s = make_session(w, d, scale=1.0, kernel=kernel)
    got = gpu_attend(w, d, session=s)
    assert s.stat("device_errors") == 0
    s.close()
    rows = np.concatenate([np.arange(d["q_off"][u], d["q_off"][u + 1]) for u in sel])
    assert_close(got[rows] * 2.0 ** -112, want, "bf16", f"{kernel} {users} {head} {queries} {ramp}")


@pytest.mark.parametrize("kernel,head,users,queries", _WIDE_LISTS)
@pytest.mark.parametrize("what", ["key -inf", "key +inf", "key nan", "value +inf", "value nan"])
def test_infinities_behind_a_first_tile(kernel, head, users, queries, what):
    """One position behind the first 64 of every other user: a key of -inf takes no weight, +inf or none at all leave no number in the
    row, a value shows in its own column alone."""
    w = _workload(head=head, users=users, hist=(200, 400), queries=queries)
    d = synth.generate(w)
    side, x = what.split()
    bits = {"-inf": 0xff80, "+inf": 0x7f80, "nan": 0x7fc0}[x]
    hit = np.arange(0, users, 2)
    for u in hit:
        d["user_K" if side == "key" else "user_V"][d["hist_off"][u] + 70 + u % 100, :, 1] = bits
    d["queries"][:, :, 1] = synth.f32_to_bf16_bits(np.full(d["queries"].shape[:2], 1.0, np.float32))
    sel = np.unique(np.concatenate([np.arange(0, users, 90), np.arange(0, users, 91)]))
    clean = {k: v.copy() for k, v in d.items()}
    for u in hit:  # the oracle's arithmetic: what such a position does to the others is known
        p = d["hist_off"][u] + 70 + u % 100
        if side == "key":
            clean["user_K"][p, :, 1] = synth.f32_to_bf16_bits(np.float32(-1e30))
        else:
            clean["user_V"][p, :, 1] = 0
    want = oracle_attend(w, clean, scale=1.0, sel=sel)
    row = 0
    for u in sel:
        n = d["q_off"][u + 1] - d["q_off"][u]
        if u % 2 == 0 and what != "key -inf":
            if side == "key": want[row:row + n] = np.nan
            else: want[row:row + n, :, 1] = np.inf if x == "+inf" else np.nan
        row += n
    s = make_session(w, d, scale=1.0, kernel=kernel)
    got = gpu_attend(w, d, session=s)
    assert s.stat("device_errors") == 0
    s.close()
    got = got[np.concatenate([np.arange(d["q_off"][u], d["q_off"][u + 1]) for u in sel])]
    odd = ~np.isfinite(want)
    assert np.array_equal(got[odd], want[odd], equal_nan=True)
    assert_close(np.where(odd, 0, got), np.where(odd, 0, want), "bf16", f"{kernel} {users} {head} {queries} {what}")


@pytest.mark.parametrize("queries", [40, 97])
def test_reference_moves_beside_rows_that_see_nothing(queries):
    """Scores that climb along a history while rows of the same warp see nothing, the first tile only, or all of it."""
    w = _workload(users=9, hist=(150, 400), queries=queries)
    d = synth.generate(w)
    for a, b in zip(d["hist_off"][:-1], d["hist_off"][1:]):
        d["user_K"][a:b, :, 0] = synth.f32_to_bf16_bits(np.linspace(0, 90, b - a, dtype=np.float32))[:, None]
    d["queries"][:, :, 0] = synth.f32_to_bf16_bits(np.full(d["queries"].shape[:2], 1.0, np.float32))
    lens = np.diff(d["hist_off"])
    vis = np.concatenate([np.where(np.arange(queries) % 3 == 0, 0, np.where(np.arange(queries) % 3 == 1, 40, L)) for L in lens]).astype(np.int32)
    want = O.attend_variants(w.dtype, w.mode, 1.0, w.head_dim, d["pool_K"], d["pool_V"], d["hist_off"], d["idx_K"],
                             d["idx_V"], d["user_K"], d["user_V"], d["q_off"], d["queries"], vis=vis)
    for kernel in (2, 3):
        s = make_session(w, d, scale=1.0, kernel=kernel)
        out = s.attend_visible(d["users"], d["q_off"], torch.from_numpy(vis).cuda(), to_dev(d["queries"], w.dtype))
        torch.cuda.synchronize()
        assert s.stat("kernel") == kernel and s.stat("device_errors") == 0
        s.close()
        assert_close(out.float().cpu().numpy().astype(np.float64), want, "bf16", f"{kernel} {queries}")
