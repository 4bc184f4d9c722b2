"""The library's host side on the CPU: its object files linked with tests/fake_cudart.cpp instead of the CUDA runtime.
Kernels do not run there; what is tested is what a call does before and between them."""
import ctypes as C
import glob
import importlib.util
import os
import subprocess
import threading
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class Config(C.Structure):
    _fields_ = [(n, C.c_int32) for n in ("n_groups", "head_dim", "dtype", "out_dtype", "mode")] + \
        [("scale", C.c_float), ("device", C.c_int32)]


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


@pytest.fixture(scope="module")
def objects():
    """The library's object files, one per source file."""
    spec = importlib.util.spec_from_file_location("ckv_build", os.path.join(ROOT, "paper_2601_19178_b200", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.build()
    return [os.path.join(mod.OBJ, os.path.basename(f)[:-3] + ".o") for f in sorted(glob.glob(os.path.join(mod.CSRC, "*.cu")))]


@pytest.fixture(scope="module")
def lib(objects, tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libckv_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include", "-o", so,
                    *objects, os.path.join(ROOT, "tests", "fake_cudart.cpp")],
                   check=True)
    lib = C.CDLL(so)
    lib.fake_count.restype = C.c_long
    lib.fake_launched.restype = C.POINTER(C.c_long)
    return lib


def device_block(lib, size):
    p = C.c_void_p()
    assert lib.cudaMalloc(C.byref(p), C.c_size_t(size)) == 0
    return p


def context(lib, G=4, D=32, d_user=1, m=2048):
    """A bf16 softmax context with a pool, and a block that stands for any device input."""
    ctx = C.c_void_p()
    assert lib.ckv_create(C.byref(Config(G, D, 1, 1, 0, 0.0, 0)), C.byref(ctx)) == 0
    block = device_block(lib, G * m * D * 2)
    assert lib.ckv_pool_load(ctx, block, block, m, D - d_user, None) == 0
    return ctx, block


def put(lib, ctx, block, users, lens, d_user=1):
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return lib.ckv_cache_put_batch(ctx, len(users), ptr(users), ptr(off), block, block, block, block, d_user, None)


def test_no_object_file_holds_many_forms_of_the_warp_level_kernel(objects):
    """Its 96 forms in one file took three times as long to compile as all others side by side."""
    per_file = [subprocess.run(["nm", "-C", o], capture_output=True, text=True, check=True).stdout.count("::attend_mma_kernel<")
                for o in objects]
    assert 0 < max(per_file) <= 32


def test_planning_a_list_costs_little_more_than_its_tables(lib):
    """A request list that the context has not seen: at most half as much again as looking its users up and writing and
    copying its tables (1.3 times; sums for the dispatch next to the look-ups, further walks over the list for its estimates
    and a division per request made it 1.6)."""
    n = 65536
    ctx, block = context(lib)
    users = np.arange(n, dtype=np.int64) * 7919 + 3
    assert put(lib, ctx, block, users, np.full(n, 512)) == 0
    q_off = np.arange(n + 1, dtype=np.int32) * 16
    rng = np.random.default_rng(0)
    lists = [rng.permutation(users) for _ in range(9)]  # more than the context keeps plans
    ratio = 1e9
    for _ in range(4):
        plan, floor = [], []
        for u in lists:
            t0 = time.perf_counter()
            assert lib.ckv_attend(ctx, n, ptr(u), ptr(q_off), block, block, None) == 0
            t1 = time.perf_counter()
            assert lib.fake_plan_floor(lib.ckv_user_length, ctx, n, ptr(u), ptr(q_off)) == 0
            t2 = time.perf_counter()
            plan.append(t1 - t0)
            floor.append(t2 - t1)
        ratio = min(ratio, min(plan) / min(floor))
    lib.ckv_destroy(ctx)
    assert ratio < 1.5


def test_contexts_share_one_block_of_mapped_words(lib):
    """Pinned memory is what creating a context spent its time on.  A reset of the device takes the block along."""
    def create(n):
        ctxs = [C.c_void_p() for _ in range(n)]
        for c in ctxs:
            assert lib.ckv_create(C.byref(Config(4, 32, 1, 1, 0, 0.0, 0)), C.byref(c)) == 0
        return ctxs

    def destroy(ctxs):
        for c in ctxs:
            assert lib.ckv_destroy(c) == 0

    destroy(create(2))
    lib.fake_reset()
    for _ in range(3):
        destroy(create(20))
    assert lib.fake_count(b"cudaHostAlloc") + lib.fake_count(b"cudaMallocHost") == 0
    live = create(500)  # no words for two at once: 448 in the block, an allocation for each of the others
    assert lib.fake_count(b"cudaHostAlloc") == 500 - 448
    destroy(live)
    assert lib.fake_count(b"cudaFreeHost") == 500 - 448
    before = create(2)
    lib.fake_device_reset()
    lib.fake_reset()
    after = create(447)
    assert lib.fake_count(b"cudaHostAlloc") == 1
    destroy(before)  # words of the old block: nothing of the new one comes free
    after += create(2)
    assert lib.fake_count(b"cudaHostAlloc") == 2
    destroy(after)


def test_a_threads_first_call_may_need_a_tensor_map(lib):
    """Encoding one is a driver call, which makes no context current by itself as a launch does: the router's calls, and a
    pool loaded again into storage that is there, on a thread that has not used the GPU."""
    G, d, m, n = 2, 64, 1024, 200
    block = device_block(lib, G * m * d * 2)
    status = {}

    def route():
        status["route"] = lib.ckv_route(0, n, G, d, m, block, block, None, block, 0, None)

    ctx, pool = context(lib, G=2, D=64, d_user=4, m=m)

    def load():
        status["load"] = lib.ckv_pool_load(ctx, pool, pool, m, 60, None)

    for f in (route, load):
        t = threading.Thread(target=f)
        t.start()
        t.join()
    assert status == {"route": 0, "load": 0}
    # with its maps the pool can be gathered by TMA
    users = np.arange(300, dtype=np.int64)
    assert put(lib, ctx, block, users, np.full(300, 40), d_user=4) == 0
    assert lib.ckv_set_option(ctx, b"mma_loader", C.c_int64(2)) == 0
    assert lib.ckv_attend(ctx, 300, ptr(users), ptr(np.arange(301, dtype=np.int32)), block, block, None) == 0
    lib.ckv_destroy(ctx)


# 2 users: kept whole (the list travels as a kernel argument).  207 users of one query: wide blocks of 16 warps although there
# are more than SMs.  75 ragged users of up to 16 queries: cut.  500 short histories: blocks enough.
@pytest.mark.parametrize("users,lo,hi,queries,threads,cut", [(2, 1000, 1000, 5, 256, False), (207, 745, 745, 1, 512, False),
                                                             (75, 50, 1000, 16, 128, True), (500, 100, 100, 1, 128, False)])
def test_cuda_core_lists_of_a_few_hundred_blocks(lib, users, lo, hi, queries, threads, cut):
    """Chunks and block size of the CUDA-core kernel (fp32, 2 groups of 32-wide heads, 148 SMs)."""
    ctx = C.c_void_p()
    assert lib.ckv_create(C.byref(Config(2, 32, 0, 0, 0, 0.0, 0)), C.byref(ctx)) == 0
    block = device_block(lib, 2 * 1024 * 32 * 4)
    assert lib.ckv_pool_load(ctx, block, block, 1024, 30, None) == 0
    ids = np.arange(users, dtype=np.int64)
    lens = np.random.default_rng(0).permutation(np.linspace(lo, hi, users).round().astype(np.int64))
    assert put(lib, ctx, block, ids, lens, d_user=2) == 0
    q_off = np.concatenate([[0], np.cumsum(np.arange(users) % queries + 1 if cut else np.full(users, queries))]).astype(np.int32)
    assert lib.ckv_attend(ctx, users, ptr(ids), ptr(q_off), block, block, None) == 0
    launched = np.ctypeslib.as_array(lib.fake_launched(), (6,))
    split = C.c_int64()
    assert lib.ckv_last_stat(ctx, b"split_items", C.byref(split)) == 0
    assert (split.value > 0) == cut
    if not cut:  # (otherwise the last launch is the merge)
        assert launched[3] == threads
    lib.ckv_destroy(ctx)


# (users, positions, queries, kernel family): few and short self-attentions go to the warp-level kernel, many and long ones
# and tails of longer histories to the tcgen05 kernel
@pytest.mark.parametrize("users,length,queries,family", [(7, 556, 556, 2), (1, 50, 50, 2), (1, 1500, 1500, 2), (20, 1500, 1500, 3),
                                                         (64, 300, 300, 3), (8, 500, 60, 2), (3, 1500, 128, 3)])
def test_kernel_of_lists_with_visible_lengths(lib, users, length, queries, family):
    ctx, block = context(lib, G=2, D=32, d_user=2)
    ids = np.arange(users, dtype=np.int64)
    assert put(lib, ctx, block, ids, np.full(users, length), d_user=2) == 0
    q_off = (np.arange(users + 1) * queries).astype(np.int32)
    assert lib.ckv_attend_visible(ctx, users, ptr(ids), ptr(q_off), block, block, block, None) == 0
    kernel = C.c_int64()
    assert lib.ckv_last_stat(ctx, b"kernel", C.byref(kernel)) == 0 and kernel.value == family
    lib.ckv_destroy(ctx)


def test_tma_loader_option_leaves_the_tcgen05_kernel_its_lists(lib):
    """The warp-level kernel's TMA loader takes neither visible lengths nor sides that are not shared: with that option set,
    short lists with either stay with the tcgen05 kernel, which has no such option, instead of being refused."""
    for sides, vis, queries in (((30, 30), True, 500), ((30, 30), True, 60), ((30, 0), False, 60), ((0, 30), False, 60)):
        ctx = C.c_void_p()
        assert lib.ckv_create(C.byref(Config(2, 32, 1, 1, 0, 0.0, 0)), C.byref(ctx)) == 0
        block = device_block(lib, 1 << 20)
        assert lib.ckv_pool_load_sides(ctx, block, block, 1000, *sides, None) == 0
        ids = np.arange(2, dtype=np.int64)
        assert put(lib, ctx, block, ids, np.full(2, 500), d_user=2) == 0
        q_off = (np.arange(3) * queries).astype(np.int32)
        call = [ctx, 2, ptr(ids), ptr(q_off)] + ([block] if vis else []) + [block, block, None]
        attend = lib.ckv_attend_visible if vis else lib.ckv_attend
        kernel = C.c_int64()
        for loader, family in ((1, 2), (2, 3)):
            assert lib.ckv_set_option(ctx, b"mma_loader", C.c_int64(loader)) == 0
            assert attend(*call) == 0
            assert lib.ckv_last_stat(ctx, b"kernel", C.byref(kernel)) == 0 and kernel.value == family
        lib.ckv_destroy(ctx)


def test_a_report_that_does_not_come_is_not_waited_for(lib):
    """Kernels of several rounds of blocks do not report: their calls go to the stream at once, not behind the 40 us that they
    watch for a report (which no kernel writes here, so that calls whose kernel reports take those 40 us)."""
    G, d = 4, 64
    block = device_block(lib, 1 << 20)
    ctx, _ = context(lib, G=G)
    user = np.zeros(1, np.int64)

    def us(call):
        best = 1e9
        for _ in range(20):
            t = time.perf_counter()
            assert call() == 0
            best = min(best, time.perf_counter() - t)
        return best * 1e6

    def route(n, m, variant):
        return us(lambda: lib.ckv_route(0, n, G, d, m, block, block, None, block, variant, None))

    assert route(200, 1024, 0) >= 40 and route(200, 1024, 2) >= 40
    assert route(20000, 64, 2) < 30 and route(1000000, 16384, 0) < 30
    assert route(300000, 8, 0) < 30  # (more blocks than the report's counter could tell apart)
    assert us(lambda: put(lib, ctx, block, user, [1000])) >= 40
    assert us(lambda: put(lib, ctx, block, user, [1100 * 8 * 32])) < 30
    lib.ckv_destroy(ctx)


# (d_in, positions, entries, groups, threads of a block: 256 where the entries are shared by its warps, 512 for the tcgen05 kernel)
@pytest.mark.parametrize("d,n,m,G,threads", [(64, 1, 8, 1, 256), (64, 1072, 8000, 2, 256), (64, 1075, 8000, 2, 512),
                                             (64, 9472, 32, 1, 256), (64, 9473, 32, 1, 512), (32, 2368, 1000, 4, 256),
                                             (32, 2369, 1000, 4, 512), (128, 4736, 16, 2, 256), (128, 4737, 16, 2, 512),
                                             (64, 1000000, 16, 1, 512), (64, 32, 16, 296, 256), (64, 32, 16, 297, 512)])
def test_kernel_of_router_calls(lib, d, n, m, G, threads):
    """The kernel for few positions takes 1.1e9 products and 296 blocks of 32 positions and a group, no more."""
    block = device_block(lib, 1 << 20)
    assert lib.ckv_route(0, n, G, d, m, block, block, None, block, 0, None) == 0
    assert np.ctypeslib.as_array(lib.fake_launched(), (6,))[3] == threads


# (users, positions, queries, groups, twelve warps per SM)
@pytest.mark.parametrize("users,lens,queries,G,dense", [
    (220, (1000, 1000), (3, 3), 2, True), (222, (1000, 1000), (3, 3), 2, True), (223, (1000, 1000), (3, 3), 2, False),
    (199, (17, 1999), (1, 40), 4, True), (6, (3059, 3059), (94, 94), 3, False), (5, (3059, 3059), (94, 94), 3, True),
    (61, (391, 391), (13, 31), 4, False),
    (241, (254, 254), (1, 24), 2, False), (50, (816, 816), (4, 9), 1, False)])
def test_resident_warps_of_lists_with_64_wide_heads(lib, users, lens, queries, G, dense):
    """Twelve warps per SM, with rings of two slots, where a list needs them and all of its blocks have room: blocks of four warps,
    empty ones included, and clusters that do not fill every place."""
    rng = np.random.default_rng(users)
    ctx, block = context(lib, G=G, D=64)
    ids = np.arange(users, dtype=np.int64)
    L, M = rng.integers(lens[0], lens[1] + 1, users), rng.integers(queries[0], queries[1] + 1, users)
    assert put(lib, ctx, block, ids, L) == 0
    q_off = np.concatenate([[0], np.cumsum(M)]).astype(np.int32)
    assert lib.ckv_set_option(ctx, b"kernel", C.c_int64(2)) == 0
    assert lib.ckv_attend(ctx, users, ptr(ids), ptr(q_off), block, block, None) == 0
    assert np.ctypeslib.as_array(lib.fake_launched(), (6,))[4] == 4 * (2 if dense else 3) * 2 * 32 * 128
    lib.ckv_destroy(ctx)


@pytest.mark.parametrize("d,n,m,G,cluster", [(64, 3359, 1424, 2, 4), (64, 1506, 1058, 4, 4), (32, 686, 1261, 8, 4), (128, 2179, 3901, 3, 4),
                                             (64, 2129, 300, 2, 2), (128, 2153, 14000, 2, 8), (128, 400, 13857, 8, 8),
                                             (128, 7159, 2786, 8, 1), (64, 131072, 16384, 4, 1)])
def test_clusters_of_router_calls(lib, d, n, m, G, cluster):
    """CTAs that share positions lie in a cluster, and clusters of four and eight leave SMs without one."""
    block = device_block(lib, 1 << 20)
    assert lib.ckv_route(0, n, G, d, m, block, block, None, block, 2, None) == 0
    assert np.ctypeslib.as_array(lib.fake_launched(), (6,))[5] == cluster
