"""What a user of the library has it do, as cases that can be timed and compared.

A case is one pass through the public calls (`CollectiveKV`, `ckv_route`, `ckv_project`) the way a serving program
makes them.  Four kinds:

  decode   users' compressed caches are resident; their candidates are attended over them.  `calls` request lists
           per pass (1: the whole resident population at once, as an offline scoring job or the benchmark does;
           more: online serving, where every call names other users than the calls before it).  `host`: queries and
           outputs live in pinned host memory.
  causal   self-attention over the cached sequence: as many queries as positions, each with its visible length.
  prefill  new users: router indices and user-specific parts of their histories, the cache entries, and the first
           decode over them.
  session  a user comes back: the packed history is loaded from the host store, the interactions since are appended,
           the candidates are attended.

Shapes are those of the benchmark workloads (`synth.WORKLOADS`) or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_19178_b200 as ckv

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
BYTES = {"f32": 4, "bf16": 2}


def listed():
    return [
        # Online requests, one user at a time: what a ranking service sends at low load.  Latency and launches count.
        dict(name="online", kind="decode", dtype="bf16", mode="softmax", groups=4, d_user=1, head_dim=32, pool=2048,
             zipf=1.05, resident=64, users=1, len_lo=512, len_hi=512, cand_lo=16, cand_hi=16, calls=8, host=False),
        # A small model in fp32 (workload cfg1).
        dict(name="small_fp32", kind="decode", dtype="f32", mode="softmax", groups=2, d_user=4, head_dim=32, pool=1024,
             zipf=0.0, resident=64, users=64, len_lo=200, len_hi=200, cand_lo=1, cand_hi=1, calls=1, host=False),
        # Ragged online batches: short and long histories, few and many candidates, another request list on every call.
        dict(name="ragged_batches", kind="decode", dtype="bf16", mode="softmax", groups=4, d_user=4, head_dim=64,
             pool=10000, zipf=1.1, resident=1200, users=199, len_lo=17, len_hi=1999, cand_lo=1, cand_hi=40, calls=6,
             host=False),
        # A hundred candidates per user (workload cfg2): the ranking stage behind a retrieval stage.
        dict(name="ranking", kind="decode", dtype="bf16", mode="softmax", groups=8, d_user=2, head_dim=32, pool=4096,
             zipf=1.1, resident=1024, users=1024, len_lo=1024, len_hi=1024, cand_lo=100, cand_hi=100, calls=1,
             host=False),
        # The same with queries and outputs in pinned host memory: the end-to-end figure of the benchmark.
        dict(name="ranking_host", kind="decode", dtype="bf16", mode="softmax", groups=8, d_user=2, head_dim=32,
             pool=4096, zipf=1.1, resident=1024, users=1024, len_lo=1024, len_hi=1024, cand_lo=100, cand_hi=100,
             calls=1, host=True),
        # HSTU-style pointwise attention over long histories with many candidates (workload cfg3).
        dict(name="pointwise", kind="decode", dtype="bf16", mode="silu_over_l", groups=8, d_user=2, head_dim=32,
             pool=8192, zipf=1.2, resident=2048, users=2048, len_lo=4096, len_hi=4096, cand_lo=128, cand_hi=128,
             calls=1, host=False),
        # Long ragged histories, one query per user (workload cfg4).
        dict(name="long_histories", kind="decode", dtype="bf16", mode="softmax", groups=4, d_user=4, head_dim=64,
             pool=16384, zipf=0.0, resident=512, users=512, len_lo=1000, len_hi=16384, cand_lo=1, cand_hi=1, calls=1,
             host=False),
        # A high-concurrency serving batch (workload cfg5).
        dict(name="serving_batch", kind="decode", dtype="bf16", mode="softmax", groups=4, d_user=1, head_dim=32,
             pool=2048, zipf=1.05, resident=65536, users=65536, len_lo=512, len_hi=512, cand_lo=16, cand_hi=16,
             calls=1, host=False),
        # A self-attention block over the cached sequences of a batch of users, causal.
        dict(name="causal", kind="causal", dtype="bf16", mode="softmax", groups=8, d_user=2, head_dim=32, pool=4096,
             zipf=1.1, users=64, len_lo=200, len_hi=1500),
        # One new user: the whole way from the history's inputs to the first scores.
        dict(name="prefill_user", kind="prefill", mode="softmax", groups=2, d_user=4, head_dim=32, pool=1024, d_in=64,
             users=1, len_lo=200, len_hi=200, cand=1),
        # A bulk load of new users into a model with a large pool (the router's benchmark shape).
        dict(name="prefill_batch", kind="prefill", mode="softmax", groups=4, d_user=4, head_dim=64, pool=16384, d_in=64,
             users=256, len_lo=128, len_hi=896, cand=1),
        # A batch of returning users: load from the host store, append what is new, score.
        dict(name="sessions", kind="session", mode="softmax", groups=4, d_user=4, head_dim=64, pool=16384, users=32,
             len_lo=1000, len_hi=16384, new=5, cand=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lengths(rng, lo, hi, ragged=0.7):
    """A range of history lengths inside [lo, hi]; fixed-length workloads are common too."""
    a = _log(rng, lo, hi)
    return (a, a) if rng.random() > ragged else tuple(sorted((a, _log(rng, lo, hi))))


def draw(rng):
    kind = rng.choice(["online", "fp32", "batch", "batch", "many", "many", "long", "host", "causal", "prefill",
                       "prefill", "session"])
    groups = rng.choice([2, 4, 8])
    mode = rng.choice(["softmax", "softmax", "silu_over_l"])
    zipf = rng.choice([0.0, 1.05, 1.1, 1.2])
    du = rng.choice([1, 2, 4])
    if kind == "causal":
        lo, hi = _lengths(rng, 50, 1500)
        return dict(kind="causal", dtype="bf16", mode=mode, groups=groups, d_user=du, head_dim=32,
                    pool=_log(rng, 1024, 10000), zipf=zipf, users=_log(rng, 1, 64), len_lo=lo, len_hi=hi)
    if kind == "prefill":
        lo, hi = _lengths(rng, 30, 900)
        return dict(kind="prefill", mode="softmax", groups=rng.choice([2, 4]), d_user=du,
                    head_dim=rng.choice([32, 64]), pool=_log(rng, 1000, 16384), d_in=rng.choice([32, 64]),
                    users=_log(rng, 1, 145), len_lo=lo, len_hi=hi, cand=rng.choice([1, 16]))
    if kind == "session":
        lo, hi = _lengths(rng, 100, 16384)
        return dict(kind="session", mode="softmax", groups=rng.choice([2, 4]), d_user=du,
                    head_dim=rng.choice([32, 64]), pool=_log(rng, 1024, 16384), users=_log(rng, 1, 32), len_lo=lo,
                    len_hi=hi, new=_log(rng, 1, 40), cand=_log(rng, 1, 40))
    case = dict(kind="decode", dtype="bf16", mode=mode, groups=groups, d_user=du, head_dim=rng.choice([32, 64]),
                pool=_log(rng, 1024, 16384), zipf=zipf)
    if kind == "online":
        lo, hi = _lengths(rng, 30, 2000)
        m_lo, m_hi = sorted((_log(rng, 1, 128), _log(rng, 1, 128)))
        users = _log(rng, 1, 16)
        return dict(case, resident=users * 12, users=users, len_lo=lo, len_hi=hi, cand_lo=m_lo, cand_hi=m_hi, calls=8,
                    host=False)
    if kind == "fp32":
        lo, hi = _lengths(rng, 30, 1000)
        users = _log(rng, 16, 512)
        m = rng.choice([1, 1, 4, 16])
        return dict(case, dtype="f32", pool=_log(rng, 512, 4096), resident=users, users=users, len_lo=lo, len_hi=hi,
                    cand_lo=1, cand_hi=m, calls=1, host=False)
    if kind == "batch":  # up to a few dozen candidates per user, other users on every call or all of them at once
        lo, hi = _lengths(rng, 30, 2000)
        m_lo, m_hi = sorted((_log(rng, 1, 40), _log(rng, 1, 40)))
        calls = rng.choice([1, 6])
        users = max(16, min(_log(rng, 16, 32768 // calls), (1 << 26) // (hi * calls * groups)))
        return dict(case, resident=users * calls, users=users, len_lo=lo, len_hi=hi, cand_lo=m_lo, cand_hi=m_hi,
                    calls=calls, host=False)
    if kind in ("many", "host"):  # dozens to hundreds of candidates per user
        lo, hi = _lengths(rng, 100, 4096)
        m_lo, m_hi = sorted((_log(rng, 50, 200), _log(rng, 50, 200)))
        users = max(8, min(_log(rng, 32, 2048), (1 << 29) // (hi * m_hi)))
        return dict(case, head_dim=32, resident=users, users=users, len_lo=lo, len_hi=hi, cand_lo=m_lo, cand_hi=m_hi,
                    calls=1, host=kind == "host")
    lo, hi = sorted((_log(rng, 500, 16384), _log(rng, 4096, 16384)))
    users = _log(rng, 16, 512)
    return dict(case, mode="softmax", pool=_log(rng, 4096, 16384), resident=users, users=users, len_lo=lo, len_hi=hi,
                cand_lo=1, cand_hi=1, calls=1, host=False)


# ---- inputs ---------------------------------------------------------------------------------------------------

class _Draws:
    """Seeded tensors on the GPU, with the distributions of the benchmark workloads."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.host = np.random.default_rng(seed)
        self.dtype = DTYPES[dtype]

    def normal(self, shape, var):
        x = torch.randn(shape, generator=self.g, device="cuda")
        return x.mul_(math.sqrt(var)).to(self.dtype)

    def indices(self, positions, groups, m, zipf):
        """[positions][groups] int32; Zipf: P(rank r) ~ r^-s, ranks mapped to rows by a permutation per group."""
        if zipf == 0.0:
            return torch.randint(0, m, (positions, groups), generator=self.g, device="cuda", dtype=torch.int32)
        w = torch.arange(1, m + 1, device="cuda", dtype=torch.float64).pow_(-zipf)
        cdf = torch.cumsum(w, 0).div_(w.sum()).float()
        out = torch.empty((positions, groups), device="cuda", dtype=torch.int32)
        for g in range(groups):
            perm = torch.randperm(m, generator=self.g, device="cuda", dtype=torch.int32)
            u = torch.rand(positions, generator=self.g, device="cuda")
            out[:, g] = perm[torch.searchsorted(cdf, u).clamp_(max=m - 1)]
        return out

    def spread(self, lo, hi, n):
        """n whole numbers spread evenly over [lo, hi], in random order."""
        return self.host.permutation(np.linspace(lo, hi, n).round().astype(np.int64))


def _offsets(counts, dtype):
    off = np.zeros(len(counts) + 1, dtype=dtype)
    np.cumsum(counts, out=off[1:])
    return off


def _user_ids(n):
    return np.arange(n, dtype=np.int64) * 7919 + 1000003


def _session(case, d, dtype):
    """A context with the model's pool loaded."""
    G, m, D = case["groups"], case["pool"], case["head_dim"]
    s = ckv.CollectiveKV(G, D, DTYPES[dtype], case["mode"])
    shape = (G, m, D - case["d_user"])
    s.pool_load(d.normal(shape, 1.0 / D), d.normal(shape, 1.0 / D))
    return s


def _put(s, case, d, users, lens):
    """The users' compressed caches, as the prefill stage hands them over."""
    G, D, du = case["groups"], case["head_dim"], case["d_user"]
    off = _offsets(lens, np.int64)
    P = int(off[-1])
    zipf = case.get("zipf", 0.0)
    s.cache_put_batch(users, off, d.indices(P, G, case["pool"], zipf), d.indices(P, G, case["pool"], zipf),
                      d.normal((P, G, du), 1.0 / D), d.normal((P, G, du), 1.0 / D))


def _prepare_decode(case, seed):
    d = _Draws(seed, case["dtype"])
    s = _session(case, d, case["dtype"])
    users = _user_ids(case["resident"])
    _put(s, case, d, users, d.spread(case["len_lo"], case["len_hi"], case["resident"]))
    turn = d.host.permutation(users)
    requests = []
    for c in range(case["calls"]):
        asked = np.ascontiguousarray(turn[c * case["users"]:(c + 1) * case["users"]])
        q_off = _offsets(d.spread(case["cand_lo"], case["cand_hi"], case["users"]), np.int32)
        q = d.normal((int(q_off[-1]), case["groups"], case["head_dim"]), 1.0)
        out = None
        if case["host"]:
            q = q.cpu().pin_memory()
            out = torch.empty_like(q).pin_memory()
        requests.append((asked, q_off, q, out))
    return dict(kind="decode", s=s, requests=requests)


def _prepare_causal(case, seed):
    d = _Draws(seed, case["dtype"])
    s = _session(case, d, case["dtype"])
    users = _user_ids(case["users"])
    lens = d.spread(case["len_lo"], case["len_hi"], case["users"])
    _put(s, case, d, users, lens)
    vis = np.concatenate([np.arange(1, n + 1) for n in lens]).astype(np.int32)
    return dict(kind="causal", s=s, users=users, q_off=_offsets(lens, np.int32), vis=torch.from_numpy(vis).cuda(),
                q=d.normal((int(lens.sum()), case["groups"], case["head_dim"]), 1.0))


def _prepare_prefill(case, seed):
    d = _Draws(seed, "bf16")
    s = _session(case, d, "bf16")
    G, m, d_in, du, D = case["groups"], case["pool"], case["d_in"], case["d_user"], case["head_dim"]
    lens = d.spread(case["len_lo"], case["len_hi"], case["users"])
    n_q = case["users"] * case["cand"]
    return dict(kind="prefill", s=s, m=m, d_in=d_in, users=_user_ids(case["users"]), off=_offsets(lens, np.int64),
                q_off=_offsets([case["cand"]] * case["users"], np.int32), q=d.normal((n_q, G, D), 1.0),
                x=d.normal((int(lens.sum()), d_in), 1.0 / d_in),
                router=[(d.normal((G, m, d_in), 1.0), d.normal((G, m), 0.01).float()) for _ in range(2)],
                linear=[(d.normal((G, du, d_in), 1.0 / D), d.normal((G, du), 0.01 / D).float()) for _ in range(2)])


def _prepare_session(case, seed):
    d = _Draws(seed, "bf16")
    s = _session(case, d, "bf16")
    G, D, du = case["groups"], case["head_dim"], case["d_user"]
    users = _user_ids(case["users"])
    lens = d.spread(case["len_lo"], case["len_hi"], case["users"])
    _put(s, case, d, users, lens)
    stored = s.export_blob(users)  # what the host store keeps
    new = [(d.indices(case["new"], G, case["pool"], 0.0), d.indices(case["new"], G, case["pool"], 0.0),
            d.normal((case["new"], G, du), 1.0 / D), d.normal((case["new"], G, du), 1.0 / D)) for _ in users]
    return dict(kind="session", s=s, users=users, lens=lens.astype(np.int32), stored=stored, new=new,
                q_off=_offsets([case["cand"]] * case["users"], np.int32),
                q=d.normal((case["users"] * case["cand"], G, D), 1.0))


def prepare(case, seed):
    return {"decode": _prepare_decode, "causal": _prepare_causal, "prefill": _prepare_prefill,
            "session": _prepare_session}[case["kind"]](case, seed)


# ---- one pass -------------------------------------------------------------------------------------------------

def _run_prefill(st):
    s, x, G = st["s"], st["x"], st["s"].n_groups
    n = x.shape[0]
    idx, part = [], []
    for W, b in st["router"]:
        idx.append(torch.empty((n, G), dtype=torch.int32, device=x.device))
        ckv.ckv_route(0, n, G, st["d_in"], st["m"], x, W, b, idx[-1])
    for W, b in st["linear"]:
        part.append(torch.empty((n, G, s.d_user), dtype=torch.bfloat16, device=x.device))
        ckv.ckv_project(0, n, G, st["d_in"], s.d_user, x, W, b, part[-1])
    s.cache_put_batch(st["users"], st["off"], idx[0], idx[1], part[0], part[1])
    return dict(idx=idx, part=part, out=s.attend(st["users"], st["q_off"], st["q"]))


def _run_session(st):
    s = st["s"]
    s.import_blob(st["users"], st["lens"], st["stored"])
    for u, new in zip(st["users"], st["new"]):
        s.cache_append(int(u), *new)
    return s.attend(st["users"], st["q_off"], st["q"])


def run(st):
    if st["kind"] == "decode":
        return [st["s"].attend(users, q_off, q, out) for users, q_off, q, out in st["requests"]]
    if st["kind"] == "causal":
        return st["s"].attend_visible(st["users"], st["q_off"], st["vis"], st["q"])
    return _run_prefill(st) if st["kind"] == "prefill" else _run_session(st)


# ---- what a pass cannot do without ----------------------------------------------------------------------------

def work(case):
    """The pool, the compressed caches, queries and outputs once each; two products per (query, position) pair."""
    G, D, du, m = case["groups"], case["head_dim"], case["d_user"], case["pool"]
    e = BYTES[case.get("dtype", "bf16")]
    mean_L = 0.5 * (case["len_lo"] + case["len_hi"])
    unit = 2 * 2 + 2 * du * e                      # two 16-bit pool indices and the user parts of K and V
    pool = 2 * G * m * (D - du) * e
    if case["kind"] == "causal":
        n = np.linspace(case["len_lo"], case["len_hi"], case["users"])
        Q, P, pairs = float(n.sum()), float(n.sum()), float((n * (n + 1) / 2).sum())
    elif case["kind"] == "decode":
        P = case["users"] * case["calls"] * mean_L
        Q = case["users"] * case["calls"] * 0.5 * (case["cand_lo"] + case["cand_hi"])
        pairs = Q * mean_L
    else:
        P = case["users"] * (mean_L + case.get("new", 0))
        Q = case["users"] * case["cand"]
        pairs = P * case["cand"]
    w = {"bytes": pool + P * G * unit + 2 * Q * G * D * e, "flops": 4.0 * D * G * pairs}
    if case["kind"] == "prefill":
        d_in = case["d_in"]
        w["bytes"] += P * d_in * 2 + 2 * G * (m + du) * (d_in * 2 + 4) + 2 * P * G * (4 + 2 * du)
        w["flops"] += 2 * 2.0 * P * G * (m + du) * d_in
    return w


def tolerance(case):
    """fp32: rounding of 32-bit sums.  bf16: attention weights and outputs are rounded to 8 bits of mantissa; router
    scores closer together than the rounding of their fp32 sums may resolve to either entry."""
    if case.get("dtype") == "f32":
        return {"rel": 1e-5}
    return {"rel": 1e-2, "differ": 1e-4}
