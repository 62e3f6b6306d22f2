"""The performance cases of the relay-race inference path, through the calls a serving process makes.

Four kinds of pass, as in the paper's serving flow:

* ``preinfer``  - users arrive: pages are reserved (the users' previous pages given back first), their prefixes run
  through every layer and the per-layer K / V land in the pool.  Output: the pool's slab.
* ``rank``      - short-term tokens and candidates attend to the cached prefixes.  Output: one score per candidate.
* ``full``      - the fallback when a user's cache is gone: prefix, short-term tokens and candidates in one call.
* ``reload_rank`` - the users' pages have left HBM (a copy is in pinned host memory): evict, reload, rank.

A state is what such a process holds for one stream of requests: a model slot (weights shared by all slots of the
process, a workspace of its own), a pool, and one batch of requests.  Weights depend on the model alone; users'
histories, short-term tokens and candidates come from the seed.  Item ids are Zipf(1.1) over the catalogue.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2601_01712_b200 import binding, runtime, synth, workloads

# The repository's own model shapes: the tiny fp32 model, the production-shaped bf16 model (with softmax and with
# pointwise attention), the long-sequence model, the paper's Table 1 shape (2K-token prefixes, 8 layers, dim 256, fp32),
# and the widest model the kernels take (the paper's dims go from 128 to 1024).
MODELS = {
    "tiny_f32": synth.MODEL_TINY,
    "prod": synth.MODEL_PROD,
    "prod_pointwise": synth.ModelShape(4, 256, 4, 64, 1024, 1_000_000, synth.DTYPE_BF16, attn_kind=1),
    "long": synth.MODEL_LONG,
    "table1_f32": synth.ModelShape(8, 256, 4, 64, 1024, 200_000, synth.DTYPE_F32),
    "wide": synth.ModelShape(4, 1024, 16, 64, 4096, 200_000, synth.DTYPE_BF16),
}


def _case(mode, model, users, prefix, short, cand, ragged=False, shuffled=False):
    """`ragged`: every user has lengths of its own, prefixes from a sixteenth of `prefix` up to it, short-term and candidate counts
    from an eighth.  `shuffled`: pages scattered over the pool, as after hours of users coming and going."""
    return {"mode": mode, "model": model, "users": users, "prefix": prefix, "short": short, "cand": cand, "ragged": ragged,
            "shuffled": shuffled}


def listed():
    return [
        # the smallest model and batch: a call is a chain of short launches
        {"name": "rank_tiny_f32", **_case("rank", "tiny_f32", 4, 256, 32, 64)},
        # one request at a time, the paper's granularity: latency of the ranking stage ...
        {"name": "rank_one", **_case("rank", "prod", 1, 2048, 64, 512)},
        # ... and of the pre-inference that ran ahead of it (a history is any number of tokens)
        {"name": "preinfer_one", **_case("preinfer", "prod", 1, 1999, 0, 0)},
        # the production-shaped batch the benchmark times: ranking and pre-inference
        {"name": "rank_batch", **_case("rank", "prod", 32, 2048, 64, 512)},
        {"name": "preinfer_batch", **_case("preinfer", "prod", 32, 2048, 0, 0)},
        # users of every kind in one call on a fragmented pool
        {"name": "rank_ragged", **_case("rank", "prod", 128, 8192, 128, 1024, ragged=True, shuffled=True)},
        # the deeper, wider model over long histories
        {"name": "rank_long", **_case("rank", "long", 16, 8192, 128, 1024)},
        # the longest history of a single user
        {"name": "preinfer_long", **_case("preinfer", "long", 1, 24576, 0, 0)},
        # a group of cache misses on the widest model
        {"name": "full_wide", **_case("full", "wide", 8, 2048, 64, 512, ragged=True)},
        # the pointwise (HSTU-style) attention of the paper's model family
        {"name": "rank_pointwise", **_case("rank", "prod_pointwise", 32, 2048, 64, 512, ragged=True)},
        # the paper's default precision at its Table 1 shape
        {"name": "rank_f32", **_case("rank", "table1_f32", 8, 2048, 64, 512)},
        # users whose pages are in the DRAM tier when their request comes
        {"name": "reload_rank", **_case("reload_rank", "prod", 8, 4096, 64, 512)},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    # at most the work of the largest listed case: a pass of its own, and with the pre-inference that a ranking case needs first
    most = {False: max(_flops(c) for c in listed() if not _f32(c)), True: max(_flops(c, True) for c in listed() if _f32(c))}
    while True:
        mode = rng.choices(["rank", "preinfer", "full", "reload_rank"], [8, 5, 4, 2])[0]
        model = "prod" if mode == "reload_rank" else rng.choices(list(MODELS), [2, 5, 2, 3, 2, 2])[0]
        if model == "tiny_f32":
            users, prefix = _spread(rng, 1, 16), _spread(rng, 32, 1024)
        else:
            users, prefix = _spread(rng, 1, 128), _spread(rng, 256, 24576)
        short, cand = (0, 0) if mode == "preinfer" else (rng.randint(0, 128), _spread(rng, 32, 1024))
        c = _case(mode, model, users, prefix, short, cand, ragged=users > 1 and rng.random() < 0.6, shuffled=rng.random() < 0.5)
        if mode == "reload_rank" and users * MODELS[model].kv_bytes(prefix) > 160 << 20:      # what is loaded, as well
            continue
        if _flops(c, _f32(c)) <= most[_f32(c)]:
            return c


def _f32(case):
    return MODELS[case["model"]].dtype == synth.DTYPE_F32


def _lengths(case):
    """(P, S, C) of every user: part of the case, not of the seed."""
    n, p, s, c = case["users"], case["prefix"], case["short"], case["cand"]
    if not case["ragged"]:
        return [(p, s, c)] * n
    rng = random.Random("%d %d %d %d" % (n, p, s, c))
    return [(_spread(rng, max(1, p // 16), p), rng.randint(s // 8, s), rng.randint(c // 8, c)) for _ in range(n)]


def _flops(case, with_prefix=False):
    shape, of = MODELS[case["model"]], workloads
    total = 0.0
    for p, s, c in _lengths(case):
        if case["mode"] == "preinfer" or (with_prefix and case["mode"] != "full"):
            total += of.flops_preinfer(shape, p)
        if case["mode"] == "full":
            total += of.flops_full(shape, p, s, c)
        elif case["mode"] != "preinfer":
            total += of.flops_rank(shape, p, s, c)
    return total


def work(case):
    shape = MODELS[case["model"]]
    es = 4 if _f32(case) else 2
    d, L, F = shape.d_model, shape.n_layers, shape.d_ff
    n_bytes = L * (4 * d * d + 2 * d * F) * es                          # the layers' matrices
    for p, s, c in _lengths(case):
        rows = {"preinfer": p, "full": p + s + c}.get(case["mode"], s + c)
        n_bytes += rows * (4 + d * es) + 4 * c                          # ids, their table rows, scores
        if case["mode"] in ("preinfer", "rank", "reload_rank"):
            n_bytes += shape.kv_bytes(p)                                # K / V of the prefix, written or read
        if case["mode"] == "reload_rank":
            n_bytes += 2 * shape.kv_bytes(p)                            # ... and brought from host memory into the pool first
    return {"bytes": n_bytes, "flops": _flops(case)}


def tolerance(case):
    # fp32 model: sums of up to a few thousand fp32 terms through eight layers.  bf16 model: operands of every matrix product
    # are rounded to bf16 (2^-9), and a different order of the fp32 sums flips some of those roundings.
    return {"rel": 1e-5} if _f32(case) else {"rel": 1e-2}


@functools.lru_cache(maxsize=None)
def _model(name):
    """The process's model: weights of the distributions of synth.make_weights, drawn on the GPU (the table alone is up to 0.5 G values)."""
    shape = MODELS[name]
    L, d, F, V = shape.n_layers, shape.d_model, shape.d_ff, shape.vocab
    gen = torch.Generator(device="cuda").manual_seed(synth.BASE_SEED + L + d)
    w = synth.Weights(shape)

    def normal(dims, mean, std):
        return torch.randn(dims, generator=gen, device="cuda", dtype=torch.float32).mul_(std).add_(mean)

    for n, dims, std in (("emb", (V, d), d ** -0.5), ("w_qkv", (L, 3 * d, d), d ** -0.5), ("w_o", (L, d, d), d ** -0.5),
                         ("w1", (L, F, d), d ** -0.5), ("w2", (L, d, F), F ** -0.5)):
        t = normal(dims, 0.0, std)
        if shape.dtype == synth.DTYPE_BF16:
            t = t.bfloat16()
            w.bits[n] = t.view(torch.int16).cpu().numpy().view(np.uint16)
            t = t.float()
        w.mat[n] = t.cpu().numpy()
    for n, dims, mean, std in (("ln1_g", (L, d), 1, 0.1), ("ln1_b", (L, d), 0, 0.1), ("ln2_g", (L, d), 1, 0.1), ("ln2_b", (L, d), 0, 0.1),
                               ("b_qkv", (L, 3 * d), 0, 0.02), ("b_o", (L, d), 0, 0.02), ("b1", (L, F), 0, 0.02), ("b2", (L, d), 0, 0.02),
                               ("lnf_g", (d,), 1, 0.1), ("lnf_b", (d,), 0, 0.1), ("w_score", (d,), 0, d ** -0.5), ("b_score", (1,), 0, 0.02)):
        w.vec[n] = normal(dims, float(mean), std).cpu().numpy()
    return runtime.Model(shape, w)


@functools.lru_cache(maxsize=None)
def _zipf(vocab):
    return synth.ZipfIds(vocab, 1.1)


class State:
    def __init__(self, case, seed):
        self.mode = case["mode"]
        self.slot, self.pool = _model(case["model"]).new_slot(), None
        shape = self.slot.shape
        self.lengths = [(int(p), int(s), int(c)) for p, s, c in _lengths(case)]
        rng = np.random.default_rng(seed)
        p, s, c = zip(*self.lengths)
        self.host_batch = synth.make_batch(_zipf(shape.vocab), rng, p, s, c)
        self.batch = runtime.DeviceBatch(self.host_batch, self.slot.device)
        self.users = [int(u) for u in self.host_batch.users]
        counts = [synth.pages_for(n) for n in p]
        rows = {"preinfer": sum(p), "full": sum(p) + sum(s) + sum(c)}.get(self.mode, max(sum(p), sum(s) + sum(c)))
        self.slot.reserve(rows, len(p), sum(counts))
        self.scores = torch.empty(max(1, sum(c)), dtype=torch.float32, device=self.slot.device)
        if self.mode == "full":
            return
        reload = self.mode == "reload_rank"
        self.pool = runtime.KvPool(self.slot, sum(counts), sum(counts) if reload else 0)
        order = np.random.default_rng(len(p)).permutation(sum(counts)) if case["shuffled"] else np.arange(sum(counts))
        self.pages = np.split(order.astype(np.int32), np.cumsum(counts)[:-1])
        for u, n, ids in zip(self.users, p, self.pages):
            self.pool.alloc(u, n, ids)
        if self.mode != "preinfer":
            self.pool.preinfer(self.batch)
        if reload:
            binding.relaygr_kv_set_max_inflight_reloads(self.pool.pool, max(64, 2 * len(p)))
            self.side = torch.cuda.Stream()
            self.done = torch.cuda.Event()
            self.done.record()
            for u in self.users:
                self.pool.evict(u, True, self.side)
                self.pool.reload(u, self.side)

    def __del__(self):
        if self.pool is not None:
            self.pool.close()
        self.slot.close()


def prepare(case, seed):
    return State(case, seed)


def run(state):
    pool = state.pool
    if state.mode == "full":
        return state.slot.rank_full(state.batch, state.scores)
    if state.mode == "preinfer":
        for u in state.users:
            pool.free(u, ok=(binding.OK, binding.E_MISS))
        for u, (p, _, _), ids in zip(state.users, state.lengths, state.pages):
            pool.alloc(u, p, ids)
        pool.preinfer(state.batch)
        return pool.slab.view(state.slot.torch_dtype)
    if state.mode == "reload_rank":
        state.done.synchronize()                       # one call in flight per pool: its users' reloads must have ended before they can be evicted
        for u in state.users:
            pool.evict(u, True, state.side)            # a host copy exists: the pages are given back and nothing is copied
        for u in state.users:
            pool.reload(u, state.side)
        scores = pool.rank(state.batch, state.scores)
        state.done.record()
        return scores
    return pool.rank(state.batch, state.scores)
