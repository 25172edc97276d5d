"""The workloads the compression pass is measured on, through the package's public entry points.

A case names one kind of call and its shape:
  compress      the fused pass, `kvc.compress` (bf16 or fp32 caches, any window, batch, options)
  unstructured  the per-head variant, `kvc.kvc_compress_unstructured`
  sharded       one rank's share of a head-sharded sequence, `sharded.run_head_sharded` (a group of one rank: the
                all-reduces are the identity, everything the GPU of a rank does is there)

Inputs come from `workloads.make_workload`: N(0, sigma^2) tensors with attention sinks and heavy hitters.  `sigma` 0 is
that recipe's own default, 1 / sqrt(head_dim) (nearly uniform attention); 1 gives logits of unit variance.
"""
import math

import torch

import paper_2509_05165_b200 as kvc
from paper_2509_05165_b200 import sharded, workloads as W
from paper_2509_05165_b200.binding import alloc_outputs

_BASE = dict(kind="compress", layers=32, q_heads=32, kv_heads=8, head_dim=128, n_ctx=8192, window=32, batch=1,
             dtype="bf16", retention=0.25, sigma=1.0, hh="uniform", hh_frac=0.01, keep=False, task_after=False,
             value_norm=False, position_order=False, min_keep=0)


def _case(**kw):
    return dict(_BASE, **kw)


def listed():
    return [
        # the smallest configuration of the benchmark: two layers in fp32, a handful of launches
        _case(name="tiny_f32", layers=2, q_heads=4, kv_heads=2, head_dim=64, n_ctx=512, window=16, dtype="f32",
              sigma=0.0, hh_frac=0.02, keep=True),
        # a short prompt on the 8B shape: latency, launches and host work
        _case(name="prompt_1k", n_ctx=1000),
        # the length the method is evaluated at, half of the cache kept, intermediates returned
        _case(name="eval_4k", n_ctx=4096, retention=0.5, keep=True),
        # the 8B shape at 8K, a fifth kept (heavy hitters of per-layer strength)
        _case(name="llama8b_8k", retention=0.20, sigma=0.0),
        # the benchmark's default: the 8B shape at 32K, heavy hitters in bursts, a quarter kept
        _case(name="llama8b_32k", n_ctx=32768, sigma=0.0, hh="bursts", hh_frac=0.005),
        # the long-context shape: GQA group of 7, window 64, 128K tokens, a tenth kept
        _case(name="gqa4_128k", layers=28, q_heads=28, kv_heads=4, n_ctx=131072, window=64, retention=0.10, sigma=0.0,
              hh="loguniform"),
        # a serving batch of prompts of an odd length, smaller heads, strong compression
        _case(name="batch4_odd_d64", head_dim=64, n_ctx=5003, batch=4, retention=0.05),
        # an fp32 cache of an odd length, intermediates returned
        _case(name="fp32_3k", layers=16, n_ctx=3001, dtype="f32", retention=0.3, keep=True),
        # the options together: value-norm weighting, K' in position order, a floor for every layer
        _case(name="options_16k", n_ctx=16384, value_norm=True, position_order=True, min_keep=256),
        # every head keeps its own tokens (ragged cache)
        _case(name="unstructured_8k", kind="unstructured", retention=0.20),
        # task-aware scoring: a question of 500 tokens after the context scores it, nothing is masked
        _case(name="question_500", n_ctx=4096, window=500, task_after=True, retention=0.10),
        # one of four tensor-parallel ranks: two KV heads of the 8B shape at 32K
        _case(name="shard_of_4_32k", kind="sharded", q_heads=8, kv_heads=2, n_ctx=32768, keep=True),
    ]


def _rows(c):
    """Scoring rows per KV head."""
    return c["q_heads"] // c["kv_heads"] * c["window"]


def _cost(c):
    """Logits of one pass: what a drawn case is bounded by."""
    return c["layers"] * c["batch"] * c["kv_heads"] * float(c["n_ctx"]) * max(128, _rows(c))


_LARGEST = 28 * 4 * 131072.0 * 448
_LARGEST_KV = 6 * 2 ** 30


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["compress"] * 5 + ["unstructured", "sharded"])
        f32 = kind == "compress" and rng.random() < 0.2
        layers = rng.choice([2, 4, 8, 16, 28, 32, rng.randint(2, 32)])
        kv_heads = rng.choice([2, 4, 8]) if kind != "sharded" else rng.choice([1, 2, 4])
        group = rng.choice([1, 2, 4, 4, 4, 7])
        window = rng.choice([8, 16, 32, 32, 32, 64, 64, 128, rng.randint(1, 128), rng.randint(129, 600)])
        n_ctx = _log_int(rng, 256, 4096) if f32 else _log_int(rng, 256, 131072)
        if rng.random() < 0.3:
            n_ctx = max(256, n_ctx // 1024 * 1024)
        c = _case(kind=kind, layers=layers, q_heads=kv_heads * group, kv_heads=kv_heads, head_dim=rng.choice([64, 128, 128]),
                  n_ctx=n_ctx, window=min(window, n_ctx), batch=rng.choice([1, 1, 1, 2, 4, 8]) if kind != "sharded" else 1,
                  dtype="f32" if f32 else "bf16", retention=round(rng.choice([0.05, 0.10, 0.20, 0.25, 0.50, rng.uniform(0.02, 0.6)]), 3),
                  sigma=rng.choice([0.0, 1.0, 1.0]), hh=rng.choice(["uniform", "uniform", "loguniform"]),
                  hh_frac=rng.choice([0.005, 0.01, 0.02]), keep=kind == "sharded" or rng.random() < 0.5,
                  task_after=kind == "compress" and rng.random() < 0.2,
                  value_norm=kind != "sharded" and rng.random() < 0.2, position_order=rng.random() < 0.2)
        if kind == "compress" and rng.random() < 0.2:
            c["min_keep"] = int(c["retention"] * n_ctx * 0.5)
        kv_bytes = 2.0 * layers * c["batch"] * kv_heads * n_ctx * c["head_dim"] * (4 if f32 else 2)
        # no larger than the largest listed case; fp32 caches stay in the range of theirs
        if _cost(c) <= _LARGEST * (0.03 if f32 else 1.0) and kv_bytes <= _LARGEST_KV:
            return c


def _config(c, seed):
    return W.WorkloadConfig("case", c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], c["n_ctx"], c["window"],
                            batch=c["batch"], dtype=c["dtype"], retention=c["retention"], hh_frac=c["hh_frac"],
                            hh_mode=c["hh"], elem_std=c["sigma"] or None, seed=seed)


def prepare(case, seed):
    """Inputs on the GPU, the descriptor, and the output buffers and workspace a serving program keeps."""
    c = dict(_BASE, **case)
    dev = torch.device("cuda")
    cfg = _config(c, seed)
    wl = W.make_workload(cfg, dev)
    if c["value_norm"]:
        # value rows of very different lengths, as real caches have them
        gen = torch.Generator(device=dev).manual_seed(seed + 1)
        for layer, v in enumerate(wl.v):
            wl.v[layer] = (v.float() * torch.exp(4.0 * torch.rand(v.shape[:-1] + (1,), generator=gen, device=dev))).to(v.dtype)
    desc = kvc.desc_from_config(cfg, value_norm=int(c["value_norm"]), keep_position_order=int(c["position_order"]),
                                min_keep_per_layer=c["min_keep"])
    if c["task_after"]:
        desc.q_pos0 = c["n_ctx"]
    st = dict(kind=c["kind"], wl=wl, desc=desc, budget=cfg.budget)
    if c["kind"] == "sharded":
        desc.augment_head_mean = 0
        st["backend"] = sharded.KvcBackend(wl.q, wl.k, wl.v, desc, cfg.budget)
        st["info"] = sharded.ShardInfo(1, c["kv_heads"], desc.agg_head)
    elif c["kind"] == "unstructured":
        n, heads, dt = cfg.budget * c["kv_heads"], c["layers"] * c["kv_heads"], wl.k[0].dtype
        st.update(entries=n, k_out=torch.empty((c["batch"], n * c["head_dim"]), dtype=dt, device=dev),
                  v_out=torch.empty((c["batch"], n * c["head_dim"]), dtype=dt, device=dev),
                  n_keep=torch.empty((c["batch"], c["layers"], c["kv_heads"]), dtype=torch.int32, device=dev),
                  offsets=torch.empty((c["batch"], heads + 1), dtype=torch.int64, device=dev),
                  status=torch.zeros(1, dtype=torch.int32, device=dev),
                  ws=torch.empty(kvc.kvc_workspace_size(desc, 0), dtype=torch.uint8, device=dev))
    else:
        st["out"] = alloc_outputs(desc, cfg.budget, wl.k[0].dtype, dev, keep_intermediates=c["keep"])
    return st


def _no_reduce(tensor, op):
    """The all-reduce of a group of one rank."""


def run(state):
    wl, desc = state["wl"], state["desc"]
    if state["kind"] == "unstructured":
        s = state
        kvc.kvc_compress_unstructured(desc, wl.q, wl.k, wl.v, s["entries"], s["k_out"], s["v_out"], s["n_keep"],
                                      s["offsets"], device_status=s["status"], workspace=s["ws"])
        return [s["k_out"], s["v_out"], s["n_keep"], s["offsets"], s["status"]]
    if state["kind"] == "sharded":
        o = sharded.run_head_sharded(state["backend"], state["info"], _no_reduce)
    else:
        o = kvc.compress(wl.q, wl.k, wl.v, desc, state["budget"], out=state["out"])
    return [o.k_out, o.v_out, o.n_keep, o.offsets, o.device_status, o.idx, o.scores, o.composite]


def work(case):
    """K and Q read once, V where it is needed, K' and V' written, the intermediates that go back to the caller; one
    product of the queries with every key (what the causal mask leaves out of it is a rounding error)."""
    c = dict(_BASE, **case)
    e = 4 if c["dtype"] == "f32" else 2
    seqs = c["layers"] * c["batch"]
    kv = float(seqs * c["kv_heads"] * c["n_ctx"] * c["head_dim"] * e)
    q = float(seqs * c["q_heads"] * c["window"] * c["head_dim"] * e)
    kept = _config(c, 0).budget / float(c["layers"] * c["n_ctx"])
    v_read = 1.0 if c["value_norm"] else kept
    back = seqs * c["n_ctx"] * (8.0 * c["kv_heads"] + 4.0) if c["keep"] else 0.0
    return {"bytes": kv * (1.0 + v_read + 2.0 * kept) + q + back,
            "flops": 2.0 * seqs * c["q_heads"] * c["window"] * float(c["n_ctx"]) * c["head_dim"]}


def tolerance(case):
    """Exact.  Which rows come out, and in what order, is decided by comparing fp32 scores that lie as close as one unit
    in the last place: sums taken in another order agree to about 1e-6 in the scores, yet move whole rows of K' and V',
    and a row that moved is as far from the one in its place as two random rows are (relative error 1.4), which no bound
    on a norm expresses.  The library's results are reproducible bit for bit, so they are compared that way."""
    return "exact"
