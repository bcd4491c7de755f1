"""Performance cases of the cached MoE layer: the calls that a program serving a model with it makes.

A "layer" case is a stack of layers under a bounded expert cache, one handle per layer, driven through
MoELayer.forward (or forward_host): decode steps of a few tokens, or prompts.  Its sizes are those of the
workload shapes in gen.CONFIGS.  A "proxy" case evaluates the cache-miss proxies of recorded routing traces,
from which a deployment chooses its layers' cache sizes.

Fields of a layer case: d, F, E, k, C (d_model, d_ff, experts, top-k, cache slots per layer), shared (always
resident experts), store ("bf16", "q4": 4-bit host store and bf16 slots, "q4slots": 4-bit store and slots),
tokens (of one call), seqs (sequences they belong to, each with a router bias of its own of concentration
alpha), layers, steps (calls of every layer in one pass, with inputs of their own), policy, host (buffers of the
call in page-locked host memory).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import gen
import paper_2602_11192_b200 as M

STATS_WORDS = 12    # int32 words of one melinoe_moe_stats record


def _layer(name, cfg, **kw):
    """A layer case with the sizes of one of the workload shapes."""
    c = gen.config_by_name(cfg)
    case = {"name": name, "kind": "layer", "d": c.d_model, "F": c.d_ff, "E": c.n_experts, "k": c.top_k, "C": c.n_experts,
            "shared": c.n_shared, "store": "bf16", "tokens": c.batch, "seqs": c.batch, "alpha": c.alphas[0], "layers": 1,
            "steps": 1, "policy": "lru", "host": False}
    case.update(kw)
    return case


def listed():
    return [
        # one token through one small layer that fits its cache: launches and latency
        _layer("tiny decode", "tiny", C=4),
        # token-by-token generation, every expert resident: one token through all 16 layers
        _layer("olmoe decode", "olmoe", layers=16),
        # the same model in the memory of a quarter of its experts: 16 tokens of one sequence, with the
        # misses that its routing makes, inputs and results in host memory
        _layer("olmoe decode small cache", "olmoe", C=16, layers=4, steps=16, host=True),
        # the same with 4-bit experts, of which almost all fit the same memory
        _layer("olmoe decode 4-bit", "olmoe", C=60, layers=16, store="q4slots"),
        # eight sequences decoded together by a wide model with few large experts
        _layer("phi35 decode batch 8", "phi35", layers=2),
        # four sequences, many small experts and two shared ones
        _layer("deepseek decode batch 4", "deepseek", layers=4),
        # a short prompt: a handful of tokens per expert, so reading the weights is the work
        _layer("olmoe prompt 128", "olmoe", tokens=128, layers=4),
        # the same prompt where only a quarter of the experts fit: the host link is the work
        _layer("olmoe prompt small cache", "olmoe", tokens=128, C=16, layers=2),
        # a prompt with 4-bit experts
        _layer("olmoe prompt 512 4-bit", "olmoe", tokens=512, C=60, layers=1, store="q4slots"),
        # the prompts of a batch: hundreds of tokens per expert, so the tensor cores are the work
        _layer("phi35 prompts 8x512", "phi35", tokens=4096, seqs=8),
        _layer("deepseek prompts 4x2048", "deepseek", tokens=8192, seqs=4),
        # cache sizes of a 16-layer model from the routing of 512 tokens: every size of every layer
        {"name": "proxies of a trace", "kind": "proxy", "layers": 16, "tokens": 512, "k": 8, "E": 64, "gamma": 0.9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.1:
        E = rng.choice((8, 16, 24, 32, 60, 64))
        return {"kind": "proxy", "layers": rng.randint(1, 16), "tokens": _log_int(rng, 64, 512),
                "k": rng.randint(1, min(8, E)), "E": E, "gamma": rng.choice((1.0, 0.9, 0.5))}
    store = rng.choice(("bf16", "bf16", "bf16", "q4slots", "q4"))
    small = rng.random() < 0.3 or store == "q4"        # the cache holds a part of the experts
    prompt = rng.random() < 0.45
    while True:
        d = rng.choice((512, 1024, 2048, 4096)) if store == "q4slots" else 256 * _log_int(rng, 1, 16)
        # mostly whole 128-row blocks of hidden units, some ragged
        F = 128 * _log_int(rng, 2, 112) if rng.random() < 0.75 else 8 * _log_int(rng, 32, 1792)
        E = _log_int(rng, 4, 64)
        k = rng.randint(1, min(8, E))
        shared = rng.choice((0, 0, 0, 1, 2)) if store != "q4" else 0
        tokens = _log_int(rng, 9, 8192) if prompt else rng.randint(1, 8)
        expert = 6 * d * F
        C = rng.randint(k, max(k, E // 2)) if small else E
        # no more than the largest listed cases: host store, arithmetic of a prompt, bytes over the host link, weights
        # read where every eight tokens may read theirs
        if E * expert > 2.6e9 or expert < 3.9e5 or 6.0 * d * F * tokens * (k + shared) > 1.1e12:
            continue
        read = min(E, tokens * k) * expert
        link = read if store == "bf16" else 0.27 * read
        if small and link > 4.5e8:
            continue
        if prompt and (F % 128 or store == "q4slots") and -(-tokens // 8) * min(E, 8 * k) * expert > 3.0e10:
            continue
        break
    layers = 1 if prompt else max(1, min(16, int(2.0e9 / read), int(12.0e9 / (C * expert))))
    steps = 1
    if small and not prompt:
        steps = max(1, min(rng.randint(2, 8), int(4.5e8 / link)))
        layers = max(1, min(layers, 4, int(4.5e8 / (link * steps))))
    return {"kind": "layer", "d": d, "F": F, "E": E, "k": k, "C": C, "shared": shared, "store": store, "tokens": tokens,
            "seqs": min(tokens, rng.randint(1, 8)) if prompt else tokens, "alpha": rng.choice((0.1, 0.3, 1.0)),
            "layers": layers, "steps": steps,
            "policy": rng.choice(("lru", "count")) if small else "lru", "host": not prompt and rng.random() < 0.25}


def _expert_bytes(c):
    return M.melinoe_moe_expert_bytes(c["d"], c["F"]) if c["store"] == "bf16" else M.melinoe_moe_expert_bytes_q4(c["d"], c["F"])


_stores = {}        # the model's page-locked expert store, shared by all states of a case as by all sessions of a server


def _random_blobs(c, n, device_slots):
    """n experts in the store's format.  A bf16 blob is a permutation of the expert's weights, so independent weights
    N(0, 0.02^2) can be drawn in blob order; a 4-bit blob is codes and positive scales (the largest weight of 64 is
    about 2.4 standard deviations, over 7 steps)."""
    g = torch.Generator(device="cuda").manual_seed(c["d"] * 131 + c["F"])
    nb = _expert_bytes(c)
    out = torch.empty((n, nb), dtype=torch.uint8, device="cuda") if device_slots else \
        torch.empty((n, nb), dtype=torch.uint8, pin_memory=True)
    for e in range(n):
        if c["store"] == "bf16":
            w = torch.empty(nb // 2, device="cuda").normal_(0.0, 0.02, generator=g).to(torch.bfloat16)
            out[e].copy_(w.view(torch.uint8))
        else:
            d, F = c["d"], c["F"]
            unit = torch.zeros((F, nb // F), dtype=torch.uint8, device="cuda")
            w = torch.empty((F, 3 * d // 2, 2), device="cuda").normal_(0.0, 1.0, generator=g)
            q = (w * (7.0 / 2.4)).round_().clamp_(-8, 7).add_(8).to(torch.uint8)
            unit[:, :3 * d // 2] = q[:, :, 0] | (q[:, :, 1] << 4)
            s = torch.empty((F, 3 * d // 64), device="cuda").uniform_(0.9, 1.1, generator=g) * (0.02 * 2.4 / 7.0)
            unit[:, 3 * d // 2:3 * d // 2 + 3 * d // 32] = s.to(torch.bfloat16).view(torch.uint8).reshape(F, -1)
            out[e].copy_(unit.reshape(-1))
    torch.cuda.synchronize()
    return out


def _store(c):
    key = (c["d"], c["F"], c["E"], c["store"], c["shared"])
    if key not in _stores:
        _stores.clear()
        # the always resident experts are in the slots' format and in device memory
        dev = dict(c, store="q4") if c["store"] == "q4slots" else dict(c, store="bf16")
        _stores[key] = (_random_blobs(c, c["E"], False), _random_blobs(dev, c["shared"], True) if c["shared"] else None)
    return _stores[key]


class _State:
    pass


def _prepare_layers(c, seed):
    s = _State()
    s.store, s.shared = _store(c)
    T, d, E, L, S = c["tokens"], c["d"], c["E"], c["layers"], c["steps"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    s.stream = torch.cuda.current_stream().cuda_stream
    s.layers = []
    nb, base = s.store.shape[1], s.store.data_ptr()
    seq = torch.arange(T, dtype=torch.int32, device="cuda") * c["seqs"] // T
    for l in range(L):
        m = M.MoELayer(d, c["F"], E, c["k"], c["C"], slots="q4" if c["store"] == "q4slots" else "bf16")
        # every layer has the store's experts in an order of its own
        ptrs = [base + (e + 5 * l) % E * nb for e in range(E)]
        if c["store"] == "bf16":
            m.register_host_experts(ptrs, nb, keep=s.store)
        else:
            m.register_host_experts_q4(ptrs, nb, keep=s.store)
        if c["shared"]:
            m.register_shared_experts([s.shared[i].data_ptr() for i in range(c["shared"])], keep=s.shared)
        m.set_router(torch.empty((E, d), device="cuda").normal_(0.0, 0.02, generator=g).to(torch.bfloat16))
        bias = np.stack([gen.router_bias(seed, l, q, c["alpha"], E) for q in range(c["seqs"])])
        m.set_router_bias(torch.from_numpy(bias).cuda(), seq, c["seqs"])
        if c["policy"] != "lru":
            m.set_policy(c["policy"], 0.9)
        m.reserve(T)
        # the experts that each sequence is expected to use are loaded before generation begins
        m.preload_pooled(np.argsort(-bias, axis=1, kind="stable")[:, :c["C"]].astype(np.int32))
        s.layers.append(m)
    x = torch.empty((S, L, T, d), device="cuda").normal_(0.0, 1.0, generator=g).to(torch.bfloat16)
    s.x = x.cpu().pin_memory() if c["host"] else x
    s.out = torch.zeros_like(x)
    s.stats = torch.zeros((S, L, STATS_WORDS), dtype=torch.int32, device="cuda")
    if c["host"]:
        s.out, s.stats = s.out.cpu().pin_memory(), s.stats.cpu().pin_memory()
    xp, op, sp = s.x.data_ptr(), s.out.data_ptr(), s.stats.data_ptr()
    s.calls = []
    for i in range(S):
        for l in range(L):
            j = i * L + l
            call = s.layers[l].forward_host if c["host"] else s.layers[l].forward
            s.calls.append((call, xp + j * T * d * 2, T, op + j * T * d * 2, sp + j * STATS_WORDS * 4))
    torch.cuda.synchronize()
    return s


def _prepare_proxy(c, seed):
    s = _State()
    g = torch.Generator(device="cuda").manual_seed(seed)
    L, T, k, E = c["layers"], c["tokens"], c["k"], c["E"]
    # routing of every layer concentrated on experts of its own, from strongly to hardly
    alphas = np.geomspace(0.1, 10.0, L) if L > 1 else np.array([0.3])
    bias = np.stack([gen.router_bias(seed, l, 0, float(alphas[l]), E) for l in range(L)])
    logits = torch.from_numpy(bias).cuda()[:, None, :] + torch.empty((L, T, E), device="cuda").normal_(0.0, 0.9, generator=g)
    s.trace = torch.topk(logits, k, dim=2).indices.to(torch.int32).contiguous()
    sizes = range(k, E + 1)
    cfg = np.zeros(L * len(sizes), dtype=np.dtype([("layer", "<i4"), ("slots", "<i4"), ("gamma", "<f8")]))
    cfg["layer"], cfg["slots"], cfg["gamma"] = np.repeat(np.arange(L), len(sizes)), np.tile(np.array(sizes), L), c["gamma"]
    s.configs = torch.from_numpy(cfg.view(np.uint8).copy()).cuda()
    s.n = len(cfg)
    s.soft = torch.zeros(s.n, dtype=torch.float64, device="cuda")
    s.hard = torch.zeros(s.n, dtype=torch.int64, device="cuda")
    s.stream = torch.cuda.current_stream().cuda_stream
    s.dims = (L, T, k, E)
    return s


def prepare(case, seed):
    return _prepare_proxy(case, seed) if case["kind"] == "proxy" else _prepare_layers(case, seed)


def run(state):
    if hasattr(state, "trace"):
        M.melinoe_trace_miss_proxies(state.stream, state.trace, *state.dims, state.configs, state.n, state.soft, state.hard)
        return {"soft": state.soft, "hard": state.hard}
    for call, x, T, out, stats in state.calls:
        call(state.stream, x, T, out, stats)
    return {"out": state.out, "stats": state.stats}


def _distinct(c):
    """Distinct experts of one call, on average over some routings of the case's distribution."""
    T, E, k = c["tokens"], c["E"], c["k"]
    if T == 1:
        return float(k)
    r, n = np.random.default_rng(1), []
    for i in range(8):
        bias = np.stack([gen.router_bias(1000 + i, 0, q, c["alpha"], E) for q in range(c["seqs"])])
        logits = bias[np.arange(T) * c["seqs"] // T] + r.normal(0.0, 0.02 * math.sqrt(c["d"]), (T, E))
        n.append(len(np.unique(np.argpartition(-logits, k - 1, axis=1)[:, :k])))
    return float(np.mean(n))


def work(case):
    c = case
    if c["kind"] == "proxy":
        n = c["layers"] * (c["E"] - c["k"] + 1)
        # the trace, configurations and results; three operations per expert and token of a configuration's recurrence
        return {"bytes": c["layers"] * c["tokens"] * c["k"] * 4 + n * 32, "flops": 3.0 * n * c["tokens"] * c["E"]}
    T, d, F = c["tokens"], c["d"], c["F"]
    slot = M.melinoe_moe_expert_bytes_q4(d, F) if c["store"] == "q4slots" else 6 * d * F
    # router, every needed expert once, tokens in and out; six operations per weight triple and token
    call = 2 * c["E"] * d + (_distinct(c) + c["shared"]) * slot + 4 * T * d
    return {"bytes": call * c["layers"] * c["steps"], "flops": 6.0 * d * F * T * (c["k"] + c["shared"]) * c["layers"] * c["steps"]}


def tolerance(case):
    if case["kind"] == "proxy":
        return {"rel": 1e-10, "max": 1e-9}      # fp64 sums; the transfers are whole numbers
    # bf16 hidden activations and outputs (8 significant bits each), fp32 sums between; the statistics are whole numbers
    return {"rel": 1e-2, "max": 5e-2}
