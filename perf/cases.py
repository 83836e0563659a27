"""What this library is asked to do in use, as cases whose time can be measured.

One pass is one call of the library on one batch of prompt caches, the way a serving program makes it: inputs, outputs
and workspace are in hand, the call is `obf_compress` / `evict_only` (device caches) or `obf_compress_host` (caches staged
in pinned host memory).

A case is a dict: layers, kv_heads, q_heads, head_dim, n_obs (observation queries per query head), rank, dtype,
budget_pct / budget (retained positions: a percentage of T, or a number when budget_pct is 0), T (one prompt length, or
several of a ragged batch as text, "1000,4096"), and `mode`:

    obf     headwise selection and Orthogonal BackFill            evict   headwise eviction only
    fast    the back-fill with the three-step subspace iteration  merge   the cache-merging comparison method
    sink    obf with a protected prefix of four positions         early   obf with the span test before the pass over V
    int8    layerwise selection, back-fill and an int8 copy       host    obf on caches in pinned host memory
"""
from __future__ import annotations

import torch

import paper_2604_13349_b200 as P
from paper_2604_13349_b200 import binding as B

MODES = {"obf": 0, "evict": 0, "host": 0, "fast": B.OBF_FLAG_FAST_PATH, "merge": B.OBF_FLAG_MERGE,
         "sink": B.OBF_FLAG_SINK(4), "early": B.OBF_FLAG_EARLY_OUT, "int8": B.OBF_FLAG_LAYERWISE}


def _case(name, layers, kv_heads, q_heads, head_dim, n_obs, T, budget=0, budget_pct=0.0, rank=1, dtype="bf16", mode="obf"):
    c = dict(layers=layers, kv_heads=kv_heads, q_heads=q_heads, head_dim=head_dim, n_obs=n_obs, T=str(T), budget=budget,
             budget_pct=budget_pct, rank=rank, dtype=dtype, mode=mode)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one fp32 layer of two heads, a short prompt (a unit of a test or a toy model)
        _case("tiny_f32", 1, 2, 8, 64, 16, 256, budget=32, dtype="f32"),
        # one layer of a model compressed by itself, as a program does that works layer by layer
        _case("one_layer", 1, 8, 32, 128, 32, 2048, budget=205),
        # the paper's regime: a whole model, relay budget 32, 40 latent steps, every head is back-filled
        _case("paper_1k", 36, 8, 32, 128, 40, 1024, budget=32, rank=2),
        # the same with a longer prompt, rank 4 and the protected prefix of the paper's appendix F
        _case("paper_2k_sink", 36, 8, 32, 128, 40, 2048, budget=32, rank=4, mode="sink"),
        # the paper's own approximation of the subspace (appendix H), a prompt of no round length
        _case("paper_fast", 36, 8, 32, 128, 40, 1187, budget=32, rank=2, mode="fast"),
        # the comparison method of the paper's appendix E on the paper's shape
        _case("paper_merge", 36, 8, 32, 128, 40, 1024, budget=32, rank=2, mode="merge"),
        # eviction alone: a whole model, a fifth of the positions kept
        _case("evict_4k", 36, 8, 32, 128, 32, 4096, budget=819, rank=0, mode="evict"),
        # the largest single cache: 40 layers, 8192 positions, a tenth of them kept
        _case("relay_8k", 40, 8, 32, 128, 32, 8192, budget=811, rank=4),
        # a relay batch: four agents with prompts of different, odd lengths in one call
        _case("relay_batch", 36, 8, 32, 128, 32, "1000,2731,4096,8191", budget_pct=15.0, rank=2),
        # the layerwise selector with the int8 copy of the relay (the paper's smallest relay)
        _case("layerwise_int8", 40, 8, 32, 128, 32, 8192, budget=811, rank=4, mode="int8"),
        # a small model with heads of 64 channels, an odd prompt
        _case("head_dim_64", 16, 8, 32, 64, 32, 3001, budget=32, rank=2),
        # the paper's regime with the caches staged in host memory: copies in, call, copies out
        _case("host_1k", 36, 8, 32, 128, 40, 1024, budget=32, rank=2, mode="host"),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


MOST_ROWS = 40 * 8 * 8192            # key rows of the largest listed case
MOST_ROWS_F32 = 36 * 8 * 1024        # the kernels for fp32 do some 10 times the work per row
MOST_ROWS_HOST = 36 * 8 * 1024       # everything crosses the host link


def draw(rng):
    mode = rng.choice(["obf", "obf", "obf", "obf", "evict", "fast", "merge", "sink", "early", "int8", "host"])
    dtype = "f32" if rng.random() < 0.12 else "bf16"
    head_dim = 64 if rng.random() < 0.25 else 128
    kv_heads = rng.choice([2, 4, 8])
    group = rng.choice([2, 4, 4, 8])
    n_obs = rng.choice([8, 16, 24, 32, 40, 48]) if group < 8 else rng.choice([8, 16, 24, 32])
    most = MOST_ROWS_F32 if dtype == "f32" or mode == "merge" else MOST_ROWS_HOST if mode == "host" else MOST_ROWS
    n = rng.choice([1, 1, 1, 2, 4]) if mode not in ("host", "int8") else 1
    Ts = [_log_int(rng, 150, 8192) for _ in range(n)]
    layers = _log_int(rng, 1, 40)
    while layers > 1 and layers * kv_heads * sum(Ts) > most:
        layers -= 1
    while layers * kv_heads * sum(Ts) > most:
        Ts = [max(150, t // 2) for t in Ts]
    paper = mode in ("fast", "merge", "sink") or (mode != "early" and rng.random() < 0.5)
    return _case("", layers, kv_heads, kv_heads * group, head_dim, n_obs, ",".join(map(str, Ts)),
                 budget=rng.choice([24, 32, 48]) if paper else 0,
                 budget_pct=0.0 if paper else round(rng.uniform(5.0, 25.0), 2),
                 rank=0 if mode == "evict" else rng.choice([1, 2, 4]), dtype=dtype, mode=mode)


def _lengths(case):
    return [int(t) for t in case["T"].split(",")]


def _budget(case, T):
    return max(1, int(round(case["budget_pct"] * T / 100.0))) if case["budget_pct"] else int(case["budget"])


def _kept(case, T):
    return B.k_eff(T, _budget(case, T), MODES[case["mode"]])


def _inputs(case, T, gen):
    """Keys, values and queries of one cache as attention meets them: the queries of a head share a direction; most of the
    positions the budget was chosen for carry keys along it, the first four (the sink) strongly, so that the attention
    mass is spread over orders of magnitude; three channels of the keys are large; the values' channels fall off in scale."""
    L, H, d = case["layers"], case["kv_heads"], case["head_dim"]
    n_q = case["q_heads"] // H * case["n_obs"]
    dev, dt = "cuda", torch.float32 if case["dtype"] == "f32" else torch.bfloat16

    def rnd(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    u = rnd(L, H, 1, d)
    u /= u.norm(dim=-1, keepdim=True)
    q = (rnd(L, H, n_q, d) + 8.0 * (d / 128) ** 0.5 * u).to(dt).reshape(L, case["q_heads"], case["n_obs"], d)
    k = rnd(L, H, T, d)
    big = torch.rand((L, H, d), generator=gen, device=dev).topk(3, dim=-1).indices
    k.mul_(torch.ones((L, H, d), device=dev).scatter_(-1, big, 8.0)[:, :, None, :])
    salient = max(1, min(T, int(0.95 * _kept(case, T))))
    place = torch.rand((L, H, T), generator=gen, device=dev)
    place[..., :4] = 2.0                                             # the sink is among them
    at = place.topk(salient, dim=-1).indices[..., None]
    weight = torch.zeros((L, H, T, 1), device=dev).scatter_(2, at, 8.5)
    weight[:, :, :4] = 14.0
    k = k.addcmul_(weight, u).to(dt)
    order = torch.rand((L, H, d), generator=gen, device=dev).argsort(dim=-1)
    fall = 4.0 / (order + 1.0).sqrt()
    v = rnd(L, H, T, d).mul_(fall[:, :, None, :]).to(dt)
    return k, v, q


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    mode, L, H, d = case["mode"], case["layers"], case["kv_heads"], case["head_dim"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    params = P.make_params(L, H, case["q_heads"], d, case["n_obs"], case["rank"],
                           P.OBF_F32 if case["dtype"] == "f32" else P.OBF_BF16, flags=MODES[mode])
    host = mode == "host"
    place = dict(device="cpu", pin_memory=True) if host else dict(device="cuda")
    caches, outs, keep = [], [], []
    for T in _lengths(case):
        kvq = _inputs(case, T, gen)
        if host:
            kvq = [torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x) for x in kvq]
        ke = _kept(case, T)
        o = {"k": torch.empty((L, H, ke, d), dtype=dt, **place), "v": torch.empty((L, H, ke, d), dtype=dt, **place),
             "idx": torch.empty((L, H, ke), dtype=torch.int32, **place)}
        q8 = None
        if mode == "int8":
            o.update(k8=torch.empty((L, H, ke, d), dtype=torch.int8, **place), v8=torch.empty((L, H, ke, d), dtype=torch.int8, **place),
                     ks=torch.empty((L, H, ke), dtype=torch.float32, **place), vs=torch.empty((L, H, ke), dtype=torch.float32, **place))
            q8 = (o["k8"], o["v8"], o["ks"], o["vs"])
        caches.append(P.make_cache(*kvq, T, _budget(case, T), o["k"], o["v"], o["idx"], q8=q8))
        outs.append(o)
        keep.append(kvq)
    size = P.obf_host_arena_bytes(params, caches) if host else P.obf_workspace_bytes(params, caches)
    work_space = torch.empty(size, dtype=torch.uint8, device="cuda")
    call = P.obf_compress_host if host else P.evict_only if mode == "evict" else P.obf_compress
    return {"call": call, "params": params, "caches": caches, "ws": work_space, "outs": outs, "keep": keep}


def run(state):
    state["call"](state["params"], state["caches"], state["ws"])
    return state["outs"]


def work(case):
    """Bytes: keys and queries read once; values read once where the call streams them, else the kept rows only; compacted
    keys, values and positions (and their int8 copy) written once.  Operations: one contraction of the queries with the
    keys, the Gram matrix of the values where they are streamed, the similarities of the merging method."""
    L, H, d, mode = case["layers"], case["kv_heads"], case["head_dim"], case["mode"]
    e = 4 if case["dtype"] == "f32" else 2
    n_q = case["q_heads"] // H * case["n_obs"]
    heads, nbytes, flops = L * H, 0, 0
    for T in _lengths(case):
        ke = _kept(case, T)
        # the values of a head are not needed where nothing is back-filled: eviction, and `early` with full spans
        streamed = mode not in ("evict",) and not (mode == "early" and ke >= d)
        nbytes += heads * (T * d * e + n_q * d * e + (T if streamed else ke) * d * e + 2 * ke * d * e + 4 * ke)
        flops += heads * 2 * T * n_q * d
        if mode == "merge":
            flops += heads * 2 * T * ke * d
        elif streamed:
            flops += heads * 2 * T * d * d
        if mode == "int8":
            nbytes += heads * 2 * ke * (d + 4)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["mode"] == "evict":
        return "exact"                                     # positions and copies of rows
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3 if case["mode"] != "merge" else 0.5, "differ": 0.0}
    # bf16: values rounded once, so a last place (2^-7 of a value at most) where the fp32 sum lies near a half; an int8 code
    # where such a value lies near a half; merging moves a value to another row where two keys are equally similar
    return {"rel": 4e-3, "max": 2e-2 if case["mode"] != "merge" else 0.5, "differ": 2e-3 if case["mode"] == "int8" else 0.0}
