"""The calls whose time is watched, as a user's program makes them.

Three kinds of work, all through the binding's public functions:

compress   one layer's prefill compression (mkv_compress): prompt keys, values
           and window queries in, retained cache and evicted-set moments out.
generate   `steps` tokens generated from one compressed prompt, through
           `layers` attention layers each (one mkv_decode_step per layer and
           token, which appends the token; every layer evicted back to the
           budget every `evict` tokens, or with evict = 1 by
           mkv_decode_evict_step at every token).  The pass starts from the
           kept compressed prompt (several completions of one prompt, each
           starting from its cache) and is captured once in a CUDA graph, as
           a serving loop keeps it.
call       a single eager call: "decode" (attention over the retained rows and
           the moment term, nothing appended: the token was appended by the
           eviction call before it) or "evict" (append one token to a cache
           that is `over` rows above the budget and evict back to it).

Inputs follow inputs.TorchGenerator's recipes: keys with outlier channels,
log-uniform channel scales or a Gaussian mixture; queries drawn near sums of
keys; everything rounded to bf16.
"""
import math

import torch

from paper_2606_01563_gb300 import inputs, mkv

TAU = 1e-6


def listed():
    return [
        # the smallest prompt: one layer of a small model, 1K tokens; launches and latency count
        {"name": "compress_d64_t1k", "kind": "compress", "batch": 1, "heads": 2, "group": 2, "dim": 64, "T": 1024,
         "budget": 128, "window": 16, "pool": 1, "adaptive": 0, "keys": "outlier"},
        # an ordinary prompt: one Llama-3.1-8B layer, 8K tokens
        {"name": "compress_t8k", "kind": "compress", "batch": 1, "heads": 8, "group": 4, "dim": 128, "T": 8192,
         "budget": 512, "window": 32, "pool": 1, "adaptive": 0, "keys": "logscale"},
        # a batch of long prompts: one Qwen3-4B layer, batch 4, 32K tokens (the most bytes of all)
        {"name": "compress_b4_t32k", "kind": "compress", "batch": 4, "heads": 8, "group": 4, "dim": 128, "T": 32768,
         "budget": 256, "window": 32, "pool": 1, "adaptive": 0, "keys": "logscale"},
        # the longest prompt: one Llama-3.1-8B layer, 128K tokens, two blocks of window rows
        {"name": "compress_t128k", "kind": "compress", "batch": 1, "heads": 8, "group": 4, "dim": 128, "T": 131072,
         "budget": 128, "window": 64, "pool": 1, "adaptive": 0, "keys": "mixture"},
        # a prompt of no round length, chunk pooling, the budget shared by the heads of a batch item
        {"name": "compress_adaptive_t20k", "kind": "compress", "batch": 2, "heads": 8, "group": 4, "dim": 128,
         "T": 20011, "budget": 384, "window": 32, "pool": 4, "adaptive": 1, "keys": "logscale"},
        # the smallest decode call, eager: one layer, one sequence
        {"name": "decode_b1_r512", "kind": "call", "what": "decode", "batch": 1, "heads": 8, "group": 4, "dim": 128,
         "rows": 512, "over": 0, "c": "f32", "order": 1, "ragged": 0},
        # a serving step's decode at a large batch, 16-bit moments, sequences of unequal lengths
        {"name": "decode_b64_r1000_c16", "kind": "call", "what": "decode", "batch": 64, "heads": 8, "group": 4,
         "dim": 128, "rows": 1000, "over": 0, "c": "bf16", "order": 1, "ragged": 1},
        # a model's layer chain: 36 Qwen3-4B layers, batch 4, 8 tokens, C' in operand form
        {"name": "chain_l36_b4_r256", "kind": "generate", "batch": 4, "heads": 8, "group": 4, "dim": 128, "rows": 256,
         "layers": 36, "steps": 8, "evict": 0, "c": "split", "ragged": 0},
        # the same chain for a larger batch: fewer layers, fp32 moments
        {"name": "chain_l8_b32_r512", "kind": "generate", "batch": 32, "heads": 8, "group": 4, "dim": 128,
         "rows": 512, "layers": 8, "steps": 4, "evict": 0, "c": "f32", "ragged": 0},
        # long-context serving with periodic eviction: Llama-3.1-8B layers, budget 128, every 64 tokens
        {"name": "chain_l8_b1_r128_evict64", "kind": "generate", "batch": 1, "heads": 8, "group": 4, "dim": 128,
         "rows": 128, "layers": 8, "steps": 64, "evict": 64, "c": "split", "ragged": 0},
        # continuous eviction: one row leaves for every token (Algorithm 1 at every step)
        {"name": "continuous_b1_r512", "kind": "generate", "batch": 1, "heads": 8, "group": 4, "dim": 128,
         "rows": 512, "layers": 1, "steps": 32, "evict": 1, "c": "f32", "ragged": 0},
        # periodic eviction of a large cache: 64 rows out of 4160
        {"name": "evict_b1_r4096", "kind": "call", "what": "evict", "batch": 1, "heads": 8, "group": 4, "dim": 128,
         "rows": 4096, "over": 63, "c": "f32", "order": 1, "ragged": 0},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _geometry(rng):
    """(heads, group, dim): mostly the 8B-class geometry, else another built one."""
    if rng.random() < 0.5:
        return 8, 4, 128
    return rng.choice([2, 4, 5, 8, 16]), rng.choice([1, 2, 4, 8]), rng.choice([64, 128])


def draw(rng):
    heads, group, dim = _geometry(rng)
    kind = rng.choice(["compress", "compress", "decode", "chain", "evict_chain", "continuous", "evict"])
    if kind == "compress":
        batch = rng.choice([1, 1, 2, 3, 4])
        T = _logint(rng, 700, min(131072, 4 * 8 * 32768 // (batch * heads)))
        window = rng.choice([w for w in (8, 16, 32, 64) if w * group <= 256])
        budget = max(window + 8, min(T // 4, _logint(rng, 64, 1024)))
        return {"kind": "compress", "batch": batch, "heads": heads, "group": group, "dim": dim, "T": T,
                "budget": budget, "window": window, "pool": rng.choice([1, 1, 4]), "adaptive": rng.choice([0, 0, 1]),
                "keys": rng.choice(["outlier", "logscale", "mixture"])}
    if kind == "decode":
        batch = _logint(rng, 1, 64)
        return {"kind": "call", "what": "decode", "batch": batch, "heads": heads, "group": group, "dim": dim,
                "rows": _logint(rng, 64, max(64, min(4096, 64 * 8 * 1000 // (batch * heads)))), "over": 0,
                "c": rng.choice(["f32", "bf16", "split"]), "order": rng.choice([1, 1, 1, 0]),
                "ragged": rng.choice([0, 1])}
    if kind == "chain":
        batch = _logint(rng, 1, 32)
        return {"kind": "generate", "batch": batch, "heads": heads, "group": group, "dim": dim,
                "rows": _logint(rng, 100, max(100, min(2048, 32 * 8 * 512 // (batch * heads)))),
                "layers": rng.randint(2, 8), "steps": rng.randint(1, 4), "evict": 0,
                "c": rng.choice(["f32", "bf16", "split"]), "ragged": rng.choice([0, 1])}
    if kind == "evict_chain":
        evict = rng.choice([16, 32, 64])
        return {"kind": "generate", "batch": 1, "heads": heads, "group": group, "dim": dim,
                "rows": _logint(rng, 100, 1000), "layers": rng.randint(1, 4), "steps": evict, "evict": evict,
                "c": rng.choice(["f32", "split"]), "ragged": 0}
    if kind == "continuous":
        return {"kind": "generate", "batch": rng.choice([1, 2]), "heads": heads, "group": group, "dim": dim,
                "rows": _logint(rng, 100, 1000), "layers": 1, "steps": rng.randint(4, 32), "evict": 1, "c": "f32",
                "ragged": 0}
    return {"kind": "call", "what": "evict", "batch": 1, "heads": min(heads, 8), "group": group, "dim": dim,
            "rows": _logint(rng, 200, 4096), "over": rng.choice([0, 15, 31, 63]), "c": "f32", "order": 1, "ragged": 0}


# ------------------------------------------------------------------ inputs
def _compress_params(c):
    return mkv.mkv_compress_params(c["budget"], c["window"], 1, 1, c["pool"], 1, 1, TAU, c["adaptive"])


def _capacity(c):
    """Rows of the cache a compress writes: the budget, or with the shared budget the most one head can keep."""
    if not c["adaptive"]:
        return min(c["T"], c["budget"])
    protected = 1 + c["window"]
    return min(c["T"], c["heads"] * (c["budget"] - protected) + protected)


def _prompt(c, seed):
    wl = inputs.Workload("prompt", inputs.Geometry(c["batch"], c["heads"], c["group"], c["dim"]), c["T"], c["budget"],
                         c["window"], c["keys"])
    return inputs.TorchGenerator(wl, seed=seed, device="cuda").prefill()


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1000003 + 29)
    return gen


def _near(gen, keys, n):
    """n queries per unit near sums of three of its keys (norm sqrt(d), noise 0.3): [units, n, d] float32."""
    units, rows, d = keys.shape
    pick = torch.randint(0, rows, (units, n, 3), generator=gen, device="cuda")
    v = keys[torch.arange(units, device="cuda")[:, None, None], pick].float().sum(2)
    v = math.sqrt(d) * v / torch.linalg.norm(v, dim=-1, keepdim=True)
    return v + 0.3 * torch.randn(v.shape, generator=gen, device="cuda")


EVICTED = 1024  # tokens behind the moments of a generated state


def _layer(c, gen, steps, rows, cap):
    """One layer's compressed prompt (rows, moments of EVICTED more tokens) and the coming tokens."""
    b, h, g, d = c["batch"], c["heads"], c["group"], c["dim"]
    units = b * h
    lo, hi = math.log(0.5), math.log(4.0)
    scale = torch.exp(lo + (hi - lo) * torch.rand(units, 1, d, generator=gen, device="cuda"))

    def keys(n):
        return (torch.randn(units, n, d, generator=gen, device="cuda") * scale).to(torch.bfloat16)

    def values(n):
        return torch.randn(units, n, d, generator=gen, device="cuda").to(torch.bfloat16)

    ke, ve = keys(EVICTED).float(), values(EVICTED).float()
    mk, mv = ke.mean(1), ve.mean(1)
    cov = torch.bmm((ve - mv[:, None]).transpose(1, 2), ke - mk[:, None]) / EVICTED
    st = {"K": torch.zeros(units, cap, d, dtype=torch.bfloat16, device="cuda")}
    st["V"] = torch.zeros_like(st["K"])
    st["K"][:, :rows] = keys(rows)
    st["V"][:, :rows] = values(rows)
    st["pos"] = torch.zeros(units, cap, dtype=torch.int32, device="cuda")
    st["pos"][:, :rows] = torch.arange(rows, dtype=torch.int32, device="cuda")
    st["len"] = torch.full((units,), rows, dtype=torch.int32, device="cuda")
    if c["ragged"]:
        st["len"] = torch.randint(max(1, rows // 2), rows + 1, (units,), generator=gen, device="cuda", dtype=torch.int32)
    st["seen"] = torch.full((units,), rows + EVICTED, dtype=torch.int32, device="cuda")
    st["n"] = torch.full((units,), EVICTED, dtype=torch.int32, device="cuda")
    st["mu_k"], st["mu_v"], st["C"] = mk, mv, cov
    st["q"] = _near(gen, st["K"][:, :rows], steps * g).view(units, steps, g, d).transpose(0, 1).to(torch.bfloat16)
    st["kn"] = keys(steps).transpose(0, 1)
    st["vn"] = values(steps).transpose(0, 1)
    return {k: v.contiguous() for k, v in st.items()}


CACHE, MOMENTS = ("K", "V", "pos", "len", "seen"), ("n", "mu_k", "mu_v", "C")
BF16, F32, I32 = torch.bfloat16, torch.float32, torch.int32


def _shape(c, cap):
    b, h, d = c["batch"], c["heads"], c["dim"]
    return {"K": (b, h, cap, d), "V": (b, h, cap, d), "pos": (b, h, cap), "n": (b, h), "mu_k": (b, h, d),
            "mu_v": (b, h, d), "C": (b, h, d, d), "packed": (b, h, d, d), "len": (b, h), "seen": (b, h),
            "y_len": (b, h)}


class _Prompt:
    """The caches and moments of a compressed prompt's layers, in one device
    buffer, and a saved copy of it that a new completion starts from."""

    def __init__(self, c, layers, cap, evicts):
        self.g = mkv.geom(c["batch"], c["heads"], c["group"], c["dim"])
        kinds = {"K": BF16, "V": BF16, "pos": I32, "n": I32, "mu_k": F32, "mu_v": F32, "C": F32}
        if c["c"] != "f32":
            kinds["packed"] = BF16 if c["c"] == "bf16" else I32
        kinds.update({"len": I32, "seen": I32, "y_len": I32})  # last: all that a completion without evictions changes
        shapes, at, size = _shape(c, cap), {}, 0
        for name, dtype in kinds.items():
            if name == "len":
                tail = size
            for l in range(len(layers)):
                at[name, l] = size
                size += -(-math.prod(shapes[name]) * dtype.itemsize // 256) * 256
        slab = torch.zeros(size, dtype=torch.uint8, device="cuda")

        def view(name, l):
            n = math.prod(shapes[name]) * kinds[name].itemsize
            return slab[at[name, l]:at[name, l] + n].view(kinds[name]).view(shapes[name])

        self.layers = []
        for l, layer in enumerate(layers):
            t = {name: view(name, l) for name in kinds}
            for name in CACHE + MOMENTS:
                t[name].copy_(layer[name].view(shapes[name]))
            y = torch.zeros(shapes["K"], dtype=F32, device="cuda") if evicts else None
            cache = mkv.Cache(t["K"], t["V"], t["pos"], t["len"], t["seen"], y, t["y_len"] if evicts else None)
            mom = mkv.Moments(t["n"], t["mu_k"], t["mu_v"], t["C"])
            packed = t.get("packed")
            self.layers.append((cache, mom, packed))
            if c["c"] == "bf16":
                mkv.mkv_moments_pack_bf16(self.g, mom, packed)
            elif c["c"] == "split":
                mkv.mkv_moments_pack_split(self.g, mom, TAU, packed)
        self.live = slab if evicts or "over" in c else slab[tail:]
        self.saved = self.live.clone()

    def restart(self):
        self.live.copy_(self.saved)

    def params(self, c, l, early):
        """Decode parameters that read layer l's C in the form the case names."""
        packed = self.layers[l][2]
        ptr = None if packed is None else packed.data_ptr()
        return mkv.mkv_decode_params(1, c.get("order", 1), TAU, ptr if c["c"] == "bf16" else None, early,
                                     ptr if c["c"] == "split" else None)


def _generate_state(c, seed):
    gen = _generator(seed)
    rows, steps, evict = c["rows"], c["steps"], c["evict"]
    cap = rows + (evict if evict else steps)
    b, h, gr, d = c["batch"], c["heads"], c["group"], c["dim"]
    layers = [_layer(c, gen, steps, rows, cap) for _ in range(c["layers"])]
    prompt = _Prompt(c, layers, cap, bool(evict))
    g = prompt.g
    outs = torch.empty(steps, c["layers"], b, h * gr, d, device="cuda")
    early = 1 if c["layers"] > 1 else 0  # the kernel before a layer's launch is another layer's
    params = [prompt.params(c, l, early) for l in range(c["layers"])]
    if evict == 1:
        ws, ws_e = mkv.alloc_workspace(mkv.mkv_decode_evict_workspace_size(g, cap)), None
    else:
        ws = mkv.alloc_workspace(mkv.mkv_decode_workspace_size(g, cap))
        ws_e = mkv.alloc_workspace(mkv.mkv_evict_workspace_size(g, cap)) if evict else None
    q = [[lay["q"][s].reshape(b, h * gr, d) for lay in layers] for s in range(steps)]
    kn = [[lay["kn"][s].view(b, h, d) for lay in layers] for s in range(steps)]
    vn = [[lay["vn"][s].view(b, h, d) for lay in layers] for s in range(steps)]

    def tokens():
        prompt.restart()
        for s in range(steps):
            for l, (cache, mom, _) in enumerate(prompt.layers):
                if evict == 1:
                    mkv.mkv_decode_evict_step(g, q[s][l], kn[s][l], vn[s][l], rows, cache, mom, params[l], outs[s, l],
                                              None, ws)
                else:
                    mkv.mkv_decode_step(g, q[s][l], kn[s][l], vn[s][l], cache, mom, params[l], outs[s, l], None, ws)
            if evict > 1 and (s + 1) % evict == 0:
                for l, (cache, mom, packed) in enumerate(prompt.layers):
                    mkv.mkv_evict_append(g, q[s][l], None, None, rows, cache, mom, TAU, ws_e)
                    if packed is not None:
                        mkv.mkv_moments_pack_split(g, mom, TAU, packed)

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        tokens()
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        tokens()
    # the graph reads the queries, tokens and workspaces: they live as long as it
    return {"case": c, "graph": graph, "prompt": prompt, "outs": outs, "held": (q, kn, vn, ws, ws_e)}


def _call_layer(c, seed):
    cap = c["rows"] + c["over"] + 1
    return _layer(c, _generator(seed), 1, c["rows"] + c["over"], cap), cap


def prepare(case, seed):
    c = case
    if c["kind"] == "generate":
        return _generate_state(c, seed)
    if c["kind"] == "compress":
        g = mkv.geom(c["batch"], c["heads"], c["group"], c["dim"])
        K, V, Q = _prompt(c, seed)
        p = _compress_params(c)
        return {"case": c, "g": g, "K": K, "V": V, "Q": Q, "p": p, "cache": mkv.alloc_cache(g, _capacity(c)),
                "mom": mkv.alloc_moments(g),
                "ws": mkv.alloc_workspace(mkv.mkv_compress_workspace_size(g, c["T"], p))}
    lay, cap = _call_layer(c, seed)
    prompt = _Prompt(c, [lay], cap, False)
    g, (cache, mom, _) = prompt.g, prompt.layers[0]
    b, h, gr, d = c["batch"], c["heads"], c["group"], c["dim"]
    s = {"case": c, "g": g, "prompt": prompt, "cache": cache, "mom": mom, "q": lay["q"][0].reshape(b, h * gr, d)}
    if c["what"] == "evict":
        s["kn"], s["vn"] = lay["kn"][0].view(b, h, d), lay["vn"][0].view(b, h, d)
        s["ws"] = mkv.alloc_workspace(mkv.mkv_evict_workspace_size(g, cap))
    else:
        s["p"] = prompt.params(c, 0, 0)
        s["ws"] = mkv.alloc_workspace(mkv.mkv_decode_workspace_size(g, cap))
        s["out"] = torch.empty(b, h * gr, d, device="cuda")
        s["lse"] = torch.empty(b, h * gr, device="cuda")
    return s


def _state_out(cache, mom, rows=None):
    """A cache's rows in use (all of them, or the first `rows`) and the moments."""
    out = {n: getattr(cache, n)[:, :, :rows] for n in ("K", "V", "pos")}
    return {**out, "len": cache.len, "seen": cache.seen, **{n: getattr(mom, n) for n in MOMENTS}}


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "generate":
        s["graph"].replay()
        layers = s["prompt"].layers[:4]
        if not c["evict"]:  # the appended rows are the inputs themselves
            return {"outs": s["outs"], "len": [cache.len for cache, _, _ in layers]}
        return {"outs": s["outs"], "layers": [_state_out(cache, mom, c["rows"]) for cache, mom, _ in layers]}
    if c["kind"] == "compress":
        mkv.mkv_compress(s["g"], c["T"], s["K"], s["V"], s["Q"], s["p"], s["cache"], s["mom"], s["ws"])
        return _state_out(s["cache"], s["mom"])
    if c["what"] == "decode":
        mkv.mkv_decode_step(s["g"], s["q"], None, None, s["cache"], s["mom"], s["p"], s["out"], s["lse"], s["ws"])
        return {"out": s["out"], "lse": s["lse"]}
    s["prompt"].restart()  # the cache as the decode steps before left it
    mkv.mkv_evict_append(s["g"], s["q"], s["kn"], s["vn"], c["rows"], s["cache"], s["mom"], TAU, s["ws"])
    return _state_out(s["cache"], s["mom"], c["rows"])


# ------------------------------------------------------------ work, tolerance
def work(case):
    c = case
    units, g, d = c["batch"] * c["heads"], c["group"], c["dim"]
    moments = (d * d + 2 * d + 1) * 4
    if c["kind"] == "compress":
        T, w, kept = c["T"], c["window"], c["budget"]
        return {"bytes": units * (4 * T * d + 2 * g * w * d + kept * (4 * d + 4) + moments),
                "flops": units * (2 * g * w * T * d + 4 * T * d * d)}

    def decode(rows, append):  # one layer's step
        c_bytes = 2 if c["c"] == "bf16" else 4
        if c.get("order", 1) == 0:
            c_bytes = 0
        by = rows * 4 * d + d * d * c_bytes + 2 * d * 4 + 4 + g * d * 6 + (8 * d if append else 0)
        return units * by, units * (4 * g * rows * d + 2 * g * d * d)

    def evict(rows, n):  # from `rows` rows, n evicted: every row read, moments updated, the evicted rows taken out
        return units * (rows * 4 * d + 2 * moments + n * 4 * d), units * (2 * rows * d * d + n * (rows * 6 * d + 2 * d * d))

    mean_rows = int(c["rows"] * (0.75 if c["ragged"] else 1))
    if c["kind"] == "call":
        by, fl = decode(mean_rows, False) if c["what"] == "decode" else evict(c["rows"] + c["over"] + 1, c["over"] + 1)
        return {"bytes": by, "flops": fl}
    by = fl = 0
    held = mean_rows
    for s in range(c["steps"]):
        x = decode(held, True)
        by, fl = by + x[0] * c["layers"], fl + x[1] * c["layers"]
        held += 1
        if c["evict"] and (s + 1) % c["evict"] == 0:
            x = evict(held, c["evict"])
            by, fl = by + x[0] * c["layers"], fl + x[1] * c["layers"]
            held -= c["evict"]
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times the distance seen from the 64-bit results: C of a long
    prompt's evicted set is a difference of 32-bit sums over its tokens (9e-6
    at 32K); decode outputs and the moments of an eviction stay near 1e-6
    (bf16 hi + lo products, 32-bit sums).  Retained rows are copies and
    positions and counts whole numbers: the same."""
    return {"rel": 4e-5 if case["kind"] == "compress" else 5e-6}


# -------------------------------------------------------------- 64-bit results
def _exact_select(scores, protected, k):
    """Ascending indices of the protected entries and the k highest others (ties: the lower index)."""
    s = scores.clone()
    s[protected] = -math.inf
    order = torch.sort(s, descending=True, stable=True).indices[:k]
    keep = protected.clone()
    keep[order] = True
    return torch.nonzero(keep)[:, 0]


def _exact_moments(K, V):
    mk, mv = K.mean(0), V.mean(0)
    return mk, mv, (V - mv).T @ (K - mk) / K.shape[0]


def _exact_compress(c, seed):
    K, V, Q = _prompt(c, seed)
    b, h, g, d, T, w = c["batch"], c["heads"], c["group"], c["dim"], c["T"], c["window"]
    cap, scale = _capacity(c), c["dim"] ** -0.5
    t = torch.arange(T, device="cuda")
    protected = (t < 1) | (t >= T - w)
    n_free = c["budget"] - int(protected.sum())

    def scores(bi, hi):
        k = K[bi, hi].double()
        x = Q[bi, hi].double().reshape(g * w, d) @ k.T * scale
        last = (T - w + torch.arange(w, device="cuda")).repeat(g)
        x.masked_fill_(t[None, :] > last[:, None], -math.inf)
        s = torch.softmax(x, -1).sum(0)
        if c["pool"] > 1:
            pad = -T % c["pool"]
            s = torch.nn.functional.pad(s, (0, pad)).view(-1, c["pool"]).sum(1).repeat_interleave(c["pool"])[:T]
        return s

    def rest(bi, hi, kept):
        out = torch.ones(T, dtype=torch.bool, device="cuda")
        out[kept] = False
        return _exact_moments(K[bi, hi].double()[out], V[bi, hi].double()[out])

    def residual(bi, hi, s, kept):
        mk, mv, C = rest(bi, hi, kept)
        C = torch.where((C * (T - len(kept))).abs() < TAU, torch.zeros_like(C), C)
        return s * torch.linalg.norm(V[bi, hi].double() - mv - scale * (K[bi, hi].double() @ C.T), dim=-1)

    def select(per_head):  # the heads' scores of one batch item -> the rows each keeps
        if not c["adaptive"]:
            return [_exact_select(s, protected, n_free) for s in per_head]
        f = _exact_select(torch.cat(per_head), protected.repeat(h), h * n_free)
        return [f[(f >= i * T) & (f < (i + 1) * T)] - i * T for i in range(h)]

    o = {"K": torch.zeros(b, h, cap, d, dtype=torch.float64, device="cuda")}
    o["V"] = torch.zeros_like(o["K"])
    o["pos"] = torch.zeros(b, h, cap, dtype=torch.int32, device="cuda")
    o["len"] = torch.zeros(b, h, dtype=torch.int32, device="cuda")
    o["seen"] = torch.full_like(o["len"], T)
    o["n"] = torch.zeros_like(o["len"])
    o["mu_k"] = torch.zeros(b, h, d, dtype=torch.float64, device="cuda")
    o["mu_v"], o["C"] = torch.zeros_like(o["mu_k"]), torch.zeros(b, h, d, d, dtype=torch.float64, device="cuda")
    for bi in range(b):
        s = [scores(bi, hi) for hi in range(h)]
        first = select(s)
        kept = select([residual(bi, hi, s[hi], first[hi]) for hi in range(h)])
        for hi, r in enumerate(kept):
            o["K"][bi, hi, :len(r)], o["V"][bi, hi, :len(r)] = K[bi, hi][r].double(), V[bi, hi][r].double()
            o["pos"][bi, hi, :len(r)] = r.int()
            o["len"][bi, hi], o["n"][bi, hi] = len(r), T - len(r)
            o["mu_k"][bi, hi], o["mu_v"][bi, hi], o["C"][bi, hi] = rest(bi, hi, r)
    return o


class _Exact:
    """One layer's cache and moments in 64 bits; every unit at once."""

    def __init__(self, c, layer):
        self.c, self.scale = c, c["dim"] ** -0.5
        self.K, self.V = layer["K"].double(), layer["V"].double()
        self.pos, self.len, self.seen = layer["pos"].clone(), layer["len"].long(), layer["seen"].clone()
        self.n = layer["n"].clone()
        self.mk, self.mv, self.C = layer["mu_k"].double(), layer["mu_v"].double(), layer["C"].double()
        self.u = torch.arange(self.K.shape[0], device="cuda")
        self.C_read = self.C.float().to(torch.bfloat16).double() if c["c"] == "bf16" else None

    def clamped(self, C):
        return torch.where((C * self.n[:, None, None]).abs() < TAU, torch.zeros_like(C), C)

    def append(self, kn, vn):
        self.K[self.u, self.len], self.V[self.u, self.len] = kn.double(), vn.double()
        self.pos[self.u, self.len] = self.seen
        self.seen += 1
        self.len += 1

    def logits(self, q):  # [units, g, cap], rows past the length at -inf
        x = torch.bmm(q.double(), self.K.transpose(1, 2)) * self.scale
        dead = torch.arange(self.K.shape[1], device="cuda")[None, :] >= self.len[:, None]
        return x.masked_fill(dead[:, None, :], -math.inf)

    def decode(self, q):
        x = self.logits(q)
        zr = torch.logsumexp(x, -1)
        o = torch.bmm(torch.softmax(x, -1), self.V)
        ze = torch.log(self.n.double())[:, None] + self.scale * torch.bmm(q.double(), self.mk[:, :, None])[:, :, 0]
        f = self.mv[:, None, :].expand_as(o)
        if self.c.get("order", 1):
            C = self.clamped(self.C if self.C_read is None else self.C_read)
            f = f + self.scale * torch.bmm(q.double(), C.transpose(1, 2))
        z = torch.logaddexp(zr, ze)
        return torch.exp(zr - z)[..., None] * o + torch.exp(ze - z)[..., None] * f, z

    def evict(self, q, budget):
        live = torch.arange(self.K.shape[1], device="cuda")[None, :] < self.len[:, None]
        x = self.logits(q)
        for _ in range(int(self.len[0]) - budget):  # every unit holds as many rows
            alpha = torch.softmax(x, -1).sum(1)
            r = self.V - self.mv[:, None] - self.scale * torch.bmm(self.K, self.clamped(self.C).transpose(1, 2))
            score = (alpha * torch.linalg.norm(r, dim=-1)).masked_fill(~live, math.inf)
            j = score.argmin(-1)
            k, v, n = self.K[self.u, j], self.V[self.u, j], self.n.double()[:, None]
            dk = k - self.mk
            self.mk = self.mk + dk / (n + 1)
            dv = v - self.mv
            self.mv = self.mv + dv / (n + 1)
            n3 = n[..., None]
            self.C = (n3 * self.C + (v - self.mv)[:, :, None] * dk[:, None, :]) / (n3 + 1)
            self.n += 1
            live[self.u, j] = False
            x = x.masked_fill(~live[:, None, :], -math.inf)
        order = torch.sort((~live).int(), stable=True).indices[:, :budget]  # survivors, in order
        for name in ("K", "V", "pos"):
            a = getattr(self, name)
            a[:, :budget] = a[self.u[:, None], order]
        self.len = torch.full_like(self.len, budget)

    def state(self):
        rows, shapes = int(self.len[0]), _shape(self.c, int(self.len[0]))
        s = {"K": self.K[:, :rows], "V": self.V[:, :rows], "pos": self.pos[:, :rows], "len": self.len.int(),
             "seen": self.seen, "n": self.n, "mu_k": self.mk, "mu_v": self.mv, "C": self.C}
        return {k: v.reshape(shapes[k]) for k, v in s.items()}


def _exact_generate(c, seed):
    gen = _generator(seed)
    rows, steps, evict = c["rows"], c["steps"], c["evict"]
    cap = rows + (evict if evict else steps)
    outs, states = [], []
    for _ in range(c["layers"]):
        lay = _layer(c, gen, steps, rows, cap)
        x = _Exact(c, lay)
        per = []
        for s in range(steps):
            x.append(lay["kn"][s], lay["vn"][s])
            if evict == 1:
                x.evict(lay["q"][s], rows)
            per.append(x.decode(lay["q"][s])[0].reshape(c["batch"], c["heads"] * c["group"], c["dim"]))
            if evict > 1 and (s + 1) % evict == 0:
                x.evict(lay["q"][s], rows)
        outs.append(torch.stack(per))
        states.append(x)
    o = {"outs": torch.stack(outs, 1)}
    if not evict:
        return dict(o, len=[x.len.int().view(c["batch"], c["heads"]) for x in states][:4])
    return dict(o, layers=[x.state() for x in states][:4])


def exact(case, seed):
    c = case
    if c["kind"] == "compress":
        return _exact_compress(c, seed)
    if c["kind"] == "generate":
        return _exact_generate(c, seed)
    lay, _ = _call_layer(c, seed)
    x = _Exact(c, lay)
    if c["what"] == "decode":
        out, lse = x.decode(lay["q"][0])
        shape = (c["batch"], c["heads"] * c["group"])
        return {"out": out.reshape(*shape, c["dim"]), "lse": lse.reshape(shape)}
    x.append(lay["kn"][0], lay["vn"][0])
    x.evict(lay["q"][0], c["rows"])
    return x.state()
