"""The work that programs have this library do, as cases that can be timed and compared.

A case is one shape of one kind of call; `run` makes one pass of it through the public entry points:

  step     one decode step of a layer stack with ra_decode_step (stacked inputs)
  layers   the same step as a model makes it: ra_decode_layer for layers 0 .. L - 1
  calls    the same step in separate calls per layer: ra_append_kv, ra_evict, ra_decode_attn
  prefill  the prompt rows of every layer (ra_prefill), each followed by the attention of the last
           prompt token over them (ra_decode_attn)
  admit    a finished slot of a running batch takes a new request (ra_set_active, ra_admit), then
           the batch makes a decode step
  resume   a run is loaded from a checkpoint, layer by layer (ra_restore, and under the scored
           policy ra_restore_queries), then makes a decode step (ra_decode_layer)

Decoding starts at steady state: a sequence holds its prompt, K random older tokens, the buffer of r
and the `phase` tokens since its last eviction.  Phases are spread over [0, r), as requests that
joined a continuous batch at different times, and sequence 0 evicts in the first pass.  Each pass
appends a token, so the passes on one state are the successive steps of one generation.

Rows are normal, keys with a log-normal scale per channel (as trained keys have a few large
channels): attention is spread over many rows with some heavier ones.  Everything a case fixes
(lengths, phases) follows from the case alone, every value from the seed.
"""
import math
import random

import torch

import paper_2609_03430_gb300 as ra

D = 128
RING = 4  # decode inputs cycled from step to step
POLICY = {"random": ra.RA_POLICY_RANDOM, "shared": ra.RA_POLICY_SHARED, "recency": ra.RA_POLICY_RECENCY,
          "block": ra.RA_POLICY_BLOCK, "scored": ra.RA_POLICY_SNAPKV}
LAYOUT = {"ordered": ra.RA_COMPACT_ORDERED, "free": ra.RA_COMPACT_HOLEFILL}


def _case(name, kind, L, B, KVH, G, lp, K, r=64, policy="random", layout="ordered", block=1):
    lo, hi = lp if isinstance(lp, tuple) else (lp, lp)
    return dict(name=name, kind=kind, layers=L, batch=B, kv_heads=KVH, group=G, prompt_lo=lo, prompt_hi=hi, budget=K,
                buffer=r, policy=policy, layout=layout, block=block)


def listed():
    return [
        # the smallest call: one layer, one sequence, a short cache (launch latency)
        _case("tiny layer", "layers", 1, 1, 8, 4, 128, 256),
        # one interactive user of a small model (Qwen3-4B shape), as the model calls it layer by layer
        _case("single user layers", "layers", 36, 1, 8, 4, 512, 2048),
        # the same through the stacked call, a 32B-shape stack and a small budget
        _case("single user step", "step", 64, 1, 8, 8, 1000, 1024),
        # a batch of a small model (Qwen3-4B shape), all its layers, both call forms
        _case("4b batch 16 step", "step", 36, 16, 8, 4, 512, 2048),
        _case("4b batch 16 layers", "layers", 36, 16, 8, 4, 512, 2048, layout="free"),
        # a large batch (Qwen3-14B shape) called layer by layer
        _case("14b batch 64 layers", "layers", 8, 64, 8, 5, 2048, 4096),
        # long caches, eight query heads per KV head (Qwen3-32B shape): the largest
        _case("32b batch 32 step", "step", 16, 32, 8, 8, 1024, 8192),
        # ragged prompts (Phi-4 shape) under the scored comparator
        _case("phi ragged scored", "layers", 6, 48, 10, 4, (256, 4096), 4096, policy="scored"),
        # an engine with its own loop over separate calls; block draws, sizes that fill no tile
        _case("separate calls", "calls", 4, 13, 8, 4, (77, 1500), 1000, r=32, policy="block", block=16),
        # prompts of a new batch
        _case("prefill batch 8", "prefill", 8, 8, 8, 4, (512, 4096), 2048),
        # a request enters a running batch
        _case("admit into batch 8", "admit", 36, 8, 8, 4, (300, 2048), 1024),
        # a run of the scored comparator resumed from a checkpoint
        _case("resume scored", "resume", 2, 16, 10, 4, (256, 2048), 2048, policy="scored"),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.99)))))))


# the largest listed pass of each kind: a drawn one costs no more
_MOST_BYTES = {"step": 18e9, "layers": 12e9, "calls": 1.5e9, "prefill": 0.8e9, "admit": 0.8e9, "resume": 1.2e9}


def draw(rng):
    kind = rng.choice(["step", "step", "layers", "layers", "layers", "calls", "prefill", "admit", "resume"])
    while True:
        KVH, G = rng.choice([(8, 4), (8, 5), (8, 8), (10, 4), (4, 7), (2, 8), (16, 1), (5, 3), (8, 2), (1, 6)])
        L = _log_uniform(rng, 1, 8 if kind in ("calls", "prefill", "resume") else 40)
        B = _log_uniform(rng, 1, 16 if kind in ("calls", "prefill", "admit", "resume") else 64)
        hi = _log_uniform(rng, 64, 4096)
        lo = hi if rng.random() < 0.4 else max(1, hi // rng.randint(2, 12))
        K = _log_uniform(rng, 128, 8192)
        r = rng.choice([16, 32, 64, 64, 64, 100, 128])
        policy = rng.choice(["random", "random", "random", "random", "shared", "recency", "block", "scored"])
        layout = rng.choice(["ordered", "ordered", "free"]) if policy != "scored" else "ordered"
        if kind == "resume":
            policy, layout = rng.choice([("scored", "ordered"), ("random", "ordered"), ("random", "free")])
        if policy == "scored" and r * G > 512:
            r = 32
        if kind == "admit":
            B = max(B, 2)
        c = _case("", kind, L, B, KVH, G, (lo, hi), K, r, policy, layout, rng.choice([8, 16, 64]))
        del c["name"]
        w = work(c)
        if w["bytes"] <= _MOST_BYTES[kind] and w["flops"] / 50 <= _MOST_BYTES[kind]:
            return c


# ------------------------------------------------------------------------------ shapes and inputs
def _prompts(c):
    rng = random.Random("%(batch)d %(prompt_lo)d %(prompt_hi)d" % c)
    return [rng.randint(c["prompt_lo"], c["prompt_hi"]) for _ in range(c["batch"])]


def _start(c):
    """(generated, cached) of every sequence: at a steady state, or nothing yet."""
    B, K, r = c["batch"], c["budget"], c["buffer"]
    if c["kind"] in ("prefill", "admit"):
        return [0] * B, [0] * B
    phases = [r - 1 - (b * r) // B for b in range(B)]
    base = -(-(2 * K + 4 * r) // r) * r
    return [base + 3 * r * (b % 5) + phases[b] for b in range(B)], [K + r + p for p in phases]


def _admitted(c):
    """Prompt lengths of the requests that enter, cycled."""
    return [c["prompt_hi"], (c["prompt_lo"] + c["prompt_hi"]) // 2 | 1, c["prompt_lo"]]


def _gen(seed, *tags):
    x = seed & 0xFFFFFFFF
    for t in tags:
        x = (x * 1000003 + t + 7) % (1 << 61)
    return torch.Generator("cuda").manual_seed(x)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)


def _key_scale(c, seed, l):
    g = _gen(seed, 1, l)
    return torch.exp(0.5 * torch.randn(c["kv_heads"], 1, D, generator=g, device="cuda"))


def _scaled(k, sc):
    return k.mul_(sc.to(torch.bfloat16))


def _prompt_rows(c, seed, l):
    g = _gen(seed, 2, l)
    shape = (c["batch"], c["kv_heads"], max(1, max(_prompts(c))), D)
    return _scaled(_randn(g, *shape), _key_scale(c, seed, l)), _randn(g, *shape)


def _cached_rows(c, seed, l, lp, g0, c0):
    """Rows and positions of the generated tokens held by each head of layer l: K at random places, then the newest."""
    g = _gen(seed, 3, l)
    B, KVH, K = c["batch"], c["kv_heads"], c["budget"]
    n = max(c0)
    k, v = _scaled(_randn(g, B, KVH, n, D), _key_scale(c, seed, l)), _randn(g, B, KVH, n, D)
    dev = "cuda"
    g0, c0, lp = (torch.tensor(x, device=dev, dtype=torch.float64)[:, None, None] for x in (g0, c0, lp))
    i = torch.arange(n, device=dev, dtype=torch.float64)
    jitter = 0.5 * torch.rand(B, KVH, n, generator=g, device=dev, dtype=torch.float64)
    span = g0 - (c0 - K)  # >= 2 K tokens older than the newest c0 - K
    pos = torch.where(i < K, torch.floor((i + jitter) * (span / K)), i - c0 + g0) + lp
    return k, v, pos.to(torch.int32).contiguous()


def _window(c, seed, l):
    return _randn(_gen(seed, 4, l), c["batch"], c["kv_heads"] * c["group"], c["buffer"], D)


def _step_inputs(c, seed, t):
    """q, k, v of decode step t: [L][B][heads][128]."""
    g = _gen(seed, 5, t)
    L, B, KVH, H = c["layers"], c["batch"], c["kv_heads"], c["kv_heads"] * c["group"]
    k = torch.stack([_scaled(_randn(g, B, KVH, D).unsqueeze(2), _key_scale(c, seed, l)).squeeze(2) for l in range(L)])
    return _randn(g, L, B, H, D), k, _randn(g, L, B, KVH, D)


def _entering(c, seed, i):
    """The prompt rows of request i that enters: [L][KVH][row stride][128]."""
    g = _gen(seed, 6, i)
    shape = (c["layers"], c["kv_heads"], max(1, c["prompt_hi"]), D)
    k = torch.empty(shape, device="cuda", dtype=torch.bfloat16)
    for l in range(c["layers"]):
        k[l] = _scaled(_randn(g, *shape[1:]), _key_scale(c, seed, l))
    return k, _randn(g, *shape)


# ------------------------------------------------------------------------------ a pass
class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.c, L, B = c, c["layers"], c["batch"]
    lp, (g0, c0) = _prompts(c), _start(c)
    pool = None
    if c["kind"] == "admit":
        pool = (c["prompt_hi"], B * -(-c["prompt_hi"] // 192) * 192)
    s.cache = ra.RandomAttentionCache(L, c["kv_heads"] * c["group"], c["kv_heads"], D, lp, c["budget"], c["buffer"],
                                      seed=seed, policy=POLICY[c["policy"]], block=c["block"],
                                      compaction=LAYOUT[c["layout"]], prompt_pool=pool)
    s.ctx, s.g0, s.c0 = s.cache.ctx, g0, c0
    s.prompt, s.saved, s.window = [], [], []
    for l in range(L):
        k, v = _prompt_rows(c, seed, l)
        ra.ra_prefill(s.ctx, l, k.data_ptr(), v.data_ptr(), k.shape[2])
        if c["kind"] == "prefill":
            s.prompt.append((k, v))
        if max(c0) > 0:
            k, v, pos = _cached_rows(c, seed, l, lp, g0, c0)
            ra.ra_restore(s.ctx, l, g0, c0, pos.data_ptr(), k.data_ptr(), v.data_ptr(), k.shape[2])
            if c["kind"] == "resume":
                s.saved.append((k, v, pos))
            if c["policy"] == "scored":
                w = _window(c, seed, l)
                ra.ra_restore_queries(s.ctx, l, w.data_ptr())
                if c["kind"] == "resume":
                    s.window.append(w)
    s.inputs = [_step_inputs(c, seed, t) for t in range(RING)]
    s.layer_inputs = [[[x[l] for x in s.inputs[t]] for l in range(L)] for t in range(RING)]
    if c["kind"] == "admit":
        s.entering = [(n,) + _entering(c, seed, i) for i, n in enumerate(_admitted(c))]
    s.out = torch.zeros(L, B, c["kv_heads"] * c["group"], D, device="cuda", dtype=torch.bfloat16)
    s.layer_out = [s.out[l] for l in range(L)]
    s.t = 0
    torch.cuda.synchronize()
    return s


def run(state):
    s, c, ctx = state, state.c, state.ctx
    kind, t = c["kind"], state.t
    s.t += 1
    if kind == "admit":  # the oldest request is finished; another one takes its slot
        slot = t % c["batch"]
        n, k, v = s.entering[t % len(s.entering)]
        ra.ra_set_active(ctx, slot, 0)
        ra.ra_admit(ctx, slot, n, k.data_ptr(), v.data_ptr(), k.shape[2])
    if kind in ("step", "admit"):
        q, k, v = s.inputs[t % RING]
        ra.ra_decode_step(ctx, q.data_ptr(), k.data_ptr(), v.data_ptr(), s.out.data_ptr())
        return s.out
    layers = s.layer_inputs[t % RING]
    if kind == "prefill":
        for l, (q, _, _) in enumerate(layers):
            k, v = s.prompt[l]
            ra.ra_prefill(ctx, l, k.data_ptr(), v.data_ptr(), k.shape[2])
            ra.ra_decode_attn(ctx, l, q.data_ptr(), s.layer_out[l].data_ptr())
        return s.out
    if kind == "calls":
        fired = []
        for l, (q, k, v) in enumerate(layers):
            ra.ra_append_kv(ctx, l, k.data_ptr(), v.data_ptr())
            fired.append(ra.ra_evict(ctx, l))
            ra.ra_decode_attn(ctx, l, q.data_ptr(), s.layer_out[l].data_ptr())
        return {"out": s.out, "fired": fired}
    if kind == "resume":
        for l, (k, v, pos) in enumerate(s.saved):
            ra.ra_restore(ctx, l, s.g0, s.c0, pos.data_ptr(), k.data_ptr(), v.data_ptr(), k.shape[2])
            if s.window:
                ra.ra_restore_queries(ctx, l, s.window[l].data_ptr())
    for l, (q, k, v) in enumerate(layers):
        ra.ra_decode_layer(ctx, l, q.data_ptr(), k.data_ptr(), v.data_ptr(), s.layer_out[l].data_ptr())
    return s.out


def work(case):
    """Rows are 512 bytes (K and V).  A step reads every attended row, its queries and new rows, and writes
    its outputs and the new rows; a round every r steps writes the survivors again (time order) or the
    refilled slots; loading reads and writes the rows loaded."""
    c = case
    L, B, KVH, G, K, r = c["layers"], c["batch"], c["kv_heads"], c["group"], c["budget"], c["buffer"]
    row, lp, kind = 4 * D, sum(_prompts(c)), c["kind"]
    io = L * B * KVH * (2 * G * D * 2 + 2 * row)
    copied = 0.0
    extra = 0.0  # flops beside the decode attention's
    if kind == "prefill":
        rows, io = lp, L * B * KVH * 2 * G * D * 2
        copied = 2.0 * lp * row
    elif kind == "admit":
        mean = sum(_admitted(c)) / 3.0
        rows = B * (mean + (B + 1) / 2.0)
        copied = 2.0 * mean * row
    else:
        cached = B * (K + r + (r + 1) / 2.0)
        rows = lp + cached
        copied = B / r * (K + r if c["layout"] == "ordered" else 2 * r) * (row + 4)
        if c["policy"] == "scored":  # the window's weights on the candidates
            extra += B / r * (K + r) * 2.0 * r * G * D
        if kind == "resume":
            copied += 2.0 * cached * (row + 4)
            if c["policy"] == "scored":  # the window's normalisers over all the rows it sees
                copied += lp * row / 2 + B * r * G * D * 4
                extra += (lp + cached) * 2.0 * r * G * D
    heads = L * KVH
    return {"bytes": heads * (rows * row + copied) + io, "flops": heads * (rows * 4.0 * G * D + extra)}


def tolerance(case):
    # bf16 outputs of fp32 sums whose weights are rounded to bf16: 2.3e-3 from 64 bits, and another
    # split of the rows gives 3e-3 between two results (largest difference 0.027 of the rms)
    return {"rel": 0.012, "max": 0.11}


# ------------------------------------------------------------------------------ in 64 bits
def _philox(x0, x1, x2, x3, k0, k1):
    """Word 0 of Philox4x32-10 (Salmon et al., SC'11), on int64 tensors that hold 32-bit words."""
    M = 0xFFFFFFFF
    for _ in range(10):
        p, q = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = ((q >> 32) & M) ^ x1 ^ k0, q & M, ((p >> 32) & M) ^ x3 ^ k1, p & M
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return x0


def _kept(c, seed, l, b, g, pos, score):
    """Slots of [KVH][n] candidates that survive a round at step g (positions `pos`), per head: a mask."""
    KVH, n = pos.shape
    K = c["budget"]
    j = torch.arange(n, device=pos.device, dtype=torch.int64).expand(KVH, n)
    if c["policy"] == "scored":
        pooled = torch.nn.functional.max_pool1d(score[:, None, :], 7, 1, 3)[:, 0, :]
        order = torch.argsort(-pooled, dim=1, stable=True)
    else:
        head = b * KVH + (torch.zeros(KVH, 1) if c["policy"] == "shared" else torch.arange(KVH)[:, None])
        word = pos if c["layout"] == "free" else j
        if c["policy"] == "block":
            word = pos // c["block"]
        if c["policy"] == "recency":
            key = 0xFFFFFFFF - word
        else:
            z = torch.zeros_like(j)
            key = _philox(word + z, z + g, z + l, z + head.to(j), z + (seed & 0xFFFFFFFF), z + (seed >> 32))
        order = torch.argsort(key * 65536 + j, dim=1)
    mask = torch.zeros(KVH, n, dtype=torch.bool, device=pos.device)
    return mask.scatter_(1, order[:, :K], True)


def _attend(q, k, v):
    """[KVH][G][128] over [KVH][n][128]."""
    return torch.softmax(q @ k.transpose(1, 2) / math.sqrt(D), dim=-1) @ v


def exact(case, seed):
    c = case
    L, B, KVH, G, K, r = c["layers"], c["batch"], c["kv_heads"], c["group"], c["budget"], c["buffer"]
    lp, (g0, c0) = _prompts(c), _start(c)
    qs, ks, vs = _step_inputs(c, seed, 0)
    out = torch.zeros(L, B, KVH * G, D, dtype=torch.float64, device="cuda")
    enter = _entering(c, seed, 0) if c["kind"] == "admit" else None
    for l in range(L):
        pk, pv = _prompt_rows(c, seed, l)
        if max(c0) > 0:
            gk, gv, pos = _cached_rows(c, seed, l, lp, g0, c0)
            window = _window(c, seed, l) if c["policy"] == "scored" else None
        for b in range(B):
            q = qs[l, b].double().view(KVH, G, D)
            n = lp[b]
            k, v = pk[b, :, :n].double(), pv[b, :, :n].double()
            if enter is not None and b == 0:
                n = _admitted(c)[0]
                k, v = enter[0][l, :, :n].double(), enter[1][l, :, :n].double()
            if c["kind"] != "prefill":
                if c0[b] > 0:
                    k = torch.cat([k, gk[b, :, :c0[b]].double()], 1)
                    v = torch.cat([v, gv[b, :, :c0[b]].double()], 1)
                k = torch.cat([k, ks[l, b].double().unsqueeze(1)], 1)
                v = torch.cat([v, vs[l, b].double().unsqueeze(1)], 1)
            g, cand = g0[b] + 1, c0[b] + 1 - r
            if c0[b] > 0 and g % r == 0 and cand > K:
                p = pos[b, :, :cand].long()
                score = None
                if window is not None:  # softmax of the r latest queries over the keys each had seen
                    w = window[b].double().view(KVH, G, r, D)
                    every = torch.cat([torch.arange(n, device="cuda").expand(KVH, n), pos[b, :, :c0[b]].long()], 1)
                    own = n + g0[b] - r + torch.arange(r, device="cuda")  # position of each query's own token
                    seen = every[:, None, None, :] <= own[None, None, :, None]
                    logit = (w.reshape(KVH, G * r, D) @ k[:, :-1].transpose(1, 2)).view(KVH, G, r, -1) / math.sqrt(D)
                    weight = torch.softmax(logit.masked_fill(~seen, -math.inf), dim=-1)
                    score = weight.sum((1, 2))[:, n:n + cand]
                mask = torch.ones(KVH, k.shape[1], dtype=torch.bool, device="cuda")
                mask[:, n:n + cand] = _kept(c, seed, l, b, g, p, score)
                k, v = k[mask].view(KVH, -1, D), v[mask].view(KVH, -1, D)
            out[l, b] = _attend(q, k, v).reshape(KVH * G, D)
    return {"out": out, "fired": None} if c["kind"] == "calls" else out
