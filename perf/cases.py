"""The work whose time is watched: what a decode loop has this library do, through its public entry points.

A case names one pass: a token (or a batch of tokens, one per sequence) through one MLP block or a short stack
of them, at the shapes of the repository's workloads, or at other sizes of the same ranges (`draw`).  The kinds:

  step        dip_mlp_step: one block, one token; between two such calls a model runs its attention
  stack       dip_stack_step: one token through several blocks with the residual + rms chaining between them
  batch       dip_mlp_step with several tokens (a mask per token, the union of the rows read once)
  tiered      dip_mlp_step_tiered: the cached columns in device memory, all weights in pinned host memory
  pruned      dip_mlp_step_neuron_pruned: Gate / Up pruning
  primitives  dip_ca_mask / dip_mask_topk and the two list-driven products as calls of their own

A state holds several tokens and takes the next one in each pass, as a decode loop does: the column caches
therefore see new masks all the time.  Inputs are synthetic: N(0, 0.02) weights, heavy-tailed activations.
"""
import math

import torch

import paper_2412_01380_b200 as dip

WTYPES = {"f32": dip.W_F32, "bf16": dip.W_BF16, "int4": dip.W_INT4_G128}
WEIGHT_BYTES = {"f32": 4.0, "bf16": 2.0, "int4": 0.5}
TOKENS = 8


def _case(kind, wtype, d_model, d_ff, keep, budget=None, policy="lru", layers=1, batch=1, graph=False,
          dist="student_t3", gamma=0.2, name=None):
    c = {"kind": kind, "wtype": wtype, "d_model": d_model, "d_ff": d_ff, "keep": keep, "budget": budget, "policy": policy,
         "layers": layers, "batch": batch, "graph": graph, "dist": dist, "gamma": gamma if budget is not None else 1.0}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one small fp32 block (an on-device assistant's model), latency and launches count
        _case("step", "f32", 1024, 2816, 0.5, name="block_f32_step"),
        # one token through blocks of a 4-billion-parameter model, called without a CUDA graph
        _case("stack", "bf16", 3072, 8192, 0.25, 0.5, layers=3, name="phi3_mini_stack"),
        # the headline: one token through Phi-3-Medium blocks, cache-aware masks, a CUDA graph per token
        _case("stack", "bf16", 5120, 17920, 0.25, 0.5, layers=3, graph=True, dist="laplace", name="phi3_medium_stack_graph"),
        # a block inside a model whose attention runs between the calls; the mask is larger than the cache, LFU
        _case("step", "bf16", 5120, 17920, 0.5, 0.25, "lfu", dist="laplace", name="phi3_medium_step_lfu"),
        # the largest single-token call: keep ratio 1, the dense product through the same path
        _case("step", "bf16", 5120, 17920, 1.0, dist="laplace", name="phi3_medium_step_dense"),
        # 4-bit weights, cache-aware masks, a CUDA graph per token
        _case("stack", "int4", 4096, 14336, 0.25, 0.4, layers=3, graph=True, name="llama3_8b_int4_stack_graph"),
        # batched decode: two sequences, a few, and the most a call takes
        _case("batch", "bf16", 5120, 17920, 0.25, batch=2, name="phi3_medium_batch_2"),
        _case("batch", "bf16", 5120, 17920, 0.25, batch=5, graph=True, name="phi3_medium_batch_5"),
        _case("batch", "bf16", 5120, 17920, 0.25, batch=16, name="phi3_medium_batch_16"),
        # weights larger than the device's share: misses are read over the host link
        _case("tiered", "bf16", 3072, 8192, 0.25, 0.5, name="phi3_mini_tiered"),
        # the neuron-wise schedule: one dense product, the rest on the kept neurons
        _case("pruned", "bf16", 5120, 17920, 0.25, dist="laplace", name="phi3_medium_gate_pruned"),
        # masks and products called one by one (a caller with its own code between them), ragged sizes
        _case("primitives", "bf16", 2080, 5472, 0.3, 0.45, name="primitives_ragged"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """A case of the same kinds and ranges: d_model 256 .. 5120, d_ff 1.5 .. 4 times that, keep ratio 0.05 .. 1."""
    kind = rng.choice(["step", "step", "step", "stack", "stack", "batch", "batch", "tiered", "pruned", "primitives"])
    wtype = rng.choice(["bf16", "bf16", "bf16", "f32"] if kind in ("batch", "pruned") else ["bf16", "bf16", "int4", "int4", "f32"])
    unit = 128 if wtype == "int4" else 32
    top = 3072 if kind == "tiered" or wtype == "f32" else 5120
    while True:
        d_model = max(256, int(_log(rng, 256, top)) // unit * unit)
        d_ff = int(d_model * rng.uniform(1.5, 4.0)) // unit * unit
        keep = round(min(1.0, _log(rng, 0.05, 1.25)), 3)
        budget = None
        if kind == "tiered" or (kind in ("step", "stack", "primitives") and rng.random() < 0.7):
            budget = round(rng.uniform(0.2, 0.6), 2)
        layers = rng.randint(2, 3) if kind == "stack" else 1
        batch = rng.randint(2, 16) if kind == "batch" else 1
        c = _case(kind, wtype, d_model, d_ff, keep, budget, rng.choice(["lru", "lfu"]), layers, batch,
                  rng.random() < 0.5, rng.choice(["student_t3", "laplace"]), round(rng.uniform(0.1, 0.5), 2))
        if d_ff <= 17920 and work(c)["bytes"] <= (60e6 if kind == "tiered" else 550e6):
            return c


# ---- inputs ------------------------------------------------------------------------------------------------------------
def _keep(c, d):
    return max(1, min(d, int(c["keep"] * d + 0.5)))


def _capacity(c, d):
    return max(0, min(d, int(c["budget"] * d)))


def _weights(gen, wtype, d_out, d_in):
    """An [d_out, d_in] matrix in its storage type, and the INT4 scales."""
    z = torch.randn((d_out, d_in), generator=gen, device="cuda").mul_(0.02)
    if wtype == "f32":
        return z, None
    if wtype == "bf16":
        return z.to(torch.bfloat16), None
    g = z.view(d_out, d_in // 128, 128)
    scale = (g.abs().amax(dim=2) / 7.0).to(torch.float16)
    q = (torch.clamp(torch.round(g / scale.float().unsqueeze(2)), -7, 7) + 8).to(torch.uint8).view(d_out, d_in)
    return (q[:, 0::2] | (q[:, 1::2] << 4)).contiguous(), scale.t().contiguous()


def _tokens(c, gen):
    """[TOKENS, (batch,) d_model] activations; a two-tier loop's are correlated in time, as real ones are."""
    shape = (TOKENS, c["batch"], c["d_model"])
    if c["dist"] == "laplace":
        u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5
        v = -torch.sign(u) * torch.log1p(-2 * u.abs())
    else:
        chi = torch.randn((3,) + shape, generator=gen, device="cuda", dtype=torch.float64).square().mean(0)
        v = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64) / chi.sqrt()
    if c["kind"] == "tiered":
        for t in range(1, TOKENS):
            v[t] = 0.95 * v[t - 1] + math.sqrt(1 - 0.95 ** 2) * v[t]
    if c["dist"] != "laplace":
        v /= v.square().mean(dim=-1, keepdim=True).sqrt()
    v = v.float().contiguous()
    return v if c["kind"] == "batch" else v[:, 0].contiguous()


class State:
    """A decode loop's objects: context, packed weights, caches, buffers, tokens, and (graph) its captured pass."""


def prepare(case, seed):
    c, s = case, State()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s.case, s.t = c, 0
    s.ctx = dip.Context(torch.cuda.current_device())
    d_model, d_ff, wt = c["d_model"], c["d_ff"], WTYPES[c["wtype"]]
    s.k_x, s.k_h, s.gamma = _keep(c, d_model), _keep(c, d_ff), c["gamma"]
    s.w = []
    for _ in range(c["layers"]):
        g, gs = _weights(gen, c["wtype"], d_ff, d_model)
        u, us = _weights(gen, c["wtype"], d_ff, d_model)
        if c["kind"] == "pruned":
            down, _ = _weights(gen, c["wtype"], d_ff, d_model)
            s.w.append(dip.NeuronWeights(wt, g, u, down))
        else:
            d, ds = _weights(gen, c["wtype"], d_model, d_ff)
            s.w.append(dip.dip_pack_weights(s.ctx, wt, d_model, d_ff, g, u, d, gs, us, ds))
        torch.cuda.synchronize()
    s.xs = _tokens(c, gen)
    s.gu = s.d = None
    if c["budget"] is not None:
        s.gu = [dip.CacheState(d_model, _capacity(c, d_model), "cuda", c["policy"]) for _ in s.w]
        s.d = [dip.CacheState(d_ff, _capacity(c, d_ff), "cuda", c["policy"]) for _ in s.w]
    lead = (c["batch"],) if c["kind"] == "batch" else ()
    ints = dict(dtype=torch.int32, device="cuda")
    s.x = torch.empty(lead + (d_model,), device="cuda")
    s.y = torch.empty(lead + (d_model,), device="cuda")
    s.h = torch.empty(lead + (d_ff,), device="cuda")
    s.mask_x = torch.zeros(lead + (d_model // 32,), **ints)
    s.mask_h = torch.zeros(lead + (d_ff // 32,), **ints)
    s.idx_x, s.idx_h = torch.zeros(s.k_x, **ints), torch.zeros(s.k_h, **ints)
    if c["kind"] == "stack":
        s.stack = dip.Stack(s.w, s.gu, s.d)
    if c["kind"] == "tiered":
        w = s.w[0]
        s.tiers = []
        for cache, packed, d, k in ((s.gu[0], w.gate_up, d_model, s.k_x), (s.d[0], w.down, d_ff, s.k_h)):
            s.tiers.append(dip.Tier(cache, packed.cpu().pin_memory(), packed.numel() // d, k, "cuda"))
        w.gate_up = w.down = None
        w.struct.gate_up = w.struct.down = None
    s.graph = None
    if c["graph"] and c["kind"] != "tiered":
        s.x.copy_(s.xs[0])
        _enqueue(s, s.x)                                # once outside the capture, then cold caches again
        torch.cuda.synchronize()
        for cache in (s.gu or []) + (s.d or []):
            cache.stamp.fill_(-1)
            cache.meta.zero_()
            if cache.count is not None:
                cache.count.zero_()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            _enqueue(s, s.x)
    torch.cuda.synchronize()
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------------
def _enqueue(s, x):
    kind, w = s.case["kind"], s.w[0]
    gu, d = (s.gu[0], s.d[0]) if s.gu else (None, None)
    if kind == "stack":
        dip.dip_stack_step(s.ctx, s.stack, x, s.k_x, s.k_h, s.gamma, s.y)
    elif kind in ("step", "batch"):
        dip.dip_mlp_step(s.ctx, w, x, s.k_x, s.k_h, s.gamma, gu, d, s.y, mask_x=s.mask_x, h=s.h, mask_h=s.mask_h)
    elif kind == "tiered":
        dip.dip_mlp_step_tiered(s.ctx, w, s.tiers[0], s.tiers[1], x, s.k_x, s.k_h, s.gamma, s.y,
                                mask_x=s.mask_x, h=s.h, mask_h=s.mask_h)
    elif kind == "pruned":
        dip.dip_mlp_step_neuron_pruned(s.ctx, w, "gate", x, s.k_h, s.y, mask=s.mask_h, h=s.h)
    else:
        for v, k, cache, mask, idx, product, out in ((x, s.k_x, gu, s.mask_x, s.idx_x, dip.dip_sparse_gemv_gate_up, s.h),
                                                     (s.h, s.k_h, d, s.mask_h, s.idx_h, dip.dip_sparse_gemv_down, s.y)):
            if cache is not None:
                dip.dip_ca_mask(s.ctx, v, k, s.gamma, cache, mask, idx)
            else:
                dip.dip_mask_topk(s.ctx, v, k, mask, idx)
            product(s.ctx, w, v, idx, k, None, out)


def run(state):
    s = state
    x = s.xs[s.t % TOKENS]
    s.t += 1
    if s.graph is not None:
        s.x.copy_(x)
        s.graph.replay()
    else:
        _enqueue(s, x)
    out = {"y": s.y}
    if s.case["kind"] != "stack":
        out.update(h=s.h, mask_h=s.mask_h)
        if s.case["kind"] != "pruned":
            out["mask_x"] = s.mask_x
    for name, caches in (("gu", s.gu), ("d", s.d)):
        for i, cache in enumerate(caches or []):
            out["%s%d" % (name, i)] = [cache.stamp, cache.meta, cache.count]
    return out


# ---- what a pass cannot do without, and how exact its results are ------------------------------------------------------
def work(case):
    c = case
    d_model, d_ff, bw = c["d_model"], c["d_ff"], WEIGHT_BYTES[c["wtype"]]
    k_x, k_h, b = _keep(c, d_model), _keep(c, d_ff), c["batch"]
    vectors = b * (8 * d_model + 4 * d_ff + (d_model + d_ff) / 8)           # x, y, h and the masks
    if c["kind"] == "pruned":
        rows = d_ff + 2 * k_h                                              # one dense product, kept rows and columns
        return {"bytes": rows * d_model * bw + vectors, "flops": 2.0 * rows * d_model}
    # several tokens: the expected union of independent masks
    rows_x = d_model * (1 - (1 - k_x / d_model) ** b)
    rows_h = d_ff * (1 - (1 - k_h / d_ff) ** b)
    weights = (rows_x * 2 * d_ff + rows_h * d_model) * bw
    if c["wtype"] == "int4":                                               # binary16 scale rows of the groups touched
        weights += (min(k_x, d_model // 128) * 2 * d_ff + min(k_h, d_ff // 128) * d_model) * 2
    state = 8 * (d_model + d_ff) if c["budget"] is not None else 0         # stamps read and written
    flops = 2.0 * b * (k_x * 2 * d_ff + k_h * d_model)
    return {"bytes": c["layers"] * (weights + vectors + state), "flops": c["layers"] * flops}


def tolerance(case):
    """Sums in another order differ by 1e-6 (2-norm; 1e-5 where bf16 pairs stand for the values).  But with the last
    bits of h the ranking of h may swap the two columns next to the threshold, seen in 1 to 8 of 1000 layers in a
    float64 comparison: one swap moves y by 2e-3 to 9e-3 of its norm and four mask or state words at most, and in a
    stack it moves the next block's input and so several columns of its masks (2e-2 of x)."""
    if case["kind"] == "stack":
        return {"rel": 3e-2, "max": 0.3, "differ": 0.01}
    if case["keep"] >= 1.0 and case["kind"] != "pruned":
        return {"rel": 4e-5, "max": 4e-4}
    return {"rel": 1e-2, "max": 0.1, "differ": 0.01}


# ---- the same in 64 bits, with plain torch -----------------------------------------------------------------------------
def _stored(weights, wtype):
    """The values that a stored matrix and its scales stand for."""
    q, scale = weights
    if wtype != "int4":
        return q.double()
    codes = torch.stack((q & 15, q >> 4), dim=2).view(q.shape[0], -1).double() - 8
    return codes * scale.t().double().repeat_interleave(128, dim=1)


def _kept(c, v, k):
    """The 0/1 mask of the k largest keys of each row (cold caches: no column is resident yet), the lower column first among
    equals, and whether another summation order of v could give another mask."""
    key = v.float().abs()
    if c["budget"] is not None:
        key = key * torch.tensor(c["gamma"], dtype=torch.float32, device=key.device)
    order = torch.argsort(key, dim=-1, descending=True, stable=True)
    mask = torch.zeros_like(v).scatter_(-1, order[..., :k], 1.0)
    if k == v.shape[-1]:
        return mask, False
    edge = key.gather(-1, order[..., k - 1:k + 1]).double()
    size = torch.maximum(edge[..., 0], key.double().square().mean(-1).sqrt())
    return mask, bool((edge[..., 0] - edge[..., 1] < (1e-4 if c["batch"] > 2 else 1e-5) * size).any())


def exact(case, seed):
    """What the first pass of a new state returns.  None for an output that hangs on the ranking of two columns whose keys are
    equal to within the rounding of their sums, or for the case where that is every output."""
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    d_model, d_ff = c["d_model"], c["d_ff"]
    stored = []
    for _ in range(c["layers"]):
        shapes = ((d_ff, d_model), (d_ff, d_model), (d_ff, d_model) if c["kind"] == "pruned" else (d_model, d_ff))
        stored.append([_weights(gen, c["wtype"], *s) for s in shapes])
    x = _tokens(c, gen)[0].double()
    silu = torch.nn.functional.silu
    near = False
    for n, layer in enumerate(stored):
        if n:
            r = x + y
            x = r / r.square().mean(-1, keepdim=True).sqrt()
        gate, up, down = (_stored(m, c["wtype"]) for m in layer)
        if c["kind"] == "pruned":
            p = silu(x @ gate.t())
            mask_h, tie_h = _kept(c, p, _keep(c, d_ff))
            h = p * (x @ up.t()) * mask_h
            y = h @ down
        else:
            mask_x, tie_x = _kept(c, x, _keep(c, d_model))
            near = near or (n > 0 and tie_x)                  # (the first block's x is given: its mask is exact)
            h = (x * mask_x) @ up.t() * silu((x * mask_x) @ gate.t())
            mask_h, tie_h = _kept(c, h, _keep(c, d_ff))
            y = (h * mask_h) @ down.t()
        near = near or tie_h
    if c["kind"] == "stack":
        r = x + y
        return None if near else {"y": r / r.square().mean(-1, keepdim=True).sqrt()}
    if near:
        return None if c["kind"] == "pruned" else {"y": None, "h": h}        # (there h itself is masked)
    return {"y": y, "h": h}
