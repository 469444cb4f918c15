"""Single-token steps whose products select for themselves, at the sizes where the kernel's branches meet: one and several
chunks of columns per thread (8192 / 8224 columns), the variants of the cache update that rides along (8192, 20480), down
products that leave SMs for updates, fill the SMs to the last one (the updates get launches of their own) or take a second
wave, row parts of one row, keep counts 1 and d, and threshold bins of 256 and 257 columns (the last that is ranked in
place, the first that is not).  What a call launches is read from the library's own timeline."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, bits_to_mask, check_step, graph_us, rel_err, upload_layer

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [
    (di.W_BF16, 8192, 96, 0.3), (di.W_BF16, 8224, 64, 0.3), (di.W_F32, 12288, 64, 0.2), (di.W_BF16, 32, 20512, 0.2),
    (di.W_BF16, 64, 8192, 0.25), (di.W_BF16, 64, 8224, 0.25), (di.W_BF16, 64, 9472, 0.25), (di.W_BF16, 32, 18944, 0.1),
    (di.W_F32, 96, 160, 0.02), (di.W_F32, 160, 96, 1.0), (di.W_BF16, 2080, 5472, 0.999),
    # 4-bit: 8, 32 and 64 columns per thread of the list, more rows than one round, quads beyond 32, and a width whose
    # keys do not fit beside the tables (select kernels in front)
    (di.W_INT4_G128, 128, 256, 0.01), (di.W_INT4_G128, 4096, 4224, 0.25), (di.W_INT4_G128, 384, 16512, 0.3),
    (di.W_INT4_G128, 4224, 384, 0.9), (di.W_INT4_G128, 16512, 128, 0.2), (di.W_INT4_G128, 256, 18048, 1.0),
    (di.W_INT4_G128, 128, 32768, 0.1),
]


def _layer(d_model, d_ff, wtype, seed):
    return di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=seed, d_model=d_model, d_ff=d_ff, wtype=wtype, n_layers=1), 0)


def launch_kinds(ctx, call):
    """The kinds of the library's launches in a call, as its own timeline records them."""
    ctx.trace_begin()
    call()
    torch.cuda.synchronize()
    kinds = [r["kind"] for r in ctx.trace_read()]
    ctx.trace_end()
    return kinds


@pytest.mark.parametrize("policy", [None, "lru", "lfu"])
@pytest.mark.parametrize("wtype,d_model,d_ff,rho", SHAPES)
def test_steps_at_the_kernels_edges(wtype, d_model, d_ff, rho, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    lw = _layer(d_model, d_ff, wtype, d_model + d_ff)
    w = upload_layer(dip, ctx, lw)
    k_x, k_h = max(1, int(rho * d_model)), max(1, int(rho * d_ff))
    refs, mine = [None, None], [None, None]
    if policy:
        for i, d in enumerate((d_model, d_ff)):
            refs[i] = oracle.Cache(d, int(0.4 * d), policy)
            mine[i] = dip.CacheState(d, int(0.4 * d), "cuda", policy)
    for t in range(4):
        check_step(dip, ctx, lw, w, di.heavy_tail_vector(70 + t, d_model), k_x, k_h, 0.2, *refs, *mine)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("wtype", [di.W_BF16, di.W_INT4_G128])
@pytest.mark.parametrize("n_tied", [1, 32, 33, 255, 256, 257])
@pytest.mark.parametrize("kept", ["one", "half", "all"])
def test_threshold_bins_of_every_size(n_tied, kept, wtype):
    """n_tied columns share the threshold's magnitude; one, half or all of them are kept."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d_model, d_ff, above = 1024, 384, 200
    lw = _layer(d_model, d_ff, wtype, n_tied)
    w = upload_layer(dip, ctx, lw)
    rng = np.random.default_rng(n_tied)
    x = np.concatenate([rng.uniform(4.0, 9.0, above), np.full(n_tied, 1.5), rng.uniform(0.01, 1.0, d_model - above - n_tied)])
    x = (rng.permutation(x) * rng.choice([-1, 1], d_model)).astype(np.float32)
    k = above + {"one": 1, "half": (n_tied + 1) // 2, "all": n_tied}[kept]
    for policy in (None, "lru"):
        refs = [None, None] if policy is None else [oracle.Cache(d, d // 3) for d in (d_model, d_ff)]
        mine = [None, None] if policy is None else [dip.CacheState(d, d // 3, "cuda") for d in (d_model, d_ff)]
        for _ in range(2):
            check_step(dip, ctx, lw, w, x, k, 80, 0.25, *refs, *mine)
    ctx.close()


@pytest.mark.parametrize("caches", ["both", "x", "h"])
@pytest.mark.parametrize("n_layers", [1, 3, 4, 9])
@pytest.mark.parametrize("wtype", [di.W_BF16, di.W_INT4_G128])
def test_stacks_leave_their_cache_updates_to_later_launches(n_layers, caches, wtype):
    """A stack's cache states equal those of its blocks stepped one by one (blocks whose updates ride with the last down
    product, fill a launch beside the products, or have no product with a cache to ride with)."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d_model, d_ff = 256, 640
    k_x, k_h = 64, 200
    ws = [upload_layer(dip, ctx, _layer(d_model, d_ff, wtype, 100 + l)) for l in range(n_layers)]

    def states():
        return [[dip.CacheState(d, d // 2, "cuda") for _ in ws] if caches in (c, "both") else None
                for d, c in ((d_model, "x"), (d_ff, "h"))]
    gu, d = states()
    gu1, d1 = states()
    stack = dip.Stack(ws, gu, d)
    out = torch.empty(d_model, device="cuda")
    y = torch.empty(d_model, device="cuda")
    for t in range(5):
        x = torch.from_numpy(di.heavy_tail_vector(300 + t, d_model)).cuda()
        dip.dip_stack_step(ctx, stack, x, k_x, k_h, 0.2, out)
        for l, w in enumerate(ws):
            dip.dip_mlp_step(ctx, w, x, k_x, k_h, 0.2, gu1[l] if gu1 else None, d1[l] if d1 else None, y)
            nxt = torch.empty_like(x)
            dip.dip_residual_rmsnorm(ctx, x, y, nxt)
            x = nxt
        torch.cuda.synchronize()
        assert torch.equal(out, x), t
        for a, b in ((gu, gu1), (d, d1)):
            for p, q in zip(a or [], b or []):
                assert torch.equal(p.stamp, q.stamp) and torch.equal(p.meta, q.meta), t
    assert ctx.device_status() == 0
    ctx.close()


# launches for cache updates alone in a stack of 1, 3, 4, 9 blocks: at most seven updates wait, for the last down product
# (F32 / BF16 with a cache) or a launch beside it; a 4-bit call ends with one for the last down input
UPDATE_LAUNCHES = {("both", False): {1: 0, 3: 0, 4: 0, 9: 2}, ("x", False): {1: 1, 3: 1, 4: 1, 9: 2}, ("h", False): {1: 0, 3: 0, 4: 0, 9: 1},
                   ("both", True): {1: 2, 3: 2, 4: 2, 9: 4}, ("x", True): {1: 1, 3: 1, 4: 1, 9: 2}, ("h", True): {1: 1, 3: 2, 4: 2, 9: 3}}


@pytest.mark.parametrize("caches", ["both", "x", "h"])
@pytest.mark.parametrize("n_layers", [1, 3, 4, 9])
@pytest.mark.parametrize("wtype,d_model,policy", [(di.W_BF16, 256, "lru"), (di.W_BF16, 5120, "lfu"), (di.W_INT4_G128, 256, "lru")])
def test_updates_of_a_stack_by_launch(n_layers, caches, wtype, d_model, policy):
    """A stack's cache states equal those of its blocks stepped one by one on a context whose selects and updates are launches
    of their own (blocks whose updates ride with the last down product, fill a launch beside the products, or have no
    product with a cache to ride with)."""
    import paper_2412_01380_b200 as dip
    ctx, plain = dip.Context(0), dip.Context(0, select_in_product=-1)
    d_ff = 640
    k_x, k_h = d_model // 4, 200
    ws = [upload_layer(dip, ctx, _layer(d_model, d_ff, wtype, 100 + l)) for l in range(n_layers)]

    def states():
        return [[dip.CacheState(d, d // 2, "cuda", policy) for _ in ws] if caches in (c, "both") else None
                for d, c in ((d_model, "x"), (d_ff, "h"))]
    gu, d = states()
    gu1, d1 = states()
    stack = dip.Stack(ws, gu, d)
    out = torch.empty(d_model, device="cuda")
    y = torch.empty(d_model, device="cuda")
    probe = dip.StackProbe(n_layers, 1, d_model, d_ff, "cuda")
    for t in range(5):
        x = torch.from_numpy(di.heavy_tail_vector(300 + t, d_model)).cuda()
        kinds = launch_kinds(ctx, lambda: dip.dip_stack_step_probed(ctx, stack, x, k_x, k_h, 0.2, out, probe))
        assert kinds.count("cache_update") == UPDATE_LAUNCHES[caches, wtype == di.W_INT4_G128][n_layers], kinds
        for l, w in enumerate(ws):
            # (each block on the stack's own input, each mask on its own h: sums in another order swap no columns)
            for v, k, c, want in ((probe.x[l, 0], k_x, gu1, probe.mask_x[l, 0]), (probe.h[l, 0], k_h, d1, probe.mask_h[l, 0])):
                mask = torch.zeros(v.numel() // 32, dtype=torch.int32, device="cuda")
                if c:
                    dip.dip_ca_mask(plain, v.clone(), k, 0.2, c[l], mask, None)
                else:
                    dip.dip_mask_topk(plain, v.clone(), k, mask, None)
                assert torch.equal(mask, want), (t, l)
        torch.cuda.synchronize()
        for a, b in ((gu, gu1), (d, d1)):
            for p, q in zip(a or [], b or []):
                assert torch.equal(p.stamp, q.stamp) and torch.equal(p.meta, q.meta), t
                assert policy == "lru" or torch.equal(p.count, q.count), t
    # and the call without the intermediates does the same
    again = states()
    twin = dip.Stack(ws, *again)
    for t in range(5):
        dip.dip_stack_step(ctx, twin, torch.from_numpy(di.heavy_tail_vector(300 + t, d_model)).cuda(), k_x, k_h, 0.2, y)
    torch.cuda.synchronize()
    assert torch.equal(y, out)
    for a, b in zip((gu, d), again):
        for p, q in zip(a or [], b or []):
            assert torch.equal(p.stamp, q.stamp) and torch.equal(p.meta, q.meta)
    assert ctx.device_status() == 0
    ctx.close()
    plain.close()


@pytest.mark.parametrize("policy", ["lru", "lfu"])
@pytest.mark.parametrize("wtype,d_model,d_ff,rho,launches", [
    # updates that ride: columns of the three variants, and a launch of two waves (149 segments: its last block waits for
    # blocks that start when others end)
    (di.W_BF16, 544, 8192, 0.25, 0), (di.W_BF16, 544, 8224, 0.25, 0), (di.W_BF16, 1056, 20480, 0.2, 0), (di.W_BF16, 544, 20512, 0.2, 0),
    (di.W_F32, 19072, 128, 0.5, 0),
    # products on all 148 SMs: 4, 2 and 1 row parts
    (di.W_BF16, 9472, 640, 0.5, 2), (di.W_BF16, 18944, 256, 0.5, 2), (di.W_F32, 18944, 128, 0.5, 2),
])
def test_updates_ride_where_a_down_product_leaves_sms(wtype, d_model, d_ff, rho, launches, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    if ctx.sm_count != 148:
        pytest.skip("shapes chosen for 148 SMs")
    lw = _layer(d_model, d_ff, wtype, d_model + d_ff)
    w = upload_layer(dip, ctx, lw)
    refs = [oracle.Cache(d, int(0.4 * d), policy) for d in (d_model, d_ff)]
    mine = [dip.CacheState(d, int(0.4 * d), "cuda", policy) for d in (d_model, d_ff)]
    for t in range(3):
        kinds = launch_kinds(ctx, lambda: check_step(dip, ctx, lw, w, di.heavy_tail_vector(t, d_model), int(rho * d_model), int(rho * d_ff),
                                                     0.2, *refs, *mine))
        assert sorted(kinds) == ["cache_update"] * launches + ["gemv_down", "gemv_gate_up"]
    assert ctx.device_status() == 0
    ctx.close()


def test_rows_of_one_segment_leave_room_for_both_updates():
    """A part per SM would leave none: 5000 rows of 256 BF16 outputs."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d_model, d_ff = 256, 8192
    lw = _layer(d_model, d_ff, di.W_BF16, 5)
    w = upload_layer(dip, ctx, lw)
    refs = [oracle.Cache(d, d // 2) for d in (d_model, d_ff)]
    mine = [dip.CacheState(d, d // 2, "cuda") for d in (d_model, d_ff)]
    for t in range(2):
        kinds = launch_kinds(ctx, lambda: check_step(dip, ctx, lw, w, di.heavy_tail_vector(t, d_model), 100, 5000, 0.3, *refs, *mine))
        assert kinds == ["gemv_gate_up", "gemv_down"]           # (no launch for the updates)
    ctx.close()


@pytest.mark.parametrize("n_tied", [1, 2, 7, 8, 9, 128, 129, 256, 257])
def test_stand_alone_selects_with_threshold_bins_of_every_size(n_tied):
    """Eight columns are the last that one thread each ranks, 128 the last that the block ranks in one go; half of them have
    equal keys, the others keys of the same 16 bits."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d, above = 1000, 100
    rng = np.random.default_rng(n_tied)
    tied = np.full(n_tied, 1.5, np.float32)
    tied[::2] = (tied[::2].view(np.uint32) + rng.integers(0, 1000, tied[::2].size).astype(np.uint32)).view(np.float32)
    x = np.concatenate([rng.uniform(4.0, 9.0, above), tied, rng.uniform(0.01, 1.0, d - above - n_tied)]).astype(np.float32)
    x = (rng.permutation(x) * rng.choice([-1, 1], d)).astype(np.float32)
    bits = torch.zeros((d + 31) // 32, dtype=torch.int32, device="cuda")
    for kept in sorted({1, (n_tied + 1) // 2, n_tied}):
        idx = torch.zeros(above + kept, dtype=torch.int32, device="cuda")
        dip.dip_mask_topk(ctx, torch.from_numpy(x).cuda(), above + kept, bits, idx)
        m, i = oracle.dip_ca_mask(x, above + kept, 1.0, None)
        assert np.array_equal(bits_to_mask(bits, d), m) and np.array_equal(idx.cpu().numpy(), i), kept
    ctx.close()


@pytest.mark.parametrize("wtype", [di.W_BF16, di.W_F32])
@pytest.mark.parametrize("where", ["weights", "x"])
def test_values_that_are_not_finite(wtype, where):
    """NaN of any bit pattern (all ones is the mark of an empty box) and infinities give what the kernel gives that adds its
    row parts up in memory, and no wait runs out."""
    import paper_2412_01380_b200 as dip
    d_model, d_ff = 256, 1536
    lw = _layer(d_model, d_ff, wtype, 77)
    x = di.heavy_tail_vector(8, d_model)
    if where == "weights":
        for m in (lw.gate, lw.up, lw.down):
            m = m.reshape(-1).view(np.uint32 if wtype == di.W_F32 else np.uint16)
            bits = (0xffffffff, 0x7fc00000, 0x7f800000, 0xff800000) if wtype == di.W_F32 else (0xffff, 0x7fc0, 0x7f80, 0xff80)
            for i, v in enumerate(bits):
                m[m.size // 5 * (i + 1)] = v
    else:
        x.view(np.uint32)[[3, 50, 99]] = (0xffffffff, 0x7f800000, 0x7fc00001)
    got = []
    for kw in ({}, {"gemv_copy_ring": True}):
        ctx = dip.Context(0, **kw)
        w = upload_layer(dip, ctx, lw)
        y, h = torch.empty(d_model, device="cuda"), torch.empty(d_ff, device="cuda")
        bits = torch.zeros(d_ff // 32, dtype=torch.int32, device="cuda")
        dip.dip_mlp_step(ctx, w, torch.from_numpy(x).cuda(), 128, 1056, 1.0, None, None, y, h=h, mask_h=bits)
        torch.cuda.synchronize()
        assert ctx.device_status() == 0
        got.append((h.cpu().numpy(), bits_to_mask(bits, d_ff), y.cpu().numpy()))
        ctx.close()
    (h0, m0, y0), (h1, m1, y1) = got
    assert not np.isfinite(h0).all() and not np.isfinite(y0).all()
    assert np.array_equal(m0, m1)
    for a, b in ((h0, h1), (y0, y1)):
        ok = np.isfinite(a)
        assert np.array_equal(a[~ok], b[~ok], equal_nan=True) and (not ok.any() or rel_err(a[ok], b[ok]) <= REL_TOL)


def test_rows_asked_for_before_the_select_are_kept_rows_for_every_gamma():
    """With nothing resident a gamma of 64 is a factor of all keys: the masks are those of gamma 1, and so are the rows that are read
    (asked for by the key alone, 4096 rows of 44 KB instead of 1024 were: 135 MB, 20 us and more)."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d_model, d_ff = 4096, 11008
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    layers = []
    for _ in range(2):
        mats = [torch.randn(s, generator=gen, device="cuda").mul_(0.02).bfloat16() for s in ((d_ff, d_model), (d_ff, d_model), (d_model, d_ff))]
        layers.append(dip.dip_pack_weights(ctx, dip.W_BF16, d_model, d_ff, *mats))
    x = torch.randn(d_model, generator=gen, device="cuda")
    us, out = {}, {}
    for gamma in (1.0, 64.0):
        caches = [[dip.CacheState(d, 0, "cuda") for _ in layers] for d in (d_model, d_ff)]
        stack = dip.Stack(layers, *caches)
        out[gamma] = torch.empty_like(x)
        us[gamma] = graph_us(lambda: dip.dip_stack_step(ctx, stack, x, d_model // 4, d_ff // 4, gamma, out[gamma]))
    assert torch.equal(out[1.0], out[64.0])
    assert us[64.0] < us[1.0] + 8, us
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("policy", [None, "lru"])
@pytest.mark.parametrize("wtype,d_model,d_ff,rho", [
    (di.W_BF16, 8224, 1056, 0.23),       # gate/up rows of 8 MB and just above it: all of them are asked for; the wide variant
    (di.W_BF16, 8224, 1056, 0.24), (di.W_BF16, 4096, 6144, 0.19), (di.W_F32, 2048, 4096, 0.31),   # few kept; 20 MB
    (di.W_BF16, 1024, 16416, 0.96),      # down rows of 32 MB, with updates beside them
])
def test_rows_asked_for_ahead(wtype, d_model, d_ff, rho, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    lw = _layer(d_model, d_ff, wtype, 12)
    w = upload_layer(dip, ctx, lw)
    k_x, k_h = int(rho * d_model), int(rho * d_ff)
    refs = [oracle.Cache(d, d // 2, policy) if policy else None for d in (d_model, d_ff)]
    mine = [dip.CacheState(d, d // 2, "cuda", policy) if policy else None for d in (d_model, d_ff)]
    for t in range(2):
        check_step(dip, ctx, lw, w, di.heavy_tail_vector(300 + t, d_model), k_x, k_h, 0.2 if policy else 1.0, *refs, *mine)
    assert ctx.device_status() == 0
    ctx.close()
