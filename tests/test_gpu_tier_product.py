"""The two-tier product at the edges of its plan: parts of more rows than one list, as many parts as SMs, rows of one segment and of a
ragged one, budgets of nothing and of everything, and a tier whose slots lie outside its arena."""
import numpy as np
import pytest
import torch

import dip_inputs as di
import oracle
from gpu_util import check_step, upload_layer
from test_gpu_tiered import _check_tier, _layer, _tiers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wtype,d_model,d_ff,k_x,k_h,beta,steps", [
    (di.W_BF16, 4160, 9504, 4160, 9504, 0.5, 2),      # 75 segments, one part: 4160 misses, then hits and misses, in lists of 2048
    (di.W_BF16, 256, 8224, 200, 5000, 0.5, 4),        # down rows of one segment: a part per SM
    (di.W_F32, 96, 1056, 1, 33, 0.4, 4),              # ragged segments, one row
    (di.W_BF16, 288, 1056, 96, 400, 0.0, 3),          # nothing cached: every column a miss
    (di.W_BF16, 288, 1056, 96, 400, 1.0, 4),          # everything fits: hits only, after a while
    (di.W_INT4_G128, 384, 1152, 100, 500, 0.5, 4),    # (fetched by a launch of its own)
])
def test_tiers_of_every_plan(wtype, d_model, d_ff, k_x, k_h, beta, steps):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    lw = _layer(d_ff, d_model, d_ff, wtype)
    w = upload_layer(dip, ctx, lw)
    gate_up, down = w.gate_up.clone(), w.down.clone()
    g_gu, g_d, t_gu, t_d = _tiers(dip, w, k_x, k_h, beta, "lru", True)
    ref_gu, ref_d = oracle.Cache(d_model, g_gu.capacity, "lru"), oracle.Cache(d_ff, g_d.capacity, "lru")
    w.struct.gate_up = w.struct.down = None
    for x in di.token_inputs(di.WORKLOADS["phi3_mini"].scaled(seed=d_ff + 1), n_tokens=steps, batch=1, d=d_model)[:, 0]:
        check_step(dip, ctx, lw, w, x, k_x, k_h, 0.2, ref_gu, ref_d, g_gu, g_d, tiers=(t_gu, t_d))
        for t, packed, ref in ((t_gu, gate_up, ref_gu), (t_d, down, ref_d)):
            _check_tier(t, packed, ref, int(ref.counters[1]))
    assert ctx.device_status() == 0
    ctx.close()


def test_slots_outside_the_arena_are_reported_and_not_read():
    import paper_2412_01380_b200 as dip
    d_model, d_ff, k_x, k_h = 512, 1024, 128, 256
    ctx = dip.Context(0)
    lw = _layer(9, d_model, d_ff, di.W_BF16)
    w = upload_layer(dip, ctx, lw)
    g_gu, g_d, t_gu, t_d = _tiers(dip, w, k_x, k_h, 0.5, "lru", False)
    stamp = np.full(d_model, -1, dtype=np.int32)
    stamp[: g_gu.capacity] = 0
    g_gu.load(stamp, g_gu.capacity, 1)
    t_gu.slot[: g_gu.capacity] = 1 << 20
    x = torch.from_numpy(di.token_inputs(di.WORKLOADS["phi3_mini"].scaled(seed=3), 1, 1, d_model)[0, 0]).cuda()
    h = torch.empty(d_ff, device="cuda")
    dip.dip_mlp_step_tiered(ctx, w, t_gu, t_d, x, k_x, k_h, 0.2, torch.empty(d_model, device="cuda"), h=h)
    assert ctx.device_status() == 2 and int(t_gu.fetch[1]) == 0
    want = torch.empty(d_ff, device="cuda")
    c2 = dip.CacheState(d_model, g_gu.capacity, "cuda")
    c2.load(stamp, g_gu.capacity, 1)
    dip.dip_mlp_step(ctx, w, x, k_x, k_h, 0.2, c2, None, torch.empty(d_model, device="cuda"), h=want)
    assert torch.allclose(h, want, rtol=1e-4, atol=1e-5 * float(want.abs().max()))    # its columns came from the slow tier
    ctx.close()


def test_two_tier_products_round_no_more_than_two_products_did():
    """Root mean square error of h and y against 64 bits, of the columns that the step kept.  A sum of 256 (704) rows meets at most ten
    roundings: its chain in a warp, five levels over the warps, the parts with their errors carried along; each is 2.5e-8 rms.  h has two
    such sums and five roundings of its own: sqrt(25) x 2.5e-8, y sqrt(10) x 2.5e-8, and a third more for what is kept unevenly."""
    import paper_2412_01380_b200 as dip
    d_model, d_ff, k_x, k_h = 1024, 2816, 256, 704
    ctx = dip.Context(0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(17)
    mats = [torch.randn(s, generator=gen, device="cuda").mul_(0.02).bfloat16() for s in ((d_ff, d_model), (d_ff, d_model), (d_model, d_ff))]
    w = dip.dip_pack_weights(ctx, dip.W_BF16, d_model, d_ff, *mats)
    gate, up, down = [m.double() for m in mats]
    _, _, t_gu, t_d = _tiers(dip, w, k_x, k_h, 0.5, "lru", False)
    h, y = torch.empty(d_ff, device="cuda"), torch.empty(d_model, device="cuda")
    m_x, m_h = [torch.zeros(d // 32, dtype=torch.int32, device="cuda") for d in (d_model, d_ff)]

    def kept(v, bits):
        return v.double() * ((bits.view(-1, 1) >> torch.arange(32, device="cuda").int()) & 1).view(-1)

    errs = []
    x = torch.randn(d_model, generator=gen, device="cuda")
    for _ in range(12):
        x = 0.95 * x + 0.3 * torch.randn(d_model, generator=gen, device="cuda")
        dip.dip_mlp_step_tiered(ctx, w, t_gu, t_d, x, k_x, k_h, 0.2, y, mask_x=m_x, h=h, mask_h=m_h)
        want_h = torch.nn.functional.silu(gate @ kept(x, m_x)) * (up @ kept(x, m_x))
        want_y = down @ kept(h, m_h)
        errs.append([float((a.double() - b).norm() / b.norm()) for a, b in ((h, want_h), (y, want_y))])
    err_h, err_y = np.mean(errs, axis=0)
    assert err_h <= 4 / 3 * 5 * 2.5e-8 and err_y <= 4 / 3 * 10 ** 0.5 * 2.5e-8, (err_h, err_y)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("wtype,d_model,d_ff,k_x,k_h,beta,ring", [
    (di.W_INT4_G128, 256, 5120, 200, 900, 0.5, 0),     # rows of two pieces and a half, of one that is not full
    (di.W_INT4_G128, 640, 2048, 300, 1500, 0.0, 0),    # nothing cached: no row has a slot
    (di.W_BF16, 1024, 1056, 700, 1000, 0.6, 1),        # more pieces than warps, behind the copy ring
    (di.W_F32, 64, 4128, 1, 40, 1.0, 1),               # one miss, then hits only
])
def test_fetched_rows_reach_their_slots(wtype, d_model, d_ff, k_x, k_h, beta, ring):
    """Launches that fetch the misses for products that do not read the slow tier themselves."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0, gemv_copy_ring=ring)
    lw = _layer(d_ff, d_model, d_ff, wtype)
    w = upload_layer(dip, ctx, lw)
    gate_up, down = w.gate_up.clone(), w.down.clone()
    g_gu, g_d, t_gu, t_d = _tiers(dip, w, k_x, k_h, beta, "lru", True)
    ref_gu, ref_d = oracle.Cache(d_model, g_gu.capacity, "lru"), oracle.Cache(d_ff, g_d.capacity, "lru")
    w.struct.gate_up = w.struct.down = None
    for x in di.token_inputs(di.WORKLOADS["phi3_mini"].scaled(seed=d_ff + 2), n_tokens=4, batch=1, d=d_model)[:, 0]:
        check_step(dip, ctx, lw, w, x, k_x, k_h, 0.2, ref_gu, ref_d, g_gu, g_d, tiers=(t_gu, t_d))
        for t, packed, ref in ((t_gu, gate_up, ref_gu), (t_d, down, ref_d)):
            _check_tier(t, packed, ref, int(ref.counters[1]))
    assert ctx.device_status() == 0
    ctx.close()
