"""Contexts, options and failure paths of the C ABI on the GPU: workspace sizing, rejected
arguments (nothing is launched), and the bounded wait that every copy-ring kernel relies on."""
import numpy as np
import pytest
import torch

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, cache_equal, check_step, rel_err, upload_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dip():
    import paper_2412_01380_b200 as m
    return m


def test_bounded_wait_runs_out_and_the_context_stays_usable(dip):
    """A wait that nothing will ever satisfy gives up after its limit: the kernel returns, the
    sticky status word reads DEVICE_WAIT_TIMEOUT, and after a reset the same context computes a
    correct step."""
    c = dip.Context(0)
    try:
        assert c.device_status() == dip.DEVICE_OK
        waited = torch.zeros(1, dtype=torch.int64, device="cuda")
        c.selftest_bounded_wait(1000, waited)                  # one millisecond
        assert c.device_status() == dip.DEVICE_WAIT_TIMEOUT
        assert 1_000_000 <= int(waited.item()) < 200_000_000   # it waited its limit, and not much more
        assert c.device_status() == dip.DEVICE_WAIT_TIMEOUT    # sticky
        c.reset_device_status()
        assert c.device_status() == dip.DEVICE_OK
        # the copy-ring kernel (INT4) on the same context right after
        wl = di.WORKLOADS["llama3_8b_int4"].scaled(seed=3, d_model=512, d_ff=1024)
        lw = di.layer_weights(wl, 0)
        w = upload_layer(dip, c, lw)
        x = di.token_inputs(wl, n_tokens=1, batch=1)[0, 0]
        check_step(dip, c, lw, w, x, wl.k_x, wl.k_h, 1.0, None, None, None, None)
        assert c.device_status() == dip.DEVICE_OK
        with pytest.raises(dip.DipError):
            c.selftest_bounded_wait(0)
        with pytest.raises(dip.DipError):
            c.selftest_bounded_wait(2_000_000)
    finally:
        torch.cuda.synchronize()
        c.close()


@pytest.mark.parametrize("policy", ["lru", "lfu"])
@pytest.mark.parametrize("d", [1056, 17920])
def test_block_waits_run_out_and_a_reset_mends_the_context(dip, d, policy):
    """Row parts and readers of a cache state that come too late: status 1, the state as it was, and after a reset the same
    boxes and the same counter serve correct steps (33 parts per segment, updates that ride along)."""
    c = dip.Context(0)
    try:
        ref, st = oracle.Cache(d, d // 2, policy), dip.CacheState(d, d // 2, "cuda", policy)
        bits = torch.zeros((d + 31) // 32, dtype=torch.int32, device="cuda")
        for t in range(3):
            v = di.heavy_tail_vector(20 + t, d)
            dip.dip_ca_mask(c, torch.from_numpy(v).cuda(), d // 3, 0.2, st, bits, None)
            oracle.dip_ca_mask(v, d // 3, 0.2, ref)
        dip.dip_mask_topk(c, torch.from_numpy(di.heavy_tail_vector(30, d)).cuda(), d // 3, bits, None)
        assert c.device_status() == dip.DEVICE_OK and cache_equal(st, ref)
        c.selftest_block_waits(1000, st, bits)
        assert c.device_status() == dip.DEVICE_WAIT_TIMEOUT
        assert cache_equal(st, ref)
        c.reset_device_status()
        lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=4, d_model=256, d_ff=1536, n_layers=1), 0)
        w = upload_layer(dip, c, lw)
        refs = [oracle.Cache(n, n // 2) for n in (256, 1536)]
        mine = [dip.CacheState(n, n // 2, "cuda") for n in (256, 1536)]
        for t in range(2):
            check_step(dip, c, lw, w, di.heavy_tail_vector(40 + t, 256), 128, 1056, 0.2, *refs, *mine)
        assert c.device_status() == dip.DEVICE_OK
        for bad in (0, 2_000_000):
            with pytest.raises(dip.DipError):
                c.selftest_block_waits(bad, st, bits)
    finally:
        torch.cuda.synchronize()
        c.close()


def test_options_size_the_workspace_and_pick_the_kernels(dip):
    wl = di.WORKLOADS["phi3_mini"].scaled(seed=8, d_model=1024, d_ff=2816)
    lw = di.layer_weights(wl, 0)
    x = di.token_inputs(wl, n_tokens=1, batch=1)[0, 0]
    free0 = torch.cuda.mem_get_info()[0]
    small = dip.Context(0, max_d=2816, max_batch=1)
    used_small = free0 - torch.cuda.mem_get_info()[0]
    try:
        w = upload_layer(dip, small, lw)
        check_step(dip, small, lw, w, x, wl.k_x, wl.k_h, 1.0, None, None, None, None)
        # beyond what the workspace was sized for
        big = torch.zeros(4096, device="cuda")
        with pytest.raises(dip.DipError) as e:
            dip.dip_mask_topk(small, big, 8, torch.zeros(128, dtype=torch.int32, device="cuda"), None)
        assert e.value.status == dip.ERR_WORKSPACE
        with pytest.raises(dip.DipError) as e:
            xb = torch.zeros((2, 1024), device="cuda")
            dip.dip_mlp_step(small, w, xb, 8, 8, 1.0, None, None, torch.zeros((2, 1024), device="cuda"))
        assert e.value.status == dip.ERR_WORKSPACE
    finally:
        torch.cuda.synchronize()
        small.close()
    free1 = torch.cuda.mem_get_info()[0]
    full = dip.Context(0)
    used_full = free1 - torch.cuda.mem_get_info()[0]
    full.close()
    assert used_small < used_full
    # forced kernels: copy ring with each segment width, and the 16-bit keys at every size
    for kw in ({"gemv_copy_ring": True}, {"gemv_copy_ring": True, "gemv_segment_bytes": 512},
               {"gemv_copy_ring": True, "gemv_segment_bytes": 1024}, {"coarse_min_d": -1},
               {"wait_limit_us": 1}):            # (for copies: the default kernels make none)
        c = dip.Context(0, **kw)
        try:
            w = upload_layer(dip, c, lw)
            ref_gu, ref_d = oracle.Cache(1024, 512), oracle.Cache(2816, 1408)
            g_gu, g_d = dip.CacheState(1024, 512, "cuda"), dip.CacheState(2816, 1408, "cuda")
            for t in range(2):
                check_step(dip, c, lw, w, x, wl.k_x, wl.k_h, 0.2, ref_gu, ref_d, g_gu, g_d)
            assert c.device_status() == dip.DEVICE_OK
        finally:
            torch.cuda.synchronize()
            c.close()
    for bad in ({"max_d": 40000}, {"max_batch": 17}, {"gemv_segment_bytes": 100}, {"wait_limit_us": -1}):
        with pytest.raises(dip.DipError):
            dip.Context(0, **bad)


def test_misaligned_pointers_are_rejected_before_any_launch(dip):
    """Every vector and mask is read with 16-byte loads somewhere: a tensor slice at a 4-byte offset
    must come back as an error code, not as a misaligned-address fault."""
    c = dip.Context(0)
    try:
        wl = di.WORKLOADS["phi3_mini"].scaled(seed=9, d_model=256, d_ff=512)
        w = upload_layer(dip, c, di.layer_weights(wl, 0))
        f = lambda n: torch.zeros(n + 4, device="cuda")
        i = lambda n: torch.zeros(n + 4, dtype=torch.int32, device="cuda")
        x, y, h = f(256), f(256), f(512)
        mx, mh, idx = i(8), i(16), i(64)

        def rejected(fn):
            with pytest.raises(dip.DipError) as e:
                fn()
            assert e.value.status == dip.ERR_INVALID_ARG

        rejected(lambda: dip.dip_mask_topk(c, x[:256], 8, mx[1:9], None))
        st = dip.CacheState(256, 128, "cuda")
        rejected(lambda: dip.dip_ca_mask(c, x[:256], 8, 0.2, st, mx[1:9], None))
        rejected(lambda: dip.dip_sparse_gemv_gate_up(c, w, x[:256], None, 64, mx[1:9], h[:512]))
        rejected(lambda: dip.dip_sparse_gemv_gate_up(c, w, x[1:257], None, 64, mx[:8], h[:512]))
        rejected(lambda: dip.dip_sparse_gemv_down(c, w, h[:512], None, 64, mh[1:17], y[:256]))
        rejected(lambda: dip.dip_sparse_gemv_down(c, w, h[:512], None, 64, mh[:16], y[1:257]))
        rejected(lambda: dip.dip_mlp_step(c, w, x[:256], 64, 128, 1.0, None, None, y[:256], mask_x=mx[1:9]))
        rejected(lambda: dip.dip_mlp_step(c, w, x[:256], 64, 128, 1.0, None, None, y[:256], mask_h=mh[1:17]))
        rejected(lambda: dip.dip_mlp_step(c, w, x[:256], 64, 128, 1.0, None, None, y[:256], h=h[1:513]))
        rejected(lambda: dip.dip_residual_rmsnorm(c, x[1:257], y[:256], x[:256]))
        rejected(lambda: dip.dip_residual_rmsnorm(c, x[:256], y[1:257], x[:256]))
        rejected(lambda: dip.dip_residual_rmsnorm(c, x[:256], y[:256], x[1:257]))
        stack = dip.Stack([w])
        rejected(lambda: dip.dip_stack_step(c, stack, x[1:257], 64, 128, 1.0, y[:256]))
        rejected(lambda: dip.dip_stack_step(c, stack, x[:256], 64, 128, 1.0, y[1:257]))
        torch.cuda.synchronize()
        # and the aligned calls still work on the same context
        dip.dip_mlp_step(c, w, x[:256], 64, 128, 1.0, None, None, y[:256], mask_x=mx[:8], mask_h=mh[:16], h=h[:512])
        torch.cuda.synchronize()
        assert c.device_status() == dip.DEVICE_OK
    finally:
        torch.cuda.synchronize()
        c.close()


def test_a_new_context_serves_any_stream_at_once(dip):
    """The first call on a context, on a stream that the default one does not order, finds the workspace set up."""
    lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=6, d_model=256, d_ff=1536, n_layers=1), 0)
    first = dip.Context(0)
    w = upload_layer(dip, first, lw)
    x = torch.from_numpy(di.heavy_tail_vector(3, 256)).cuda()
    want = torch.empty(256, device="cuda")
    dip.dip_mlp_step(first, w, x, 128, 1056, 1.0, None, None, want)
    torch.cuda.synchronize()
    first.close()
    for _ in range(5):
        y = torch.empty(256, device="cuda")
        torch.cuda.synchronize()
        c = dip.Context(0)
        s = torch.cuda.Stream()                                # (torch's streams do not wait for the default stream)
        with torch.cuda.stream(s):
            dip.dip_mlp_step(c, w, x, 128, 1056, 1.0, None, None, y)
            assert c.device_status() == dip.DEVICE_OK
        assert torch.equal(y, want)
        torch.cuda.synchronize()
        c.close()


@pytest.mark.parametrize("wtype", [di.W_BF16, di.W_INT4_G128])
def test_a_stack_with_a_bad_block_launches_nothing(dip, wtype):
    """A cache state that only the last block refuses: an error code, no launch, states untouched; the next good call is right."""
    c = dip.Context(0)
    try:
        wl = di.WORKLOADS["phi3_mini"].scaled(seed=12, d_model=256, d_ff=640, wtype=wtype, n_layers=3)
        ws = [upload_layer(dip, c, di.layer_weights(wl, l)) for l in range(3)]
        caches = [[dip.CacheState(d, d // 2, "cuda") for _ in range(3)] for d in (256, 640)]
        x, y = torch.from_numpy(di.heavy_tail_vector(1, 256)).cuda(), torch.empty(256, device="cuda")
        for which in (0, 1):
            stack = dip.Stack(ws, *caches)
            arr = (stack.gu_arr, stack.d_arr)[which]
            arr[2].capacity = arr[2].d + 1
            c.trace_begin()
            with pytest.raises(dip.DipError) as e:
                dip.dip_stack_step(c, stack, x, 64, 160, 0.2, y)
            assert e.value.status == dip.ERR_INVALID_ARG
            assert c.trace_read() == []
            c.trace_end()
        with pytest.raises(dip.DipError) as e:
            dip.dip_stack_step(c, dip.Stack(ws, *caches), x, 64, 641, 0.2, y)
        assert e.value.status == dip.ERR_INVALID_ARG
        with pytest.raises(dip.DipError) as e:
            dip.dip_stack_step(c, dip.Stack(ws, *caches), x.expand(2, 256).contiguous(), 64, 160, 0.2, y.expand(2, 256).contiguous())
        assert e.value.status == dip.ERR_UNSUPPORTED
        assert all(int(s.meta.abs().sum()) == 0 and int(s.stamp.max()) == -1 for half in caches for s in half)
        dip.dip_stack_step(c, dip.Stack(ws, *caches), x, 64, 160, 0.2, y)
        torch.cuda.synchronize()
        assert all(int(s.meta[1]) == 1 for half in caches for s in half) and c.device_status() == dip.DEVICE_OK
    finally:
        torch.cuda.synchronize()
        c.close()


def test_every_kind_of_block_wait_runs_out(dip):
    """The self-test's waits come one after another where they are of another kind (row parts and readers; the moves of a two-tier launch;
    row parts four sums at a time): each takes its limit.  After a reset a two-tier step and a batch, which use the same words and
    boxes, are right."""
    c = dip.Context(0)
    try:
        d_model, d_ff, k_x, k_h = 512, 2048, 256, 1024
        lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=6, d_model=d_model, d_ff=d_ff, n_layers=1), 0)
        w = upload_layer(dip, c, lw)
        st, bits = dip.CacheState(d_ff, d_ff // 2, "cuda"), torch.zeros(d_ff // 32, dtype=torch.int32, device="cuda")
        limit_us = 3000
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        c.selftest_block_waits(limit_us, st, bits)
        b.record()
        assert c.device_status() == dip.DEVICE_WAIT_TIMEOUT
        assert 3 * limit_us <= a.elapsed_time(b) * 1e3 <= 4 * limit_us
        c.reset_device_status()

        refs = [oracle.Cache(n, n // 2) for n in (d_model, d_ff)]
        mine = [dip.CacheState(n, n // 2, "cuda") for n in (d_model, d_ff)]
        tiers = [dip.Tier(s, p.cpu().pin_memory(), p.numel() // s.d, k, "cuda") for s, p, k in zip(mine, (w.gate_up, w.down), (k_x, k_h))]
        for t in range(2):
            check_step(dip, c, lw, w, di.heavy_tail_vector(60 + t, d_model), k_x, k_h, 0.2, *refs, *mine, tiers=tiers)
        xs = np.stack([di.heavy_tail_vector(70 + t, d_model) for t in range(4)])
        ys, y = torch.empty((4, d_model), device="cuda"), torch.empty(d_model, device="cuda")
        dip.dip_mlp_step(c, w, torch.from_numpy(xs).cuda(), k_x, k_h, 1.0, None, None, ys)
        for t in range(4):
            dip.dip_mlp_step(c, w, torch.from_numpy(xs[t]).cuda(), k_x, k_h, 1.0, None, None, y)
            assert rel_err(ys[t].cpu().numpy(), y.cpu().numpy()) <= REL_TOL
        assert c.device_status() == dip.DEVICE_OK
    finally:
        torch.cuda.synchronize()
        c.close()
