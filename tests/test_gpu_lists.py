"""Products from index lists, which each of their blocks turns into a bit set for itself, and the lists that the mask calls leave:
lists in any order, with columns named twice and columns outside the input, list lengths around a trip of loads, and masks
whose last word or byte is not full."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, bits_to_mask, cache_equal, graph_us, oracle_mats, rel_err, upload_layer

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wtype,d_model,d_ff,ring", [
    (di.W_BF16, 288, 8224, False), (di.W_F32, 96, 1056, False), (di.W_INT4_G128, 256, 8320, False), (di.W_BF16, 288, 1056, True),
])
def test_product_from_any_list(wtype, d_model, d_ff, ring):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0, gemv_copy_ring=ring)
    lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=d_ff, d_model=d_model, d_ff=d_ff, wtype=wtype, n_layers=1), 0)
    w = upload_layer(dip, ctx, lw)
    Wg, Wu, Wd = oracle_mats(lw)
    rng = np.random.default_rng(d_ff)
    for which, d in ((0, d_model), (1, d_ff)):
        v = di.heavy_tail_vector(7 + which, d)
        out = torch.empty(d_ff if which == 0 else d_model, device="cuda")
        for n in sorted({1, 2, 31, d // 3, min(d, 1024), min(d, 1025), min(d, 8192), d}):
            cols = rng.choice(d, n, replace=False).astype(np.int32)
            lists = [np.sort(cols), cols, np.where(rng.random(n) < 0.3, cols[0], cols).astype(np.int32)]
            if n > 2:
                bad = cols.copy()
                bad[: n // 2] = np.array([-1, d, d + 31, 2 ** 31 - 1], dtype=np.int32)[np.arange(n // 2) % 4]
                lists.append(bad)
            for li in lists:
                m = np.zeros(d, dtype=np.uint8)
                m[li[(li >= 0) & (li < d)]] = 1
                product = dip.dip_sparse_gemv_gate_up if which == 0 else dip.dip_sparse_gemv_down
                product(ctx, w, torch.from_numpy(v).cuda(), torch.from_numpy(li).cuda(), n, None, out)
                want = oracle.glu(oracle.masked_matvec(Wg, v, m), oracle.masked_matvec(Wu, v, m)) if which == 0 else \
                    oracle.masked_matvec(Wd, v, m)
                assert rel_err(out.cpu().numpy(), want) <= REL_TOL, (which, n)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("policy", ["lru", "lfu"])
@pytest.mark.parametrize("d", [1, 7, 33, 1000, 8185, 8192, 8193, 20481, 32768])
def test_mask_calls_leave_lists(d, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    bits = torch.zeros((d + 31) // 32, dtype=torch.int32, device="cuda")
    for k in sorted({1, max(1, d // 3), d}):
        cap = d // 2
        idx = torch.full((k,), -7, dtype=torch.int32, device="cuda")
        ref, g = oracle.Cache(d, cap, policy), dip.CacheState(d, cap, "cuda", policy)
        for t in range(3):
            x = di.heavy_tail_vector(50 + t, d)
            if t == 2:
                x = np.sign(x).astype(np.float32)                                    # one magnitude: the general select
            dip.dip_ca_mask(ctx, torch.from_numpy(x).cuda(), k, 0.2, g, bits, idx)
            m, want = oracle.dip_ca_mask(x, k, 0.2, ref)
            assert np.array_equal(bits_to_mask(bits, d), m) and np.array_equal(idx.cpu().numpy(), want), (k, t)
            assert cache_equal(g, ref), (k, t)
        xs = np.stack([di.heavy_tail_vector(60 + t, d) for t in range(3)])
        rows = torch.full((3, k), -7, dtype=torch.int32, device="cuda")
        dip.dip_mask_topk(ctx, torch.from_numpy(xs).cuda(), k, None, rows)
        for r in range(3):
            assert np.array_equal(rows[r].cpu().numpy(), oracle.dip_ca_mask(xs[r], k, 1.0, None)[1]), (k, r)
    ctx.close()


@pytest.mark.parametrize("policy", [None, "lru", "lfu"])
@pytest.mark.parametrize("d", [2049, 8192, 8224, 32768])
def test_lists_around_the_longest_that_is_written_directly(d, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    bits = torch.zeros((d + 31) // 32, dtype=torch.int32, device="cuda")
    for k in (2048, 2049):
        idx = torch.full((k,), -7, dtype=torch.int32, device="cuda")
        ref = g = None
        if policy:
            ref, g = oracle.Cache(d, d // 2, policy), dip.CacheState(d, d // 2, "cuda", policy)
        for t in range(2):
            x = di.heavy_tail_vector(80 + t, d)
            if policy:
                dip.dip_ca_mask(ctx, torch.from_numpy(x).cuda(), k, 0.2, g, bits, idx)
            else:
                dip.dip_mask_topk(ctx, torch.from_numpy(x).cuda(), k, bits, idx)
            m, want = oracle.dip_ca_mask(x, k, 0.2 if policy else 1.0, ref)
            assert np.array_equal(bits_to_mask(bits, d), m) and np.array_equal(idx.cpu().numpy(), want), (k, t)
            assert not policy or cache_equal(g, ref), (k, t)
    ctx.close()


def test_a_long_list_costs_little_beside_its_mask():
    """32768 entries are 128 KB: a few microseconds out of one SM (written 4 bytes of a sector at a time they took over 30)."""
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    d = 32768
    x = torch.from_numpy(di.heavy_tail_vector(90, d)).cuda()
    bits, idx = torch.zeros(d // 32, dtype=torch.int32, device="cuda"), torch.zeros(d, dtype=torch.int32, device="cuda")
    without = graph_us(lambda: dip.dip_mask_topk(ctx, x, d, bits, None))
    assert graph_us(lambda: dip.dip_mask_topk(ctx, x, d, bits, idx)) < without + 15
    ctx.close()
