"""Batched products on the tensor cores, which read a table of the tokens' values and send their row parts to one of their blocks:
unions of a round, of less, of none in some parts, of all columns; as many parts as SMs and rows without parts; columns
that no multiple of 128 is; every number of tokens; and what a wide row, a wide input and a short limit of the waits cost."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, graph_us, oracle_mats, rel_err, upload_layer

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_model,d_ff,batches", [(256, 8224, (3, 5, 16)), (1056, 2080, tuple(range(3, 17))), (288, 19008, (4, 9))])
def test_batched_products_from_masks(d_model, d_ff, batches):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=d_ff, d_model=d_model, d_ff=d_ff, wtype=di.W_BF16, n_layers=1), 0)
    w = upload_layer(dip, ctx, lw)
    Wg, Wu, Wd = oracle_mats(lw)
    for batch in batches:
        for which, d in ((0, d_model), (1, d_ff)):
            v = np.stack([di.heavy_tail_vector(70 * batch + b + which, d) for b in range(batch)])
            for k in sorted({1, 20, 64, d // 4, d}):
                masks = np.stack([oracle.dip_ca_mask(x, k, 1.0, None)[0] for x in v])
                if k == 20:
                    masks[1:] = masks[0]                                             # every token keeps the same columns
                bits = torch.from_numpy(np.packbits(masks, axis=1, bitorder="little").view(np.int32)).cuda()
                out = torch.empty(batch, d_ff if which == 0 else d_model, device="cuda")
                product = dip.dip_sparse_gemv_gate_up if which == 0 else dip.dip_sparse_gemv_down
                product(ctx, w, torch.from_numpy(v).cuda(), None, min(d, batch * k), bits, out)
                for b in {0, batch // 2, batch - 1}:
                    want = oracle.glu(oracle.masked_matvec(Wg, v[b], masks[b]), oracle.masked_matvec(Wu, v[b], masks[b])) \
                        if which == 0 else oracle.masked_matvec(Wd, v[b], masks[b])
                    assert rel_err(out[b].cpu().numpy(), want) <= REL_TOL, (batch, which, k, b)
    assert ctx.device_status() == 0
    ctx.close()


def test_batched_products_around_the_parts_that_are_added_up_apart():
    """Two segments in 1 to 74 parts, collected by one block or, from 16 parts and 96 KB on, by a launch behind."""
    test_batched_products_from_masks(288, 6176, (5, 6, 8))


def _product(dip, d_model, d_ff, which, batch, k, **options):
    """A call of one product, all tokens keeping the same k columns; its context and output."""
    ctx = dip.Context(0, **options)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d_ff + k)
    mats = [torch.randn(s, generator=gen, device="cuda").mul_(0.02).bfloat16() for s in ((d_ff, d_model), (d_ff, d_model), (d_model, d_ff))]
    w = dip.dip_pack_weights(ctx, dip.W_BF16, d_model, d_ff, *mats)
    d = d_model if which == 0 else d_ff
    v = torch.randn((batch, d), generator=gen, device="cuda")
    bits = torch.zeros((batch, (d + 31) // 32), dtype=torch.int32, device="cuda")
    dip.dip_mask_topk(ctx, v[0].contiguous(), k, bits[0], None)
    bits[1:] = bits[0]
    out = torch.empty((batch, d_ff if which == 0 else d_model), device="cuda")
    product = dip.dip_sparse_gemv_gate_up if which == 0 else dip.dip_sparse_gemv_down
    return ctx, out, lambda: product(ctx, w, v, None, k, bits, out), (mats, v, bits)


@pytest.mark.parametrize("batch", [4, 16])
def test_a_segment_more_than_sms_does_not_stall(batch):
    """One segment more than fits at a time takes a second wave, a few microseconds; no block waits for that wave to start."""
    import paper_2412_01380_b200 as dip
    us = {}
    for extra in (0, 64):
        ctx, _, call, _ = _product(dip, 288, 128 * dip.Context(0).sm_count + extra, 0, batch, 64)
        us[extra] = graph_us(call)
        assert ctx.device_status() == 0
        ctx.close()
    assert us[64] < us[0] + 30, us


@pytest.mark.parametrize("d_model,d_ff,which", [(256, 8192, 1), (8192, 256, 0)])
def test_few_rows_of_a_wide_input_take_no_longer_than_many(d_model, d_ff, which):
    import paper_2412_01380_b200 as dip
    us = {}
    for k in (64, 4096):
        ctx, _, call, _ = _product(dip, d_model, d_ff, which, 3, k)
        us[k] = graph_us(call)
        ctx.close()
    assert us[64] < us[4096] + 2, us


def test_a_short_limit_for_copies_bounds_copies_only():
    import paper_2412_01380_b200 as dip
    d_ff = 128 * dip.Context(0).sm_count + 64
    ctx, out, call, (mats, v, bits) = _product(dip, 288, d_ff, 0, 4, 64, wait_limit_us=60)
    call()
    assert ctx.device_status() == 0
    keep = torch.from_numpy(np.unpackbits(bits.cpu().numpy().view(np.uint8), axis=1, bitorder="little")[:, :288].astype(np.float64)).cuda()
    x = v.double() * keep
    want = torch.nn.functional.silu(x @ mats[0].double().t()) * (x @ mats[1].double().t())
    assert rel_err(out.cpu().numpy(), want.cpu().numpy()) <= REL_TOL
    ctx.close()


@pytest.mark.parametrize("d_model,batch,k", [(256, 16, 4096), (256, 16, 1024), (256, 8, 1024), (1024, 16, 4096)])
def test_many_parts_of_many_tokens_are_not_one_blocks_work(d_model, batch, k):
    """The parts of 3 tokens and of many: what lies between the two times is the collecting of the parts (15 us and more by one block)."""
    import paper_2412_01380_b200 as dip
    us = {}
    for b in (3, batch):
        ctx, _, call, _ = _product(dip, d_model, 8192, 1, b, k)
        us[b] = graph_us(call)
        assert ctx.device_status() == 0
        ctx.close()
    assert us[batch] < us[3] + (2 if batch == 16 else 0.7), us
