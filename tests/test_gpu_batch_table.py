"""Batched products on the tensor cores, whose blocks share the making of a table of the tokens' values and send their row parts to
one of them: unions of a round, of less, of none in some parts, of all columns; as many parts as SMs and rows without parts; columns
that no multiple of 128 is; and every number of tokens."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, oracle_mats, rel_err, upload_layer

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
