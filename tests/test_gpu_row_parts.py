"""Row parts of narrow products, whose sums meet in the last part's block: one part, as many as one trip collects (9 parts
are 8 boxes), one more, several trips' worth, and a part per SM, for rows of one and two 512-byte segments.  Products from
a list, from bit sets of two tokens, and of a step that selects for itself, against the oracle."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, check_step, oracle_mats, rel_err, upload_layer

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = [1, 31, 32, 63, 64, 287, 288, 319, 320, 1055, 1056, 1700, 4703, 5000, 8192]


@pytest.mark.parametrize("wtype,d_model", [(di.W_BF16, 256), (di.W_BF16, 288), (di.W_F32, 96), (di.W_F32, 256)])
def test_down_products_of_every_number_of_parts(wtype, d_model):
    import paper_2412_01380_b200 as dip
    d_ff = 8192
    ctx = dip.Context(0)
    lw = di.layer_weights(di.WORKLOADS["phi3_mini"].scaled(seed=d_model, d_model=d_model, d_ff=d_ff, wtype=wtype, n_layers=1), 0)
    w = upload_layer(dip, ctx, lw)
    Wd = oracle_mats(lw)[2]
    h = np.stack([di.heavy_tail_vector(900 + b, d_ff) for b in range(2)])
    x = di.heavy_tail_vector(950, d_model)
    for n in ROWS:
        masks = np.stack([oracle.dip_ca_mask(v, n, 1.0, None)[0] for v in h])
        want = [oracle.masked_matvec(Wd, v, m) for v, m in zip(h, masks)]
        idx = torch.from_numpy(np.flatnonzero(masks[0]).astype(np.int32)).cuda()
        y = torch.empty(d_model, device="cuda")
        dip.dip_sparse_gemv_down(ctx, w, torch.from_numpy(h[0]).cuda(), idx, n, None, y)
        assert rel_err(y.cpu().numpy(), want[0]) <= REL_TOL, n
        bits = torch.from_numpy(np.packbits(masks, axis=1, bitorder="little").view(np.int32)).cuda()
        y2 = torch.empty(2, d_model, device="cuda")
        union = int((masks[0] | masks[1]).sum())
        dip.dip_sparse_gemv_down(ctx, w, torch.from_numpy(h).cuda(), None, union, bits, y2)
        for b in range(2):
            assert rel_err(y2[b].cpu().numpy(), want[b]) <= REL_TOL, (n, b)
        check_step(dip, ctx, lw, w, x, max(1, d_model // 3), n, 1.0, None, None, None, None)
    assert ctx.device_status() == 0
    ctx.close()
