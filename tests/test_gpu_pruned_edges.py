"""Gate / Up pruning where the ranking product leaves 16-bit keys for the select: masses of equal keys (the general select), one kept
neuron, all of them, rows that need several and ragged trips of loads, and more kept rows than warps."""
import numpy as np
import pytest
import torch

import dip_inputs as di
import oracle
from gpu_util import REL_TOL, bits_to_mask, oracle_mats, rel_err
from test_gpu_neuron_pruning import _neuron_weights, _silu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("by", ["gate", "up"])
@pytest.mark.parametrize("wtype,d_model,d_ff", [(di.W_BF16, 2720, 4128), (di.W_F32, 1312, 4096), (di.W_BF16, 96, 8192)])
def test_pruning_from_the_products_keys(wtype, d_model, d_ff, by):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    wl = di.WORKLOADS["phi3_mini"].scaled(seed=d_ff, d_model=d_model, d_ff=d_ff, wtype=wtype)
    lw = di.layer_weights(wl, 0)
    nw = _neuron_weights(dip, lw)
    Wg, Wu, Wd = oracle_mats(lw)
    x0 = di.token_inputs(wl, n_tokens=1, batch=1, d=d_model)[0, 0]
    ones = np.ones(d_model, dtype=np.uint8)
    for x in (x0, np.zeros_like(x0)):                       # (p = 0 everywhere: the first k neurons are kept)
        g, u = oracle.masked_matvec(Wg, x, ones), oracle.masked_matvec(Wu, x, ones)
        for k in sorted({1, 33, d_ff // 4, min(d_ff, 4800), d_ff}):
            y, p, h = (torch.empty(n, device="cuda") for n in (d_model, d_ff, d_ff))
            mask = torch.zeros(d_ff // 32, dtype=torch.int32, device="cuda")
            idx = torch.zeros(k, dtype=torch.int32, device="cuda")
            dip.dip_mlp_step_neuron_pruned(ctx, nw, by, torch.from_numpy(x).cuda(), k, y, p=p, mask=mask, idx=idx, h=h)
            p_gpu, h_gpu = p.cpu().numpy(), h.cpu().numpy()
            m, idx_ref = oracle.dip_ca_mask(p_gpu, k, 1.0, None)
            assert np.array_equal(bits_to_mask(mask, d_ff), m) and np.array_equal(idx.cpu().numpy(), idx_ref)
            assert rel_err(p_gpu, _silu(g) if by == "gate" else u) <= REL_TOL
            assert rel_err(h_gpu, m * p_gpu.astype(np.float64) * (u if by == "gate" else _silu(g))) <= REL_TOL
            assert rel_err(y.cpu().numpy(), oracle.masked_matvec(Wd, h_gpu, m)) <= REL_TOL
    assert ctx.device_status() == 0
    ctx.close()
