"""The cache update of Algorithm 1 from states of any age, against the oracle: the kernel's variants by column count (8192
and 20480 columns are the last that the narrower ones take), row lengths that are no multiple of four or of 32,
eviction keys of one, two and three radix digits, and quotas that run out inside a group of ties."""
import numpy as np
import pytest

import dip_inputs as di
import oracle
from gpu_util import bits_to_mask, cache_equal, gpu_cache_from_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", ["lru", "lfu"])
@pytest.mark.parametrize("d,k,cap", [
    (5, 2, 3), (127, 40, 60), (129, 64, 64), (1030, 700, 200), (8192, 2048, 4096), (8193, 2000, 4100),
    (20480, 5000, 9000), (20481, 9000, 5000), (32768, 8192, 16384),
])
def test_update_from_states_of_any_age(d, k, cap, policy):
    import paper_2412_01380_b200 as dip
    ctx = dip.Context(0)
    bits = torch.zeros((d + 31) // 32, dtype=torch.int32, device="cuda")
    for step, oldest in ((7, 6), (5000, 4990), (5000, 40), (9000000, 8999000)):      # keys of 3, 13 and 24 bits; few ages
        rng = np.random.default_rng(d + step + oldest)
        ref = oracle.Cache(d, cap, policy)
        held = rng.choice(d, cap - (cap > 50) * 7, replace=False)                    # nearly full: free places, then evictions
        ref.stamp[held] = (step - rng.integers(0, oldest, held.size)).astype(np.int32)
        ref.count[:] = rng.integers(0, oldest, d).astype(np.int32) if policy == "lfu" else 0
        ref.n_resident[0], ref.step[0] = held.size, step
        g = gpu_cache_from_oracle(dip, ref)
        for t in range(3):
            x = di.heavy_tail_vector(50 + t, d)
            dip.dip_ca_mask(ctx, torch.from_numpy(x).cuda(), k, 0.2, g, bits, None)
            torch.cuda.synchronize()
            m, _ = oracle.dip_ca_mask(x, k, 0.2, ref)
            assert np.array_equal(bits_to_mask(bits, d), m), (step, t)
            assert cache_equal(g, ref), (step, t)
    ctx.close()
