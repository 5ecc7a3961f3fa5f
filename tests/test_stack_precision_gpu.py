"""A stacked step's attention against 64 bits, row by row: what the output's rounding to bf16 leaves (half a unit of the
last place) and 2e-5 of the weighted mean of |v|.  The second part covers weights of 16 bits (2^-18), fp32 logits and
exponentials (1e-6) and fp32 sums of a few hundred products (1e-5); weights of 8 bits alone miss it by far.  Both kernel
shapes, and every way the residuals of the weights take: free columns (G <= 4), products of their own (narrow, G > 4),
free rows (wide).  V's infinities stay infinities."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [1, 2], ids=["wide", "narrow"])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 8])
def test_rows_against_64_bits(G, shape):
    import torch

    import paper_2609_03430_gb300 as ra

    L, KVH, D, lps = 3, 3, 128, [1500, 17, 700]
    B, H, n = len(lps), G * KVH, max(lps)
    g = torch.Generator("cuda").manual_seed(G)

    def rows(*s):
        return torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)

    cache = ra.RandomAttentionCache(L, H, KVH, D, lps, 64, 16, seed=1)
    ra.ra_set_attention_shape(cache.ctx, shape)
    K, V = rows(L, B, KVH, n, D), rows(L, B, KVH, n, D)
    V[1, 2, 1, 650, 5] = math.inf
    for l in range(L):
        ra.ra_prefill(cache.ctx, l, K[l].data_ptr(), V[l].data_ptr(), n)
    q, kn, vn = rows(L, B, H, D), rows(L, B, KVH, D), rows(L, B, KVH, D)
    out = torch.zeros_like(q)
    ra.ra_decode_step(cache.ctx, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), out.data_ptr())
    got = out.double().view(L, B, KVH, G, D)
    for b, lp in enumerate(lps):
        k = torch.cat([K[:, b, :, :lp], kn[:, b, :, None]], 2).double()
        v = torch.cat([V[:, b, :, :lp], vn[:, b, :, None]], 2).double()
        p = torch.softmax(q[:, b].double().view(L, KVH, G, D) @ k.transpose(2, 3) / math.sqrt(D), -1)
        ref, spread = p @ v, p @ v.abs()
        bound = torch.exp2(torch.floor(torch.log2(ref.abs())) - 8) + 2e-5 * spread
        inf = torch.isinf(ref)
        assert int(inf.sum()) == (G if b == 2 else 0)
        assert bool((got[:, b][inf] == ref[inf]).all())
        over = ((got[:, b] - ref).abs() > bound) & ~inf
        assert not bool(over.any()), (b, int(over.sum()), float(((got[:, b] - ref).abs() / bound)[~inf].max()))
    ra.ra_check_device(cache.ctx)
    cache.close()
