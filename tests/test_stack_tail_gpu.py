"""Long stacked launches hand out their last tiles in small chunks: every output row against the same step made
layer by layer (another launch form, one chunk per warp), on a stack just long enough and a longer one, ragged
prompts and heads that cross many chunks, over several steps (the claim counter is ready again each time)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,G", [(14, 4), (40, 8)], ids=["just", "long"])
def test_stacked_step_equals_layer_calls(L, G):
    import torch

    import paper_2609_03430_gb300 as ra

    KVH, K, r, D = 8, 8000, 64, 128
    lps = [700, 1500, 1, 64, 2000, 900, 333, 48, 1100]
    B, c = len(lps), K + r + 5
    g = torch.Generator("cuda").manual_seed(L)
    caches = [ra.RandomAttentionCache(L, G * KVH, KVH, D, lps, K, r, seed=1) for _ in range(2)]

    def rows(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)

    pos = torch.stack([lp + torch.arange(20000 * r + 5 - c, 20000 * r + 5, dtype=torch.int32) for lp in lps])
    pos = pos[:, None, :].expand(B, KVH, c).contiguous().cuda()
    for l in range(L):
        pk, pv, k, v = rows(B, KVH, max(lps), D), rows(B, KVH, max(lps), D), rows(B, KVH, c, D), rows(B, KVH, c, D)
        for x in caches:
            ra.ra_prefill(x.ctx, l, pk.data_ptr(), pv.data_ptr(), max(lps))
            ra.ra_restore(x.ctx, l, [20000 * r + 5] * B, [c] * B, pos.data_ptr(), k.data_ptr(), v.data_ptr(), c)
        torch.cuda.synchronize()
    for _ in range(3):
        q, kn, vn = rows(L, B, G * KVH, D), rows(L, B, KVH, D), rows(L, B, KVH, D)
        a, b = torch.zeros_like(q), torch.zeros_like(q)
        ra.ra_decode_step(caches[0].ctx, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), a.data_ptr())
        for l in range(L):
            ra.ra_decode_layer(caches[1].ctx, l, q[l].data_ptr(), kn[l].data_ptr(), vn[l].data_ptr(), b[l].data_ptr())
        torch.cuda.synchronize()
        # both round the weights and the output to bf16 (2^-9 each, relative): every row's norm within 1e-2
        err = (a.float() - b.float()).norm(dim=-1) / b.float().norm(dim=-1)
        assert float(err.max()) < 1e-2, float(err.max())
    for x in caches:
        ra.ra_check_device(x.ctx)
        x.close()
