"""A launch whose bounded wait ran out leaves the attention's claim and arrival counters behind.  Once the timeout is
reported the context is usable again: the counters are zero, and a long stacked step, which takes every chunk of its
tail by the claim counter, gives what the layer calls give.  The counters are set from the host, as such a launch
leaves them; nothing on the device waits but the timeout probe, for 1 ms."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_counters_are_ready_again_after_a_reported_timeout():
    import torch

    import paper_2609_03430_gb300 as ra

    L, G, KVH, K, r, D = 14, 4, 8, 8000, 64, 128
    lps = [700, 1500, 1, 64, 2000, 900, 333, 48, 1100]
    B, c, g0 = len(lps), K + r + 5, 20000 * r + 5
    g = torch.Generator("cuda").manual_seed(3)
    caches = [ra.RandomAttentionCache(L, G * KVH, KVH, D, lps, K, r, seed=1) for _ in range(2)]

    def rows(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)

    pos = torch.stack([lp + torch.arange(g0 - c, g0, dtype=torch.int32) for lp in lps])
    pos = pos[:, None, :].expand(B, KVH, c).contiguous().cuda()
    for l in range(L):
        pk, pv, k, v = rows(B, KVH, max(lps), D), rows(B, KVH, max(lps), D), rows(B, KVH, c, D), rows(B, KVH, c, D)
        for x in caches:
            ra.ra_prefill(x.ctx, l, pk.data_ptr(), pv.data_ptr(), max(lps))
            ra.ra_restore(x.ctx, l, [g0] * B, [c] * B, pos.data_ptr(), k.data_ptr(), v.data_ptr(), c)
        torch.cuda.synchronize()

    # the error word stands before the sets computed ahead, the arena's last part; the claim counter 128 bytes after
    # it, the arrival counters before it (and before those the partial records, which no launch reads before writing)
    x, stream = caches[0], torch.cuda.current_stream().cuda_stream
    err = x.nbytes - (2 * L * B * KVH * (r + 1) * 4 + 255) // 256 * 256 - 256
    words = x.arena[x.base - x.arena.data_ptr():][:x.nbytes].view(torch.int32)
    assert ra.lib().ra_debug_timeout_probe(x.ctx, ctypes.c_uint64(1_000_000), stream) == ra.RA_OK
    torch.cuda.synchronize()
    assert int(words[err // 4]) == 1
    words[err // 4 + 32] = 3
    words[err // 4 - 4096:err // 4] = 1
    assert ra.lib().ra_check_device(x.ctx, stream) == ra.RA_ERR_DEVICE_TIMEOUT
    torch.cuda.synchronize()
    assert int(words[err // 4]) == 0 and int(words[err // 4 + 32]) == 0
    assert not bool(words[err // 4 - 4096:err // 4].any())
    assert ra.lib().ra_check_device(x.ctx, stream) == ra.RA_OK

    q, kn, vn = rows(L, B, G * KVH, D), rows(L, B, KVH, D), rows(L, B, KVH, D)
    a, b = torch.zeros_like(q), torch.zeros_like(q)
    ra.ra_decode_step(caches[0].ctx, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), a.data_ptr())
    for l in range(L):
        ra.ra_decode_layer(caches[1].ctx, l, q[l].data_ptr(), kn[l].data_ptr(), vn[l].data_ptr(), b[l].data_ptr())
    torch.cuda.synchronize()
    # both round the output to bf16 and one the weights (2^-9 each, relative): every row's norm within 1e-2
    error = (a.float() - b.float()).norm(dim=-1) / b.float().norm(dim=-1)
    assert float(error.max()) < 1e-2, float(error.max())
    for x in caches:
        ra.ra_check_device(x.ctx)
        x.close()
