"""A scored round of a layer call right behind the call that wrote that layer's query window, another layer's call in
between the loaded rows and it: the scoring pass reads the window (and its normalisers) only once it is complete.  The
window holds other queries before, so that a read ahead of the write shows in the scores, which are compared with the
fp64 oracle's.  Rounds go layer by layer (two kernels), or their sets are selected for every layer in layer 0's call, in
which case the write drops the layer's set, whose round has not run yet.  The writers: a loaded window, and both attention calls, which
record the latest step's query."""
import numpy as np
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("by_layer", [True, False], ids=["two-kernels", "auto"])
@pytest.mark.parametrize("writer", ["window", "attend", "noalloc"])
def test_scores_behind_the_window_writer(writer, by_layer):
    import paper_2609_03430_gb300 as ra

    G, KVH, r, K, lps = 4, 4, 64, 700, [900, 65, 300]
    run = Runner(2, G * KVH, KVH, lps, K, r, eseed=1, dseed=61, fused=True, policy=4)
    if by_layer:
        ra.ra_set_eviction_kernel(run.ctx, ra.RA_EVICT_TWO_KERNELS)
    B, c = run.B, K + 2 * r - 1
    g = -(-4 * c // r) * r - 1  # the next step fires
    run.restore_full(g, layers=(0, 1))
    for b in range(B):
        run.qsteps[b] = list(range(g))
    run.step_scale = [0.0] * g

    def window(l, shift, last_shift):
        steps = [s + shift for s in range(g - r, g - 1)] + [g - 1 + last_shift]
        return run.up(np.stack([np.stack([run.qrows(l, b, s) for s in steps], axis=1) for b in range(B)]))

    right = [window(l, 0, 0) for l in (0, 1)]
    before = window(1, 5000 if writer == "window" else 0, 5000)
    latest = run.up(np.stack([run.qrows(1, b, g - 1) for b in range(B)]))
    out = run.torch.zeros((B, run.H, run.D), dtype=run.torch.int16, device="cuda")
    ra.ra_restore_queries(run.ctx, 0, right[0].data_ptr())
    ra.ra_restore_queries(run.ctx, 1, before.data_ptr())

    class Between:  # the binding, with the writer's call right before layer 1's
        def __getattr__(self, name):
            return getattr(ra, name)

        def ra_decode_layer(self, ctx, layer, *args):
            if layer == 1:
                assert all(ra.ra_get_counters(ctx, b, 1) == (g, c, 0) for b in range(B))
                if writer == "window":
                    ra.ra_restore_queries(ctx, 1, right[1].data_ptr())
                elif writer == "attend":
                    ra.ra_decode_attn(ctx, 1, latest.data_ptr(), out.data_ptr())
                else:
                    ra.ra_decode_attn_noalloc(ctx, 1, latest.data_ptr(), out.data_ptr())
            ra.ra_decode_layer(ctx, layer, *args)

    run.ra = Between()
    fired = run.step(check_attn_layers=(0, 1))
    assert fired == {0: B, 1: B} and run.scored_rounds == 2 * B * KVH
    run.check_state()
    run.close()
