"""The normalisers that ra_restore_queries computes, through the window scores of the round that follows
(compared with the fp64 oracle's): one to four 128-row tiles of window rows, prompts and caches that end
inside, at and past the 64-row runs and 192-row pages, several runs per CTA and one, and cached tokens with
gaps among the newest r (a query's newest keys are then not simply the newest rows)."""
import numpy as np
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gaps", [False, True], ids=["newest", "gaps"])
@pytest.mark.parametrize("G,r,K,lps", [(1, 8, 41, [0, 64, 65]), (3, 33, 30, [1, 191]), (4, 64, 129, [192, 193, 63]),
                                       (5, 64, 200, [700, 0]), (8, 64, 128, [130, 600])],
                         ids=["rows8", "rows99", "rows256", "rows320", "rows512"])
def test_scores_after_restored_queries(G, r, K, lps, gaps):
    import paper_2609_03430_gb300 as ra

    run = Runner(1, 2 * G, 2, lps, K, r, eseed=G, dseed=40 + G, fused=True, policy=4)
    rng = np.random.default_rng(r + gaps)
    c = K + 2 * r - 1
    g = -(-4 * c // r) * r - 1  # the next step fires
    B, KVH = run.B, run.KVH
    pos = np.zeros((B, KVH, c), np.int32)
    kk = np.zeros((B, KVH, c, run.D), np.uint16)
    vv = np.zeros_like(kk)
    for b in range(B):
        for h in range(KVH):
            p = np.sort(rng.choice(g, c, replace=False)) if gaps else np.arange(g - c, g)
            p = run.lp[b] + p
            pos[b, h], kk[b, h], vv[b, h] = p, run.krows(0, b, h, p), run.vrows(0, b, h, p)
            run.orc.gen[(b, 0, h)] = p.astype(np.int32)
        run.orc.g[b, 0] = g
        run.qsteps[b] = list(range(g))
    run.step_scale = [0.0] * g
    run.step_idx = g
    tp, tk, tv = run.torch.from_numpy(pos).cuda(), run.up(kk), run.up(vv)
    ra.ra_restore(run.ctx, 0, [g] * B, [c] * B, tp.data_ptr(), tk.data_ptr(), tv.data_ptr(), c)
    w = np.stack([np.stack([run.qrows(0, b, s) for s in range(g - r, g)], axis=1) for b in range(B)])
    tw = run.up(w)  # [B][H][r][D]
    ra.ra_restore_queries(run.ctx, 0, tw.data_ptr())
    assert run.step(check_attn_layers=(0,))[0] == B
    assert run.scored_rounds == B * KVH
    run.check_state()
    run.close()
