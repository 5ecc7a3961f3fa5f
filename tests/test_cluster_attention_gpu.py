"""Layers of few heads: a cluster per head, against the oracle at every step, through both call forms.  Every
group size; heads of one tile (most CTAs of the cluster hold none), of tiles that end at, before and past 32
rows while the cache grows, and of several tiles per warp; sequences without a prompt, finished ones, pages out
of order; one layer (the tiles requested ahead of the wait leave out the row that the step before wrote) and two.
The rule's other side, too many heads for clusters, runs the same checks."""
import numpy as np
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [True, False], ids=["layer", "calls"])
@pytest.mark.parametrize("L,G,KVH,lps", [(1, 4, 8, [1]), (2, 8, 1, [33, 0, 95]), (1, 1, 5, [3200]), (2, 3, 2, [64, 31]),
                                         (1, 5, 8, [0, 700, 20]), (1, 7, 2, [192]), (2, 2, 19, [40, 1, 0, 66]),
                                         (1, 6, 4, [130, 500]), (1, 4, 26, [50, 30, 9, 100, 64, 2])])
def test_every_step(L, G, KVH, lps, fused):
    run = Runner(L, G * KVH, KVH, lps, 40, 16, eseed=G, dseed=50 + G, fused=fused)
    steps = 75 if KVH < 26 else 4
    for t in range(steps):  # rounds at 64 and 72 tokens; the cache crosses 32 and 64 rows
        if t == 40 and len(lps) > 2:
            run.set_active(1, False)
        run.step(check_attn_layers=range(L))
    run.check_state()
    run.close()


def test_pages_out_of_order():
    run = Runner(1, 8, 2, [200, 400, 10], 24, 8, eseed=1, dseed=2, fused=True, prompt_pool=(600, 9 * 192))
    for t in range(3):
        run.step(check_attn_layers=(0,))
    run.admit(0, 5)
    run.admit(2, 590)
    run.admit(0, 300)
    for t in range(12):
        run.step(check_attn_layers=(0,))
    run.check_state()
    run.close()


def test_layer_call_after_separate_calls():
    """What a call of its own has just written is not read ahead of it: appends, rounds, loaded rows."""
    import paper_2609_03430_gb300 as ra

    run = Runner(2, 8, 2, [70, 33], 24, 8, eseed=3, dseed=4)
    for t in range(60):
        run.fused = t % 2 == 0
        run.step(check_attn_layers=(0, 1))
    run.restore_full(79, layers=(1, 0))
    run.fused = True
    run.step(check_attn_layers=(0, 1))
    run.check_state()
    run.close()


def test_compaction_inside_the_pass_of_one_layer():
    """The step behind a compacting attention launch does not read the regions that launch writes ahead of it."""
    run = Runner(1, 8, 2, [70, 0], 200, 16, eseed=5, dseed=6, fused=True, compaction=2)
    run.restore_full(639)
    for t in range(36):
        run.step(check_attn_layers=(0,))
    run.check_state()
    run.close()


def test_one_layer_called_again():
    """A layer of a stack stepped on its own, several steps in a row, then the other."""
    import paper_2609_03430_gb300 as ra

    run = Runner(2, 8, 2, [70, 3], 24, 8, eseed=7, dseed=8, fused=True)
    for layer in (0, 1):
        for t in range(70):
            k = run.torch.zeros((run.B, run.KVH, run.D), dtype=run.torch.int16, device="cuda")
            v = run.torch.zeros_like(k)
            for b in range(run.B):
                pos = run.orc.append(b, layer)
                for h in range(run.KVH):
                    k[b, h] = run.up(run.krows(layer, b, h, [pos])[0])
                    v[b, h] = run.up(run.vrows(layer, b, h, [pos])[0])
                run.orc.evict(b, layer)
            q = np.stack([run.qrows(layer, b, t) for b in range(run.B)])
            tq, out = run.up(q), run.torch.zeros((run.B, run.H, run.D), dtype=run.torch.int16, device="cuda")
            ra.ra_decode_layer(run.ctx, layer, tq.data_ptr(), k.data_ptr(), v.data_ptr(), out.data_ptr())
            run.check_layer_attention(layer, q, out.cpu().numpy())
    run.check_state()
    run.close()
