"""Layers of few heads: a cluster per head, against the oracle at every step, through both call forms.  Every
group size; heads of one tile (most CTAs of the cluster hold none), of tiles that end at, before and past 32
rows while the cache grows, and of several tiles per warp; sequences without a prompt, finished ones, pages out
of order; one layer (the tiles requested ahead of the wait leave out the row that the step before wrote) and two.
The rule's other side, too many heads for clusters, runs the same checks."""
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
