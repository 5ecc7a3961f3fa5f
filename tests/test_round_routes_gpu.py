"""Rounds at a step's start go for all layers at once only where that is the shorter way: on both sides of the rules'
lines the launches are the expected ones, and the caches bit for bit the oracle's.  Scored rounds, whose in-place
compaction does not share a buffer of more than 128 rows between CTAs, and which between layer calls only select ahead;
sets planned in the step whose plan takes the radix passes."""
import numpy as np
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


def _step(run):
    """One ra_decode_step of a scored run of one sequence; the oracle's rounds take the kernel's scores."""
    import paper_2609_03430_gb300 as ra

    L, t = run.L, run.step_idx
    run.qsteps[0].append(t)
    run.step_scale.append(0.0)
    pos = [run.orc.append(0, l) for l in range(L)]
    q = np.stack([run.qrows(l, 0, t)[None] for l in range(L)])
    k, v = (np.stack([np.stack([f(l, 0, h, [pos[l]])[0] for h in range(run.KVH)])[None] for l in range(L)])
            for f in (run.krows, run.vrows))
    tq, tk, tv = run.up(q), run.up(k), run.up(v)
    out = run.torch.zeros(q.shape, dtype=run.torch.int16, device="cuda")
    ra.ra_decode_step(run.ctx, tq.data_ptr(), tk.data_ptr(), tv.data_ptr(), out.data_ptr())
    for l in range(L):
        run.orc.evict(0, l, scorer=run.scorer)
        run.check_layer_attention(l, q[l], out[l].cpu().numpy())
    run.step_idx += 1


# launches of (select, evict, the stack's compaction): every layer's selection is one launch in all three
@pytest.mark.parametrize("form,L,launches", [("step", 4, (1, 4, 0)), ("step", 6, (1, 0, 1)), ("layers", 6, (1, 6, 0))])
def test_scored_rounds_of_a_long_buffer(form, L, launches):
    import paper_2609_03430_gb300 as ra

    K, r = 1024, 130
    run = Runner(L, 2, 2, [65], K, r, eseed=1, dseed=71, fused=True, policy=4)
    g = -(-4 * (K + 2 * r) // r) * r - 1  # the next step fires
    run.restore_full(g, layers=range(L))
    run.qsteps[0] = list(range(g))
    run.step_scale = [0.0] * g
    for l in range(L):
        w = run.up(np.stack([run.qrows(l, 0, s) for s in range(g - r, g)], axis=1)[None])
        ra.ra_restore_queries(run.ctx, l, w.data_ptr())
    ra.ra_profile_reset(run.ctx)
    for t in range(2):
        if form == "step":
            _step(run)
        else:
            run.step(check_attn_layers=range(L))
        run.check_state()
    kinds = (ra.RA_KERNEL_SELECT, ra.RA_KERNEL_EVICT, ra.RA_KERNEL_STACK)
    assert tuple(ra.ra_profile_read(run.ctx, k)[1] for k in kinds) == launches
    assert run.scored_rounds == 2 * L
    run.close()


@pytest.mark.parametrize("L,planned", [(4, False), (16, True)], ids=["by-layer", "planned"])
def test_sets_of_a_long_buffer_planned_in_the_step(L, planned):
    import paper_2609_03430_gb300 as ra

    run = Runner(L, 2, 2, [33], 2000, 512, eseed=2, dseed=72, fused=True)
    run.restore_full(512 * 20 - 1, layers=range(L))
    ra.ra_profile_reset(run.ctx)
    run.step(check_attn_layers=(0, L - 1))
    evict, stack = (ra.ra_profile_read(run.ctx, k)[1] for k in (ra.RA_KERNEL_EVICT, ra.RA_KERNEL_STACK))
    assert (evict, stack) == ((0, 1) if planned else (L, 0))
    run.step(check_attn_layers=(0, L - 1))
    run.check_state()
    run.close()
