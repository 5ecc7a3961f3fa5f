"""Sequences that fire without a set computed ahead, in stacks deep enough for it (4, 8, 12 or 24 layers, by policy
and layout): the sets are computed in the step and every layer's round runs in one launch, in both layouts, for every
policy of the plans, bit for bit against the oracle; a slot switched on again at its firing step, beside one whose
set was computed ahead."""
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compaction", [0, 1], ids=["ordered", "free"])
@pytest.mark.parametrize("policy,block", [(0, 1), (1, 1), (2, 1), (3, 16)], ids=["random", "shared", "recency", "block"])
def test_first_round_of_a_loaded_run(policy, block, compaction):
    import paper_2609_03430_gb300 as ra

    # the shallowest stack that plans in the step
    L = 4 * (2 if policy >= 2 else 1) * (3 if policy == 3 or compaction else 1)
    KVH = 2 if L <= 8 else 1
    run = Runner(L, 2 * KVH, KVH, [33, 0, 90], 100, 16, eseed=policy, dseed=9, fused=True, policy=policy, block=block,
                 compaction=compaction)
    run.restore_full(639, layers=range(L))  # all fire at the next step
    ra.ra_profile_reset(run.ctx)
    for t in range(35):
        if t == 10:
            run.set_active(1, False)
        if t == 26:  # on again: it fires 6 steps later than the others, once more after
            run.set_active(1, True)
        run.step(check_attn_layers=(0, L - 1) if t in (0, 1, 16, 31, 32) else ())
        if t in (0, 1, 16, 32):
            run.check_state()
    assert ra.ra_profile_read(run.ctx, ra.RA_KERNEL_EVICT)[1] == 0 and ra.ra_profile_read(run.ctx, ra.RA_KERNEL_SELECT)[1] == 0
    run.check_state()
    run.close()


def test_slot_on_again_at_its_round():
    run = Runner(4, 4, 2, [20, 20], 60, 8, eseed=3, dseed=4, fused=True)
    run.restore_full(399, layers=range(4))
    run.step()
    for _ in range(7):
        run.step()
    run.set_active(1, False)  # both would fire at the next step: slot 1's set is ready, and not used
    run.step(check_attn_layers=(0, 3))
    run.set_active(1, True)
    run.step(check_attn_layers=(0, 3))  # slot 1's round
    run.check_state()
    for _ in range(10):
        run.step()
    run.check_state()
    run.close()
