"""The stacked attention launch (ra_decode_step: every layer's heads in one launch) against the oracle: group
sizes in both kernel shapes, sequences without a prompt, finished ones at the ends and in the middle of the
batch (the walk skips them from layer to layer), heads whose regions moved (rounds with no set computed ahead
swap them layer by layer), one tile per head and several.  Then the layer-by-layer route where the layers'
counters differ, and after a stacked step the layer calls, which must not read ahead of it."""
import numpy as np
import pytest

from ra_testlib import Runner, check_attention

pytestmark = pytest.mark.gpu


def _step(run, t):
    """One ra_decode_step with every output row checked; the oracle appends and evicts alike."""
    import oracle
    import paper_2609_03430_gb300 as ra

    L, B, H, KVH, G, D = run.L, run.B, run.H, run.KVH, run.G, run.D
    k = np.zeros((L, B, KVH, D), np.uint16)
    v = np.zeros_like(k)
    q = np.stack([np.stack([run.qrows(l, b, t) for b in range(B)]) for l in range(L)])
    for l in range(L):
        for b in range(B):
            if not run.active[b]:
                continue
            pos = run.orc.append(b, l)
            for h in range(KVH):
                k[l, b, h] = run.krows(l, b, h, [pos])[0]
                v[l, b, h] = run.vrows(l, b, h, [pos])[0]
            run.orc.evict(b, l)
    tq, tk, tv = run.up(q), run.up(k), run.up(v)
    out = run.torch.full((L, B, H, D), 77, dtype=run.torch.int16, device="cuda")
    ra.ra_decode_step(run.ctx, tq.data_ptr(), tk.data_ptr(), tv.data_ptr(), out.data_ptr())
    got = out.cpu().numpy()
    for l in range(L):
        for b in range(B):
            if not run.active[b]:
                assert (got[l, b] == 77).all()
                continue
            for h in range(KVH):
                pos = run.orc.positions(b, l, h)
                ref = oracle.attend(q[l, b, h * G:(h + 1) * G], run.krows(l, b, h, pos), run.vrows(l, b, h, pos))
                check_attention(got[l, b, h * G:(h + 1) * G], ref, f"step {t} layer {l} seq {b} head {h}")


@pytest.mark.parametrize("shape", [1, 2], ids=["wide", "narrow"])
@pytest.mark.parametrize("G,KVH,lps", [(1, 3, [0, 31, 33]), (4, 2, [200, 0, 48, 500]), (5, 1, [1, 0]), (8, 2, [97, 193, 0])])
def test_every_layer_in_one_launch(G, KVH, lps, shape):
    run = Runner(3, G * KVH, KVH, lps, 24, 8, eseed=5, dseed=6, attn_shape=shape)
    t = 0
    for stage in (None, 0, len(lps) - 1):  # all, then without the first, then without the last too
        if stage is not None and len(lps) > 2:
            run.set_active(stage, False)
        for _ in range(22):  # rounds at 40, 48, 56, 64: the first with no set computed ahead
            _step(run, t)
            t += 1
        run.check_state()
    run.close()


def test_layers_apart_and_mixed_calls():
    run = Runner(2, 8, 2, [70, 3], 24, 8, eseed=7, dseed=8, fused=True)
    for t in range(44):
        _step(run, t)
    run.step_idx = 44
    run.restore_full(79, layers=(1,))  # layer 1 elsewhere than layer 0: layer by layer
    for t in range(80, 84):
        _step(run, t)
    run.check_state()
    run.restore_full(79, layers=(0, 1))  # alike again; layer calls right behind stacked ones
    run.step_idx = 79
    for t in range(79, 99):
        if t % 3 == 2:
            run.step(check_attn_layers=(0, 1))
        else:
            _step(run, t)
            run.step_idx = t + 1
    run.check_state()
    run.close()
