"""In-place rounds of a whole stack with few heads: clusters share a head's array.  Caches of one chunk of 128
rows less, exactly, more and several, positions that do and do not start 16-byte aligned, evicted sets spread
over the cache (random), all at its start (recency, every row moves by m) and chosen by score (one launch for
every layer), against the oracle bit for bit."""
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [0, 2, 4], ids=["random", "recency", "scored"])
@pytest.mark.parametrize("K,r", [(96, 16), (97, 16), (98, 16), (226, 15), (225, 16), (130, 127), (900, 64), (1001, 33)])
def test_rounds_of_few_heads(K, r, policy):
    L, KVH = (3, 1) if r % 2 else (2, 2)
    run = Runner(L, 4 * KVH if r < 100 else KVH, KVH, [3, 70], K, r, eseed=K, dseed=r, fused=True, policy=policy)
    if policy == 4:  # (the window needs every query: from the start, two rounds)
        steps = (K + r) // r * r + 2 * r + 1
    else:  # from a full cache: the next step's round selects in place of its plan, two later ones have theirs
        g = -(-(3 * K + 4 * r) // r) * r - 1
        run.restore_full(g, layers=range(L))
        steps = 2 * r + 2
    fired = 0
    for t in range(steps):
        n = run.step(check_attn_layers=range(L) if t > steps - 3 else ())
        fired += n[0]
        if n[0]:
            run.check_state()
    assert fired >= 2 * run.B
    run.check_state()
    run.close()
