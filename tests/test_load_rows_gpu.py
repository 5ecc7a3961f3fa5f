"""Rows loaded into the caches (ra_prefill, ra_restore, ra_admit) arrive bit-exactly at the sizes where the
copy's chunks of 64 rows and the pages of 192 end: one row more and less, none at all, several layers."""
import pytest

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 63, 64, 65, 191, 192, 193, 257]


@pytest.mark.parametrize("first,second", [(0, 4), (3, 7), (5, 1), (8, 2)])
def test_prompt_edges(first, second):
    from ra_testlib import Runner

    lps = [EDGES[first], EDGES[second], EDGES[(first + second) % len(EDGES)]]
    run = Runner(3, 4, 2, lps, 8, 4, eseed=1, dseed=2, prompt_pool=(384, 6 * 192))
    run.check_state()
    for b, n in ((1, EDGES[first]), (0, EDGES[second]), (2, 384)):
        run.admit(b, n)
        run.check_state()
    run.close()


@pytest.mark.parametrize("K,r", [(1, 1), (59, 3), (58, 4), (64, 32), (61, 65)])
def test_restore_edges(K, r):  # K + 2 r - 1 rows: 2, 64, 65, 127, 190
    from ra_testlib import Runner

    run = Runner(2, 3, 1, [5, 0], K, r, eseed=3, dseed=4)
    run.restore_full(4 * (K + 2 * r), layers=(0, 1))
    run.check_state()
    run.close()
