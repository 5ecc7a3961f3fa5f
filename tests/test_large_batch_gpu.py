"""Layer calls of more than 64 sequences (their launch parameters are another size) against the oracle, through a round,
with finished sequences among them, in both call forms."""
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [True, False], ids=["layer", "calls"])
@pytest.mark.parametrize("B,G", [(65, 4), (100, 1)])
def test_more_than_64_sequences(B, G, fused):
    run = Runner(2, 2 * G, 2, [(37 * b) % 120 for b in range(B)], 12, 8, eseed=B, dseed=G, fused=fused)
    for t in range(34):  # rounds at 24 and 32 tokens
        if t == 20:
            run.set_active(64, False)
            run.set_active(3, False)
        run.step(check_attn_layers=(0, 1) if t in (0, 23, 24, 33) else ())
    run.check_state()
    run.close()
