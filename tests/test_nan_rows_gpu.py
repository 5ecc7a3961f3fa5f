"""Cache rows of NaN make their head's output NaN, wherever the split puts them: the pieces that hold them have no
maximum, in a merge of many records as in one of few (eight at a time; on 152 SMs the narrow shape cuts 60000 rows of
two heads into 960 per record), and in every form of the attention."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [0, 1, 2], ids=["auto", "wide", "narrow"])
@pytest.mark.parametrize("rows", [7680, 20000, 32], ids=["eight-records", "many-records", "one-tile"])
@pytest.mark.parametrize("lp", [60000, 5000])
def test_rows_of_nan(shape, rows, lp):
    import torch

    import paper_2609_03430_gb300 as ra

    G, D = 3, 128
    g = torch.Generator("cuda").manual_seed(lp)
    cache = ra.RandomAttentionCache(1, 2 * G, 2, D, [lp], 64, 16, seed=1)
    ra.ra_set_attention_shape(cache.ctx, shape)
    k, v = (torch.randn(1, 2, lp, D, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    k[0, 0, :min(rows, lp - 100), 7] = float("nan")
    ra.ra_prefill(cache.ctx, 0, k.data_ptr(), v.data_ptr(), lp)
    q = torch.randn(1, 2 * G, D, generator=g, device="cuda", dtype=torch.bfloat16)
    out = torch.zeros_like(q)
    ra.ra_decode_attn(cache.ctx, 0, q.data_ptr(), out.data_ptr())
    assert bool(out[0, :G].isnan().all())
    ref = torch.softmax(q[0, G:].double() @ k[0, 1].double().T / D ** 0.5, -1) @ v[0, 1].double()
    # weights and output rounded to bf16 (2^-9 each, relative, in the mean)
    assert float((out[0, G:].double() - ref).norm() / ref.norm()) < 6e-3
    cache.close()
