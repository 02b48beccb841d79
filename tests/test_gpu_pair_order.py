"""Unsplit prefill attention over 4096 keys and more in several waves: its CTAs
run group of pairs by group (half of every request's query pairs, then quarters),
with 5 (one group and a lone pair), 6, 7, 10 and 12 pairs a request, so that every
(pair, kv head, request) has to come up exactly once.  Against the same call split
in two, whose order is request by request, and rotate-on-load (clusters of two
pairs) against the stitched cache, bit for bit.  Bound: both sides round their
probabilities to bf16 (2^-8 each, of values below 8 in a mean over thousands of
keys) and the split one its rows to fp16, inside 1e-2 for these outputs of size
2^-4, and both the output to bf16."""
import pytest
import torch

from paper_2607_28069_gb300.workloads import custom_spec, generate
from tests.helpers import attn_close, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("query", [260, 330, 400, 560, 740])
def test_pair_order(cuda_lib, query, dim):
    import paper_2607_28069_gb300 as pic
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    spec = custom_spec(name="order", q_heads=32, kv_heads=8, head_dim=dim, rope_base=5e5, batch=4,
                       pool_docs=4, docs_per_request=4, doc_len=(1001, 1030), prefix_len=(3, 9),
                       query_len=query, span_len=(1, 9))
    wl = generate(spec, device="cuda", gen_device="cpu")
    outs = []
    for splits in (1, 2):
        path = CacheHitPath(wl, prefill_splits=splits)
        path.compose()
        path.relocate()
        path.append(0)
        path.out.fill_(float("nan"))
        path.attend(0)
        outs.append(path.out.clone())
    fused = CacheHitPath(wl, prefill_splits=1)
    fused.out.fill_(float("nan"))
    fused.fused_pass()
    assert pic.pic_device_status() == (0, 0)
    for b in range(4):
        T = int(wl.inline_len[b])
        assert torch.equal(outs[0][0, b, :T], fused.out[0, b, :T])
        ok, worst, rel = attn_close(f64(outs[0][0, b, :T]).reshape(-1, dim),
                                    f64(outs[1][0, b, :T]).reshape(-1, dim), abs_tol=1e-2,
                                    row_rel=2e-2)
        assert ok, (b, worst, rel)
