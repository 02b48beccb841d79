"""pic_attention_deviation at the edges of its 32-key chunks: documents of 1 to
40 tokens (several region and document boundaries in one chunk), of exactly a
chunk, and long ones; two to eight regions, an empty one among them; a document
table that leaves room for three key stages and one that leaves two.  Reference:
64-bit softmax over the same bf16 keys and rotated queries; the sums are of
32-bit terms whose exponentials are good to 2^-22 of a probability (both
configurations' probabilities sum to one per row): bound 1e-3 of the sum plus
1e-5 per row and head."""
import math

import pytest
import torch

from paper_2607_28069_gb300.workloads import custom_spec, generate

pytestmark = pytest.mark.gpu

CASES = {
    "short_docs": (dict(pool_docs=60, docs_per_request=60, doc_len=(1, 40), head_dim=128),
                   (0.0, 0.1, 0.9)),
    "chunk_docs": (dict(pool_docs=20, docs_per_request=20, doc_len=(32, 32), head_dim=64),
                   (0.0, 0.25, 0.25, 0.5, 1.0)),
    "long_docs": (dict(pool_docs=4, docs_per_request=4, doc_len=(400, 900), head_dim=128,
                       span_len=(0, 5)), (0.0, 0.1, 0.9)),
    "eight_regions": (dict(pool_docs=5, docs_per_request=5, doc_len=(30, 500), head_dim=64),
                      tuple(i / 8 for i in range(9))),
    "two_stages": (dict(pool_docs=150, docs_per_request=150, doc_len=(1, 9), head_dim=128),
                   (0.0, 0.1, 0.9)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_deviation_edges(cuda_lib, name):
    import paper_2607_28069_gb300 as pic
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    kw, edges = CASES[name]
    spec = custom_spec(name=name, q_heads=8, kv_heads=2, rope_base=5e5, batch=2,
                       prefix_len=(1, 30), query_len=37, **kw)
    wl = generate(spec, device="cuda", gen_device="cpu")
    wl.q_inline.mul_(2.0)
    path = CacheHitPath(wl, with_lse=True, prefill_splits=1)
    path.ttft_pass(linked=False)
    k_b = path.k_cache.clone()
    pic.pic_relocate_mapped(path.geom, wl.k_pool, wl.v_pool, path.tok_map,
                            torch.zeros_like(path.doc_delta), path.slot_mapping, wl.num_pages, k_b,
                            path.v_cache.clone(), 0, 1)
    G, D, T = 4, spec.head_dim, spec.query_len
    pad = -(-path.max_inline * G // 128) * 128
    q = path.ws_prefill[:2 * 2 * pad * D * 2].view(torch.bfloat16).view(2, 2, pad, D).double()
    R = len(edges) - 1
    want = torch.zeros((2, R), dtype=torch.float64, device="cuda")
    n_want = torch.zeros((2, R), dtype=torch.int64, device="cuda")
    lse_b = torch.zeros_like(path.lse[0])
    lse_a = torch.zeros_like(lse_b)
    for b in range(2):
        ctx, tin = int(path.ctx_len[b]), int(wl.inline_len[b])
        sl = path.slot_mapping[b, :ctx]
        pos = path.inline_pos[b, tin - T:tin].repeat_interleave(G)
        mask = torch.arange(ctx, device="cuda")[None] > pos[:, None]
        region = torch.full((ctx,), -1, device="cuda")
        for k, i in enumerate(wl.meta["docs"][b]):
            o, n = int(path.doc_offset[b, k]), int(wl.doc_len[i])
            for r in range(R):
                lo, hi = math.ceil(edges[r] * n), math.ceil(edges[r + 1] * n)
                region[o + lo:o + hi] = r
                n_want[b, r] += max(hi - lo, 0) * T * 8
        for h in range(2):
            p = []
            for kc, lse in ((path.k_cache, lse_a), (k_b, lse_b)):
                K = kc[0, sl // 16, h, sl % 16].double()
                sc = (q[b, h, (tin - T) * G:tin * G] @ K.T / math.sqrt(D)).masked_fill(mask, -math.inf)
                s = torch.logsumexp(sc, 1)
                lse[b, tin - T:tin, h * G:(h + 1) * G] = s.view(T, G).float()
                p.append(torch.exp(sc - s[:, None]))
            d = (p[0] - p[1]).abs().sum(0)
            for r in range(R):
                want[b, r] += d[region == r].sum()
    sums = torch.full((2, R), -1.0, dtype=torch.float64, device="cuda")
    counts = torch.full((2, R), -1, dtype=torch.int64, device="cuda")
    pic.pic_attention_deviation(path.geom, 0, path.inline_pos, wl.inline_len, wl.query_len,
                                wl.req_doc_ids, wl.doc_len, path.doc_offset, path.slot_mapping,
                                wl.num_pages, path.k_cache, k_b, lse_a, lse_b, path.ws_prefill,
                                sums, counts, edges=edges, max_query_len=T)
    assert pic.pic_device_status() == (0, 0)
    assert torch.equal(counts, n_want)
    err = (sums - want).abs()
    assert bool((err <= 1e-3 * want + 1e-5 * T * 8).all()), (sums, want)
