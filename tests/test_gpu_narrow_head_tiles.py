"""Prefill attention at d = 64, where S_t(j) is computed while softmax t still
works on tile j - 1 and three S buffers are passed round among the steps: the
smallest numbers of key tiles, one and two query tiles, a second tile that needs
fewer key tiles than the first (rows of a short prefix), none of a split's, and
splits of unequal length, with rows that rescale O in between (a key near the
end of each tile is scaled up).  Reference: 64-bit softmax over the same bf16
cache and bf16 rotated queries.  Bound: a row is a mean of values weighted with
probabilities rounded to bf16 (2^-8 of each), a split's row is rounded to fp16
(2^-11), and 32-bit scores and sums add less than 2^-13: (2^-8 + 2^-11 + 2^-13)
times the largest value, above the output's own rounding.  (A row that one key
dominates comes near it, so 1e-2, right for |v| < 2, is not enough here.)"""
import numpy as np
import pytest
import torch

from paper_2607_28069_gb300.workloads import custom_spec, generate
from tests.helpers import attn_close, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [1, 2, 3])
@pytest.mark.parametrize("prefix,query", [(1, 1), (7, 33), (33, 32), (32, 40)])
@pytest.mark.parametrize("doc", [16, 40, 100, 165, 230, 300, 420])
def test_key_tiles(cuda_lib, doc, prefix, query, splits):
    import paper_2607_28069_gb300 as pic
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    spec = custom_spec(name="tiles", q_heads=8, kv_heads=2, head_dim=64, rope_base=5e5,
                       pool_docs=2, docs_per_request=2, doc_len=(doc, doc),
                       prefix_len=(prefix, prefix), query_len=query)
    wl = generate(spec, device="cuda", gen_device="cpu")
    path = CacheHitPath(wl, with_lse=True, prefill_splits=splits)
    path.compose()
    path.relocate()
    path.append(0)
    G, T, ctx = 4, int(wl.inline_len[0]), int(path.ctx_len[0])
    slots = path.slot_mapping[0]
    for i, t in enumerate(range(120, ctx, 128)):
        s = int(slots[t])
        path.k_cache[0, s // 16, :, s % 16] *= 3.0 * (i + 1)
    path.attend(0)
    assert pic.pic_device_status() == (0, 0)
    pad = -(-path.max_inline * G // 128) * 128
    q = f64(path.ws_prefill[:2 * pad * 64 * 2].view(torch.bfloat16).view(2, pad, 64))
    sl = slots[:ctx].cpu().numpy()
    K = f64(path.k_cache[0])[sl // 16, :, sl % 16]
    V = f64(path.v_cache[0])[sl // 16, :, sl % 16]
    pos = path.inline_pos[0, :T].cpu().numpy()
    out, lse = f64(path.out[0, 0, :T]), f64(path.lse[0, 0, :T])
    for g in range(2):
        sc = q[g, :T * G] @ K[:, g].T / 8.0
        sc[np.arange(ctx)[None, :] > np.repeat(pos, G)[:, None]] = -np.inf
        m = sc.max(1, keepdims=True)
        p = np.exp(sc - m)
        ref = (p / p.sum(1, keepdims=True)) @ V[:, g]
        ok, worst, rel = attn_close(out[:, g * G:(g + 1) * G].reshape(T * G, 64), ref,
                                    abs_tol=(2**-8 + 2**-11 + 2**-13) * np.abs(V[:, g]).max(),
                                    row_rel=1e-2)
        assert ok, (worst, rel)
        ref_lse = (m + np.log(p.sum(1, keepdims=True)))[:, 0].reshape(T, G)
        assert np.abs(lse[:, g * G:(g + 1) * G] - ref_lse).max() < 2e-3
