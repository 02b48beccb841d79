"""Prefill attention when a row's scores jump far past its running maximum in
the middle of a context.  The kernel exponentiates against the running maximum
and hands the first 64 keys' probabilities of a 128-key tile over before the
rest; a jump in either half has to be noticed before that and the tile redone.
Keys at chosen positions of later tiles are scaled up so that many rows jump by
more than 57 in the log2 domain, in the first half, the second half, both and
the last (masked) tile.  Reference: 64-bit softmax over the same bf16 cache and
the same bf16 rotated queries; bound: probabilities and outputs rounded to bf16
(2^-8 each, rows of size O(1)) and 32-bit scores of up to about 2000 (2^-24 of
that, 1.2e-4, in the exponent), within the bars of the other attention tests."""
import numpy as np
import pytest
import torch

from paper_2607_28069_gb300.workloads import custom_spec, generate
from tests.helpers import attn_close, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [1, 3])
@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("jumps", [(3 * 128 + 10,), (2 * 128 + 63,), (2 * 128 + 64,),
                                   (4 * 128 + 127,), (1 * 128, 3 * 128 + 70, 5 * 128 + 5)])
def test_score_jumps(cuda_lib, jumps, dim, splits):
    import paper_2607_28069_gb300 as pic
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    spec = custom_spec(name="jumps", q_heads=8, kv_heads=2, head_dim=dim, rope_base=5e5,
                       pool_docs=2, docs_per_request=2, doc_len=(350, 350), prefix_len=(7, 7),
                       query_len=33)
    wl = generate(spec, device="cuda", gen_device="cpu")
    wl.q_inline.mul_(8.0)
    path = CacheHitPath(wl, with_lse=True, prefill_splits=splits)
    path.compose()
    path.relocate()
    path.append(0)
    slots = path.slot_mapping[0]
    for i, t in enumerate(jumps):
        s = int(slots[t])
        path.k_cache[0, s // 16, :, s % 16] *= 16.0 * (i + 1)
    path.attend(0)
    assert pic.pic_device_status() == (0, 0)
    G, T, ctx = 4, int(wl.inline_len[0]), int(path.ctx_len[0])
    pad = -(-path.max_inline * G // 128) * 128
    q = f64(path.ws_prefill[:2 * pad * dim * 2].view(torch.bfloat16).view(2, pad, dim))
    sl = slots[:ctx].cpu().numpy()
    K = f64(path.k_cache[0])[sl // 16, :, sl % 16]
    V = f64(path.v_cache[0])[sl // 16, :, sl % 16]
    pos = path.inline_pos[0, :T].cpu().numpy()
    out, lse = f64(path.out[0, 0, :T]), f64(path.lse[0, 0, :T])
    jumped = 0
    for g in range(2):
        sc = q[g, :T * G] @ K[:, g].T / np.sqrt(dim)
        sc[np.arange(ctx)[None, :] > np.repeat(pos, G)[:, None]] = -np.inf
        for t in jumps:  # rows whose key t tops everything before its tile by 2^57
            before = sc[:, :t // 128 * 128].max(1)
            jumped += int(((sc[:, t] - before) / np.log(2) > 57).sum())
        m = sc.max(1, keepdims=True)
        p = np.exp(sc - m)
        ref = (p / p.sum(1, keepdims=True)) @ V[:, g]
        got = out[:, g * G:(g + 1) * G].reshape(T * G, dim)
        ok, worst, rel = attn_close(got, ref, abs_tol=1e-2, row_rel=1e-2)
        assert ok, (worst, rel)
        ref_lse = (m + np.log(p.sum(1, keepdims=True)))[:, 0].reshape(T, G)
        assert np.abs(lse[:, g * G:(g + 1) * G] - ref_lse).max() < 2e-3
    assert jumped > 20, jumped
