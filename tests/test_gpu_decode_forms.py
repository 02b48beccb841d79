"""pic_attend_decode's forms: the append inside the attention kernel and the
splits merged in a cluster (2 to 16 splits on a grid that fits the GPU) or by
the merge kernel.  Positions at the edges of pages and splits (first and last
row of a page, the only key, a new page of its own), 1 to 17 splits, GQA groups
of 1, 7 and 16, both head dims and RoPE styles.  Reference: 64-bit softmax over
the bf16 cache and bf16 rotated queries; bars as in the parity tests.  The new
key is bit-identical to pic_append_inline's, the new value to its input, and
nothing else in the cache changes."""
import numpy as np
import pytest
import torch

from tests.helpers import attn_close, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [1, 2, 7, 16, 17])
@pytest.mark.parametrize("heads,dim,style", [((4, 4), 128, 0), ((14, 2), 64, 1), ((32, 2), 128, 1),
                                             ((7, 1), 128, 0), ((16, 1), 64, 0)])
def test_decode_forms(cuda_lib, heads, dim, style, splits):
    import paper_2607_28069_gb300 as pic
    hq, hkv = heads
    G = hq // hkv
    pos_l = [0, 15, 16, 17 * 16 - 1, 17 * 16, 300, 351]
    B, max_ctx, pages = len(pos_l), 352, 22
    gen = torch.Generator(device="cuda").manual_seed(splits * 131 + hq)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()  # noqa: E731
    g = pic.Geometry(2, hq, hkv, dim, 5e5, rope_style=style)
    n_pages = B * pages
    kc, vc = rnd(2, n_pages, hkv, 16, dim), rnd(2, n_pages, hkv, 16, dim)
    bt = torch.randperm(n_pages, generator=gen, device="cuda").int().view(B, pages)
    q, k, v = rnd(B, hq, dim) * 2, rnd(B, hkv, dim), rnd(B, hkv, dim)
    pos = torch.tensor(pos_l, dtype=torch.int32, device="cuda")
    out = torch.empty((B, hq, dim), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((B, hq), dtype=torch.float32, device="cuda")
    ws = torch.empty(pic.pic_decode_workspace_size(g, B, max_ctx, splits), dtype=torch.uint8,
                     device="cuda")
    # the append on its own: new keys and rotated queries to compare with
    k_ref, v_ref = kc.clone(), vc.clone()
    slot = (bt.gather(1, (pos // 16).long()[:, None]).long() * 16 + (pos % 16).long()[:, None])
    slots = torch.full((B, max_ctx), -1, dtype=torch.int64, device="cuda")
    slots.scatter_(1, pos.long()[:, None], slot)
    wp = torch.zeros(pic.pic_prefill_workspace_size(g, B, 1, max_ctx, 1), dtype=torch.uint8,
                     device="cuda")
    pic.pic_append_inline(g, 1, q[:, None].contiguous(), k[:, None].contiguous(),
                          v[:, None].contiguous(), pos[:, None].contiguous(),
                          torch.ones(B, dtype=torch.int32, device="cuda"), slots, n_pages, k_ref,
                          v_ref, wp)
    pic.pic_attend_decode(g, 1, q, k, v, pos - 3, bt, n_pages, kc, vc, out, max_ctx, lse=lse,
                          num_splits=splits, workspace=ws, pos_offset=3)
    assert pic.pic_device_status() == (0, 0)
    assert torch.equal(kc, k_ref) and torch.equal(vc, v_ref)
    qr = f64(wp[:B * hkv * 128 * dim * 2].view(torch.bfloat16).view(B, hkv, 128, dim))
    for b, p in enumerate(pos_l):
        t = np.arange(p + 1)
        page = bt[b].cpu().numpy()[t // 16]
        K, V = f64(kc[1])[page, :, t % 16], f64(vc[1])[page, :, t % 16]
        for h in range(hq):
            sc = K[:, h // G] @ qr[b, h // G, h % G] / np.sqrt(dim)
            m = sc.max()
            w = np.exp(sc - m)
            ref = w @ V[:, h // G] / w.sum()
            ok, worst, rel = attn_close(f64(out[b, h])[None], ref[None], abs_tol=1e-2, row_rel=1e-2)
            assert ok, (b, h, worst, rel)
            assert abs(float(lse[b, h]) - (m + np.log(w.sum()))) < 2e-3


def test_bad_token_positions_are_reported(cuda_lib):
    """A position outside the block table, and a page outside the cache: the
    request's token is not appended, the others are."""
    import paper_2607_28069_gb300 as pic
    g = pic.Geometry(1, 4, 1, 64, 1e4)
    z = lambda *s: torch.ones(s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    bt = torch.tensor([[0, 1], [2, 9]], dtype=torch.int32, device="cuda")
    for pos, code in (([40, 5], 7), ([3, 20], 6)):
        kc, vc = z(1, 4, 1, 16, 64) * 0, z(1, 4, 1, 16, 64) * 0
        ws = torch.empty(pic.pic_decode_workspace_size(g, 2, 64, 2), dtype=torch.uint8, device="cuda")
        pic.pic_attend_decode(g, 0, z(2, 4, 64), z(2, 1, 64), z(2, 1, 64),
                              torch.tensor(pos, dtype=torch.int32, device="cuda"), bt, 4, kc, vc,
                              z(2, 4, 64), 64, num_splits=2, workspace=ws)
        assert pic.pic_device_status()[0] in (code, 5)
        written = vc[0, :, 0, :, 0].nonzero().tolist()
        assert written == ([[2, 5]] if code == 7 else [[0, 3]])
