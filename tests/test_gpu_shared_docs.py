"""Documents that several listed occurrences share: pic_relocate reads each once
and writes it to every occurrence (relocate_docs_kernel), in large relocations
with enough document tokens for groups of two or more, and large pic_links use
the same kernel.  Both are compared bit for bit with pic_relocate_mapped, which
moves position by position and knows no sharing: groups of two to kMaxShare = 8
occurrences, more occurrences than a group takes, a document repeated in one
request, head counts that leave a remainder block of heads, chunks of 8, 16 and
32 tokens with remainders, both RoPE styles, per-layer rotary tables, document
lists beyond the 2048 a CTA searches, and relocations too small to search."""
import pytest
import torch

from paper_2607_28069_gb300.workloads import custom_spec, generate

pytestmark = pytest.mark.gpu


def _spec(name, **kw):
    return custom_spec(name=name, rope_base=5e5, prefix_len=(3, 70), query_len=19, **kw)


CASES = {
    # name: (spec, rope style, per-layer tables, group size)
    "pairs": (_spec("pairs", layers=2, q_heads=32, kv_heads=8, head_dim=128, batch=3, pool_docs=9,
                    docs_per_request=6, doc_len=(900, 2100)), 0, False, 3),
    "groups_over_8": (_spec("groups_over_8", layers=2, q_heads=32, kv_heads=8, head_dim=128,
                            batch=19, pool_docs=3, docs_per_request=3, doc_len=(1001, 1333),
                            span_len=(0, 5)), 1, False, 8),
    "repeated": (_spec("repeated", layers=2, q_heads=8, kv_heads=4, head_dim=128, batch=2,
                       pool_docs=4, docs_per_request=7, doc_len=(2900, 5100),
                       fixed_order=(0, 2, 1, 0, 3, 1, 0)), 0, True, 4),
    "heads_12": (_spec("heads_12", layers=2, q_heads=24, kv_heads=12, head_dim=128, batch=4,
                       pool_docs=5, docs_per_request=4, doc_len=(1500, 2400)), 1, False, 4),
    "d64_h3": (_spec("d64_h3", layers=2, q_heads=6, kv_heads=3, head_dim=64, batch=5, pool_docs=6,
                     docs_per_request=5, doc_len=(5000, 7000)), 0, False, 5),
    "d64_h16_tables": (_spec("d64_h16_tables", layers=3, q_heads=16, kv_heads=16, head_dim=64,
                             batch=4, pool_docs=5, docs_per_request=5, doc_len=(900, 2200)), 0, True,
                       4),
    "beyond_scan": (_spec("beyond_scan", layers=2, q_heads=8, kv_heads=4, head_dim=128, batch=17,
                          pool_docs=130, docs_per_request=128, doc_len=(1, 30)), 0, False, 2),
    # one request: nothing shared, and too few tokens to look for it
    "one_request": (_spec("one_request", layers=10, q_heads=8, kv_heads=2, head_dim=128, batch=1,
                          pool_docs=20, docs_per_request=12, doc_len=(300, 1000)), 0, False, 1),
}


def _path(name):
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    spec, style, tables, _ = CASES[name]
    wl = generate(spec, device="cuda", gen_device="cuda")
    # a capacity from which the link is three launches (2200 CTAs of a page or two)
    wl.max_ctx = max(wl.max_ctx, -(-2200 // spec.batch) * 32)
    table = torch.full((spec.batch, -(-wl.max_ctx // 16)), -1, dtype=torch.int32, device="cuda")
    table[:, :wl.block_table.shape[1]] = wl.block_table
    wl.block_table = table
    freqs = None
    if tables:
        i = torch.arange(spec.head_dim // 2, dtype=torch.float64)
        freqs = torch.stack([(1e4 if l % 2 else 5e5) ** (-2.0 * i / spec.head_dim)
                             for l in range(spec.layers)]).cuda()
    return CacheHitPath(wl, rope_style=style, layer_inv_freq=freqs)


@pytest.mark.parametrize("name", list(CASES))
def test_shared_documents_bit_identical(cuda_lib, name):
    import paper_2607_28069_gb300 as pic
    path = _path(name)
    spec = path.wl.spec
    # the group size is what the test says it is
    row = spec.kv_heads * spec.head_dim
    tokens = spec.batch * spec.docs_per_request * path.wl.k_pool.shape[1] / spec.pool_docs
    chunk = 8 if row >= 1024 else 16 if row >= 512 else 32
    large = 8 * tokens * row * spec.layers >= 128e6
    group = max(1, min(8, int(tokens / chunk / 912))) if large else 1
    assert group == CASES[name][3]
    path.compose()
    path.relocate_mapped()
    k_ref, v_ref = path.k_cache.clone(), path.v_cache.clone()
    path.k_cache.zero_(), path.v_cache.zero_()
    path.relocate()
    assert torch.equal(path.k_cache, k_ref) and torch.equal(path.v_cache, v_ref)
    # pic_link against the three calls: caches, layout, packed queries
    path.append(0)
    k_ref, v_ref = path.k_cache.clone(), path.v_cache.clone()
    packed = path.B * spec.kv_heads * (-(-path.max_inline * spec.q_heads // spec.kv_heads // 128) * 128) \
        * spec.head_dim * 2
    ws_ref = path.ws_prefill[:packed].clone()
    maps = ("doc_offset", "doc_delta", "slot_mapping", "tok_map", "inline_pos", "ctx_len")
    ref = {m: getattr(path, m).clone() for m in maps}
    path.k_cache.zero_(), path.v_cache.zero_(), path.ws_prefill.zero_()
    for m in maps:
        getattr(path, m).fill_(-7)
    before = pic.pic_launch_count()
    path.link(0)
    assert pic.pic_launch_count() - before == 3
    assert torch.equal(path.k_cache, k_ref) and torch.equal(path.v_cache, v_ref)
    assert torch.equal(path.ws_prefill[:packed], ws_ref)
    for m in maps:
        assert torch.equal(getattr(path, m), ref[m]), m
    assert pic.pic_device_status() == (0, 0)


def test_large_link_refuses_what_the_small_one_does(cuda_lib):
    """Device checks of the three-launch link: a request with a negative
    prefix is left alone (nothing of it is written), one with a document id
    outside the pool is refused as a whole, the others are linked."""
    import paper_2607_28069_gb300 as pic
    path = _path("pairs")
    path.link(0)
    good = path.k_cache.clone()
    bt = path.wl.block_table
    path.k_cache.zero_(), path.v_cache.zero_()
    path.wl.prefix_len = path.wl.prefix_len.clone()
    path.wl.prefix_len[0] = -1
    path.wl.req_doc_ids = path.wl.req_doc_ids.clone()
    path.wl.req_doc_ids[1, 2] = 99
    path.link(0)
    assert pic.pic_device_status()[0] in (1, 3)
    assert path.ctx_len.tolist()[:2] == [-1, -1]
    pages = lambda b: bt[b][bt[b] >= 0].long()  # noqa: E731
    assert not path.k_cache[:, pages(0)].any()
    assert not path.k_cache[:, pages(1)].any()
    assert torch.equal(path.k_cache[:, pages(2)], good[:, pages(2)])


def test_large_links_back_to_back(cuda_lib):
    """Large links with different prefixes, document orders and block tables,
    one right behind the other into the same layout buffers: each link's caches
    and packed queries against the three separate calls, bit for bit.  (A
    launch of the chain that read the layout before its wait would find the
    link's before.)"""
    import paper_2607_28069_gb300 as pic
    path = _path("pairs")
    wl, spec = path.wl, path.wl.spec
    gen = torch.Generator().manual_seed(5)
    requests = []
    for i in range(4):
        prefix = wl.prefix_len - torch.randint(0, 3, (path.B,), generator=gen, dtype=torch.int32).cuda() * (i > 0)
        order = torch.randperm(spec.docs_per_request, generator=gen).cuda()
        pages = torch.randperm(wl.num_pages, generator=gen).int().cuda()
        requests.append(dict(prefix_len=prefix, inline_len=prefix + wl.query_len,
                             req_doc_ids=wl.req_doc_ids[:, order].contiguous(),
                             block_table=pages[wl.block_table.long().clamp(min=0)].contiguous()))
    kc = [torch.zeros_like(path.k_cache) for _ in requests]
    vc = [torch.zeros_like(path.v_cache) for _ in requests]
    ws = [torch.zeros_like(path.ws_prefill) for _ in requests]

    def take(i):
        for name, value in requests[i].items():
            setattr(wl, name, value)
        path.k_cache, path.v_cache, path.ws_prefill = kc[i], vc[i], ws[i]

    ref = []
    for i in range(len(requests)):
        take(i)
        path.compose(), path.relocate_mapped(), path.append(0)
        ref.append((kc[i].clone(), vc[i].clone(), ws[i].clone()))
    for _ in range(5):
        for t in kc + vc + ws:
            t.zero_()
        for i in range(len(requests)):
            take(i)
            path.link(0)
        for got, want in zip(zip(kc, vc, ws), ref):
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert pic.pic_device_status() == (0, 0)


@pytest.mark.parametrize("docs,capacity,launches", [((4, 300), 1, 1), ((4, 300), 8, 1),
                                                    ((4, 300), 32, 3), ((40, 1000), 1, 3)])
def test_link_form_follows_the_documents(cuda_lib, docs, capacity, launches):
    """The link of a short request stays one launch where the capacity max_ctx is
    several times its context; many CTAs or much to move make it three.  Both
    forms give the three separate calls' caches and layout, bit for bit."""
    import paper_2607_28069_gb300 as pic
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    spec = _spec("form", layers=2, q_heads=32, kv_heads=8, head_dim=128, batch=2, pool_docs=docs[0],
                 docs_per_request=docs[0], doc_len=(docs[1], docs[1]))
    wl = generate(spec, device="cuda", gen_device="cuda")
    table = torch.full((2, wl.block_table.shape[1] * capacity), -1, dtype=torch.int32, device="cuda")
    table[:, :wl.block_table.shape[1]] = wl.block_table
    wl.block_table, wl.max_ctx = table, wl.max_ctx * capacity
    path = CacheHitPath(wl)
    path.compose(), path.relocate_mapped(), path.append(0)
    maps = ("doc_offset", "doc_delta", "slot_mapping", "tok_map", "inline_pos", "ctx_len")
    ref = [path.k_cache.clone(), path.v_cache.clone()] + [getattr(path, m).clone() for m in maps]
    path.k_cache.zero_(), path.v_cache.zero_()
    before = pic.pic_launch_count()
    path.link(0)
    assert pic.pic_launch_count() - before == launches
    got = [path.k_cache, path.v_cache] + [getattr(path, m) for m in maps]
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
    assert pic.pic_device_status() == (0, 0)
