"""The native part of the Python binding: what it refuses before any call, and
sub-tensors given as tuples (tensor, i[, j])."""
import pytest
import torch

import paper_2607_28069_gb300 as pic


def _args(**kw):
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32)  # noqa: E731
    a = dict(doc_len=i32(2), doc_base_pos=i32(2), doc_token_start=torch.zeros(2, dtype=torch.int64),
             req_doc_ids=i32(1, 2), req_num_docs=i32(1), prefix_len=i32(1), query_len=i32(1),
             block_table=i32(1, 4), num_pages=4, max_ctx=64, max_inline=16, doc_offset=i32(1, 2),
             doc_delta=i32(1, 2), slot_mapping=torch.zeros((1, 64), dtype=torch.int64),
             tok_map=torch.zeros((1, 64), dtype=torch.int64), inline_pos=i32(1, 16), ctx_len=i32(1))
    a.update(kw)
    return a


def test_refusals_before_any_call():
    g = pic.Geometry(1, 4, 1, 64, 1e4)
    with pytest.raises(ValueError, match="doc_len must be a CUDA tensor"):
        pic.pic_compose(g, **_args())
    with pytest.raises(ValueError, match="doc_len is required"):
        pic.pic_compose(g, **_args(doc_len=None))
    with pytest.raises(TypeError):
        pic.pic_compose(g, **_args(doc_len=3))
    with pytest.raises(AttributeError):
        pic.pic_compose(None, **_args())
    bad = pic.Geometry(1, 4, 1, 64, 1e4, layer_inv_freq=torch.zeros((2, 32), dtype=torch.float64))
    with pytest.raises(ValueError, match="layer_inv_freq"):
        pic.pic_compose(bad, **_args())


@pytest.mark.gpu
def test_refusals_of_device_tensors(cuda_lib):
    g = pic.Geometry(1, 4, 1, 64, 1e4)
    dev = {k: v.cuda() if isinstance(v, torch.Tensor) else v for k, v in _args().items()}
    for name, value, text in (
            ("doc_len", dev["doc_len"].long(), "must be torch.int32, got torch.int64"),
            ("block_table", torch.zeros((1, 8), dtype=torch.int32, device="cuda")[:, ::2],
             "block_table must be contiguous"),
            ("req_doc_ids", dev["req_num_docs"], "req_doc_ids must have two dimensions")):
        with pytest.raises(ValueError, match=text):
            pic.pic_compose(g, **dict(dev, **{name: value}))


@pytest.mark.gpu
def test_sub_tensors_as_tuples(cuda_lib):
    src = torch.arange(3 * 4 * 32, dtype=torch.int32, device="cuda").view(3, 4, 32)
    dst = torch.zeros(32, dtype=torch.int32, device="cuda")
    for at in ((0, 0), (2, 3), (-1, 1)):
        pic.pic_copy_async(dst, (src, *at))
        assert torch.equal(dst, src[at])
    # a strided leading dimension, each sub-tensor contiguous
    wide = torch.as_strided(src, (3, 32), (128, 1))
    pic.pic_copy_async(dst, (wide, 1))
    assert torch.equal(dst, wide[1])
    with pytest.raises(IndexError):
        pic.pic_copy_async(dst, (src, 3, 0))
    with pytest.raises(IndexError):
        pic.pic_copy_async(dst, (src, 0, 0, 0, 0))
    with pytest.raises(ValueError, match="contiguous"):
        pic.pic_copy_async(dst, (src.transpose(1, 2), 0))
    with pytest.raises(ValueError, match="differ in size"):
        pic.pic_copy_async(dst, (src, 0))


@pytest.mark.gpu
def test_served_pass_host_buffers(cuda_lib):
    """served_pass takes the outputs' host buffer as one tensor or as a list of
    one per layer, and refuses buffers of another shape or type."""
    from paper_2607_28069_gb300.pipeline import CacheHitPath
    from paper_2607_28069_gb300.workloads import custom_spec, generate
    spec = custom_spec(name="served_forms", layers=3, q_heads=8, kv_heads=2, head_dim=64, rope_base=1e4,
                       batch=2, pool_docs=4, docs_per_request=3, doc_len=(20, 90), prefix_len=(3, 17),
                       query_len=11)
    path = CacheHitPath(generate(spec, device="cuda", gen_device="cuda"))
    host = path.pack_request_inputs()
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    path.out.zero_()
    out = torch.zeros(path.out.shape, dtype=path.out.dtype, pin_memory=True)
    path.served_pass(host, out, up, down)
    torch.cuda.synchronize()
    per_layer = [torch.zeros(path.out.shape[1:], dtype=path.out.dtype, pin_memory=True) for _ in range(3)]
    path.served_pass(host, per_layer, up, down)
    torch.cuda.synchronize()
    assert out.any() and torch.equal(torch.stack(per_layer), out)
    B, T = path.out.shape[1:3]
    for bad in (torch.zeros((3, B, T - 1) + path.out.shape[3:], dtype=path.out.dtype, pin_memory=True),
                torch.zeros(path.out.shape, dtype=torch.float16, pin_memory=True)):
        with pytest.raises(ValueError):
            path.served_pass(host, bad, up, down)
        torch.cuda.synchronize()
    for bad in (host[:-512], host.view(torch.int32), host.view(2, -1)):
        with pytest.raises(ValueError):
            path.served_pass(bad, out, up, down)
        torch.cuda.synchronize()
    with pytest.raises(TypeError):
        path.served_pass(host, ["no tensor"] * 3, up, down)
    torch.cuda.synchronize()
    assert pic.pic_device_status() == (0, 0)


@pytest.mark.gpu
def test_one_of_a_list_as_a_tuple(cuda_lib):
    src = [torch.arange(64, dtype=torch.int32, device="cuda").view(2, 32) + 100 * i for i in range(3)]
    dst = torch.zeros(32, dtype=torch.int32, device="cuda")
    for i, j in ((0, 0), (2, 1), (-1, 0)):
        pic.pic_copy_async(dst, (src, i, j))
        assert torch.equal(dst, src[i][j])
    for at in ((3, 0), (0, 2), (0, 0, 0, 0)):
        with pytest.raises(IndexError):
            pic.pic_copy_async(dst, (src, *at))
