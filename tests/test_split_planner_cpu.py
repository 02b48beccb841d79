"""Host-side split planning (no GPU): the inline positions the pipeline
derives on the host agree with the oracle's layout, and the planner returns
a count the kernels accept."""
import numpy as np
import pytest
import torch

import paper_2607_28069_gb300 as pic
from paper_2607_28069_gb300.pipeline import host_inline_positions
from paper_2607_28069_gb300.workloads import WORKLOADS, generate

from helpers import oracle_layout
from test_gpu_parity import SMALL


@pytest.mark.parametrize("name", ["tiny", "ragged_b3", "spans_b2", "boundary_blocks",
                                  "base_mixed", "no_docs"])
def test_host_inline_positions_match_the_oracle_layout(name):
    wl = generate(SMALL[name], device="cpu", gen_device="cpu")
    lens, pos = host_inline_positions(wl)
    for b in range(wl.spec.batch):
        ref = oracle_layout(wl, b).inline_pos
        assert int(lens[b]) == len(ref) == int(wl.inline_len[b])
        assert np.array_equal(pos[b, :len(ref)].numpy(), np.asarray(ref, dtype=np.int32))


def test_planner_returns_a_valid_split_count():
    spec = WORKLOADS["llama8b_32layer_b8"]
    g = pic.Geometry(1, spec.q_heads, spec.kv_heads, spec.head_dim, spec.rope_base)
    # query rows that see ~16.7k keys behind prefixes of 32..128 tokens
    B, tmax = 8, 128 + 256
    lens = torch.zeros(B, dtype=torch.int32)
    pos = torch.zeros((B, tmax), dtype=torch.int32)
    for b in range(B):
        p = 32 + 12 * b
        row = list(range(p)) + list(range(16384 + p, 16384 + p + 256))
        lens[b] = len(row)
        pos[b, :len(row)] = torch.tensor(row, dtype=torch.int32)
    s = pic.pic_prefill_plan_splits(g, 16384 + 128 + 256, lens, pos)
    assert 1 <= s <= 32
    # a single short request fills a fraction of the GPU: more splits than one
    one = pic.pic_prefill_plan_splits(g, 4096, torch.tensor([192], dtype=torch.int32),
                                      torch.arange(4096 - 192, 4096, dtype=torch.int32)[None])
    assert one > 1
    with pytest.raises(ValueError):
        pic.pic_prefill_plan_splits(g, 4096, lens, pos[0])


def test_decode_split_count_fills_the_gpu():
    """The automatic split count of a decoding step: CTAs for four waves (eight a
    streaming multiprocessor) with at least 16 pages each.  A batch of a few
    dozen (request, kv head) pairs is not left with one or two splits."""
    for hq, hkv, d in ((32, 8, 128), (28, 4, 128), (12, 12, 64), (16, 1, 64), (64, 64, 128)):
        g = pic.Geometry(1, hq, hkv, d, 5e5)
        for batch in (1, 3, 12, 16, 24, 200):
            for ctx in (1, 16, 17, 400, 2049, 4097, 33000, 140000):
                pages = -(-ctx // 16)
                want = min(-(-8 * 152 // (batch * hkv)), max(1, pages // 16), 64, pages)
                assert pic.pic_decode_num_splits(g, batch, ctx, 0) == want, (hkv, batch, ctx)


@pytest.mark.parametrize("heads,batch,ctx,query", [((32, 8, 128), 4, 1024, 16), ((28, 4, 128), 8, 1024, 1),
                                                   ((16, 2, 64), 16, 1024, 1), ((28, 4, 128), 4, 4096, 1),
                                                   ((8, 2, 128), 16, 1024, 16), ((16, 2, 64), 1, 1024, 512)])
def test_planner_keeps_rotate_on_load_in_one_wave(heads, batch, ctx, query):
    """Counts beyond the library's own suit the materialised grid, whose short
    pairs are cheap, but not rotate-on-load's clusters of two pairs, which then
    take a second wave; the one count both calls use stays at or below it."""
    hq, hkv, d = heads
    g = pic.Geometry(1, hq, hkv, d, 5e5)
    T = 56 + query
    lens = torch.full((batch,), T, dtype=torch.int32)
    row = list(range(56)) + list(range(56 + ctx, 56 + ctx + query))
    pos = torch.tensor([row] * batch, dtype=torch.int32)
    own = pic.pic_prefill_num_splits(g, batch, T, ctx + T, 0)
    assert 1 <= pic.pic_prefill_plan_splits(g, ctx + T, lens, pos) <= own
