"""Performance cases of the cache-hit path.

Each case is one call (or one pass) that a serving program makes through the
public entry points: ``CacheHitPath`` (pipeline.py) where a pass is several
calls, the ``pic_*`` functions of the package otherwise.  Sizes are those of
workloads.py, bench.py and the parity tests, or lie between them; values are
the N(0,1) bf16 draws of workloads.py, with the queries scaled up in some
cases so that the softmax has the peaks that trained models show.

A case is a dict of plain values: ``kind`` names the call, the other keys the
request shape (see ``_spec``), the rotary options and the query scale.
``exact`` restates layout, re-rotation (Eq. 3), stitching and GQA attention in
64 bits with plain torch.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2607_28069_gb300 as pic
from paper_2607_28069_gb300.pipeline import CacheHitPath
from paper_2607_28069_gb300.workloads import custom_spec, draw_structure, generate

DEV = "cuda"
EDGES = (0.0, 0.1, 0.9)  # the paper's pre and int regions

# (query heads, kv heads, head dim, RoPE base): the geometries of workloads.py
# and of the parity tests (GQA groups of 4, 7, 8 and 16; head dims 64 and 128)
GEOMS = {
    "32/8/128": (32, 8, 128, 5e5),
    "28/4/128": (28, 4, 128, 1e6),
    "8/2/128": (8, 2, 128, 5e5),
    "32/2/128": (32, 2, 128, 5e5),
    "16/2/64": (16, 2, 64, 1e4),
    "4/1/64": (4, 1, 64, 1e4),
}


def _case(kind, geom, batch, docs, doc_len, prefix, query, layers=1, pool=None, span=(0, 0),
          base_hi=0, rope_style=0, layer_rope=False, q_scale=1.0, lse=False):
    return dict(kind=kind, geom=geom, layers=layers, batch=batch, docs=docs,
                pool=pool or docs, doc_lo=doc_len[0], doc_hi=doc_len[1], prefix_lo=prefix[0],
                prefix_hi=prefix[1], query=query, span_lo=span[0], span_hi=span[1],
                base_hi=base_hi, rope_style=rope_style, layer_rope=layer_rope,
                q_scale=q_scale, lse=lse)


def listed():
    c = []

    def add(name, *a, **k):
        c.append(dict(_case(*a, **k), name=name))

    # The smallest request: two short records behind a 16-token prefix (the
    # "tiny" workload), link + attention.  Launches and host work only.
    add("ttft_tiny", "ttft", "4/1/64", 1, 2, (64, 64), (16, 16), 16)
    # One request of multi-document QA, one layer (the "llama8b_1layer"
    # workload): what a layer costs when requests come one at a time.
    add("ttft_1req", "ttft", "32/8/128", 1, 8, (512, 512), (64, 64), 128, pool=32, q_scale=2.0)
    # An ordinary serving batch: four layers of the batch-8 workload (16 of 64
    # shared documents each, ~16.8k positions), the whole pass to the first
    # token: link, then per layer append, attention and split merge.
    add("ttft_b8", "ttft", "32/8/128", 8, 16, (1024, 1024), (32, 128), 256, layers=4, pool=64)
    # A pass as served: inputs read from and outputs written to pinned host
    # memory, two layers of one request (both copy routes run).
    add("served_1req", "served", "32/8/128", 1, 8, (512, 512), (64, 64), 128, layers=2, pool=32)
    # One layer's prefill of a ragged batch with a 64-wide head, interleaved
    # RoPE, GQA groups of 8, documents of odd lengths, LSE wanted.
    add("prefill_d64_ragged", "prefill", "16/2/64", 5, 9, (37, 1201), (3, 61), 203, pool=12,
        rope_style=1, q_scale=2.0, lse=True)
    # The longest contexts: one layer of the 4 x ~139k-token workload, every
    # document of the pool in a shuffled order, 512-token query chunk.
    add("prefill_128k", "prefill", "32/8/128", 4, 128, (128, 2048), (64, 64), 512)
    # Rotate-on-load (documents read from the pool, no stitched copy), one
    # layer of the batch-8 workload with an inline span after each document.
    add("fused_spans_b8", "fused", "32/8/128", 8, 16, (1024, 1024), (32, 128), 256, pool=64,
        span=(16, 64))
    # Relocation alone, documents of mixed lengths compiled at various bases,
    # four layers: the bandwidth-bound stitch.
    add("relocate_b8", "relocate", "32/8/128", 8, 16, (300, 1700), (32, 128), 64, layers=4,
        pool=64, base_hi=2000)
    # The fused link step with a rotary table per layer and a narrow cache row.
    add("link_layer_rope", "link", "28/4/128", 6, 20, (200, 1024), (5, 70), 100, layers=3, pool=40,
        layer_rope=True)
    # Decoding one request (a chat after a cache hit): one step, two layers.
    add("decode_1req", "decode", "32/8/128", 1, 8, (512, 512), (64, 64), 128, layers=2, pool=32,
        q_scale=2.0)
    # Decoding a batch over ~33k-token contexts, four layers of the batch-16
    # workload.
    add("decode_b16", "decode", "28/4/128", 16, 32, (1024, 1024), (64, 64), 128, layers=4, pool=64)
    # The attention-deviation diagnostic over one layer of two requests.
    add("deviation_b2", "deviation", "32/8/128", 2, 16, (700, 1024), (32, 128), 256, pool=24)
    return c


# ---------------------------------------------------------------- drawn cases
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    """One more case of the listed ranges: any kind, any geometry, sizes
    log-uniform from the smallest listed ones to the largest."""
    top = None
    while True:
        kind = rng.choice(["ttft", "ttft", "served", "prefill", "prefill", "fused", "relocate",
                           "link", "decode", "decode", "deviation"])
        geom = rng.choice(list(GEOMS))
        batch = _log_int(rng, 1, 16)
        docs = _log_int(rng, 2, 128)
        hi = _log_int(rng, 64, 2048)
        lo = rng.choice([hi, max(1, hi // rng.randint(2, 16))])
        phi = rng.choice([0, rng.randint(1, 130)])
        plo = rng.randint(0, phi)
        query = _log_int(rng, 1, 512)
        layers = rng.choice([1, 1, 2, 3, 4]) if kind in ("ttft", "served", "relocate", "link",
                                                         "decode") else 1
        span = rng.choice([(0, 0), (0, 0), (0, rng.randint(1, 64))])
        case = _case(kind, geom, batch, docs, (lo, hi), (plo, phi), query, layers=layers,
                     pool=docs + rng.randint(0, docs), span=span,
                     base_hi=rng.choice([0, 0, 2000, 140000]), rope_style=rng.randint(0, 1),
                     layer_rope=layers > 1 and rng.random() < 0.25,
                     q_scale=rng.choice([1.0, 1.0, 2.0]), lse=rng.random() < 0.3)
        w = work(case)
        if top is None:
            ws = [work(x) for x in listed()]
            top = (max(x["bytes"] for x in ws), max(x["flops"] for x in ws))
        # positions held on the device bound the memory and the preparation
        held = batch * (docs * hi + phi + docs * span[1] + query) * layers
        if (w["bytes"] < top[0] and w["flops"] < 0.5 * top[1] and held < 1_500_000 and
                (kind != "served" or batch * layers * (phi + query + docs * span[1]) < 4000)):
            return case


# ------------------------------------------------------------- input building
def _spec(c):
    hq, hkv, d, base = GEOMS[c["geom"]]
    return custom_spec(name=c["kind"], layers=c["layers"], q_heads=hq, kv_heads=hkv, head_dim=d,
                       rope_base=base, batch=c["batch"], pool_docs=c["pool"],
                       docs_per_request=c["docs"], doc_len=(c["doc_lo"], c["doc_hi"]),
                       prefix_len=(c["prefix_lo"], c["prefix_hi"]), query_len=c["query"],
                       span_len=(c["span_lo"], c["span_hi"]), base_pos=(0, c["base_hi"]),
                       decode_steps=1 if c["kind"] == "decode" else 0)


def _structure(c, seed):
    """The selections of a case: lengths and choices from the case alone (so
    that every seed has the same shapes), each request's document order and
    the physical pages from the seed."""
    st = draw_structure(_spec(c), 1)
    rng = np.random.default_rng(seed)
    st.docs = [[int(x) for x in rng.permutation(ids)] for ids in st.docs]
    perm = rng.permutation(st.num_pages).astype(np.int32)
    st.block_table = np.where(st.block_table >= 0, perm[st.block_table], np.int32(-1))
    return st


def _workload(c, seed):
    wl = generate(_spec(c), device=DEV, gen_device=DEV, value_seed=seed, select_seed=1)
    st = _structure(c, seed)
    wl.req_doc_ids = torch.tensor(st.docs, dtype=torch.int32, device=DEV)
    wl.block_table = torch.as_tensor(st.block_table, dtype=torch.int32).to(DEV)
    wl.meta["docs"] = st.docs
    if c["q_scale"] != 1.0:
        wl.q_inline.mul_(c["q_scale"])  # a power of two: exact in bf16
        if wl.q_dec is not None:
            wl.q_dec.mul_(c["q_scale"])
    return wl


def _layer_freqs(c):
    """A rotary table per layer: bases 1e4 and 5e5 in turn."""
    d = GEOMS[c["geom"]][2]
    i = torch.arange(d // 2, dtype=torch.float64)
    return torch.stack([torch.pow(torch.tensor(1e4 if l % 2 == 0 else 5e5, dtype=torch.float64),
                                  -2.0 * i / d) for l in range(c["layers"])]).to(DEV)


def prepare(case, seed):
    c = case
    wl = _workload(c, seed)
    path = CacheHitPath(wl, with_lse=c["lse"] or c["kind"] == "deviation",
                        rope_style=c["rope_style"],
                        layer_inv_freq=_layer_freqs(c) if c["layer_rope"] else None)
    s = SimpleNamespace(kind=c["kind"], wl=wl, path=path)
    # rows past a request's inline tokens are never written
    path.out.zero_()
    if path.lse is not None:
        path.lse.zero_()
    if s.kind == "served":
        s.host_in = path.pack_request_inputs()
        s.host_out = torch.zeros(path.out.shape, dtype=path.out.dtype, pin_memory=True)
        s.up, s.down = torch.cuda.Stream(), torch.cuda.Stream()
    if s.kind in ("prefill", "fused", "relocate", "decode", "deviation"):
        path.compose()
    if s.kind in ("prefill", "decode", "deviation"):
        path.relocate()
    if s.kind == "decode":  # the prompt's inline tokens are in the cache already
        for layer in range(c["layers"]):
            path.append(layer)
    if s.kind == "deviation":
        # configuration B: the documents at their compiled positions
        path.prefill(0)
        s.k_b, s.lse_a = path.k_cache.clone(), path.lse[0].clone()
        v_b = path.v_cache.clone()
        pic.pic_relocate_mapped(path.geom, wl.k_pool, wl.v_pool, path.tok_map,
                                torch.zeros_like(path.doc_delta), path.slot_mapping, wl.num_pages,
                                s.k_b, v_b, 0, 1)
        s.lse_b = torch.zeros_like(s.lse_a)
        out_b = torch.zeros_like(path.out[0])
        pic.pic_attend_prefill(path.geom, 0, path.inline_pos, wl.inline_len, path.max_ctx,
                               wl.block_table, wl.num_pages, s.k_b, v_b, out_b, s.lse_b,
                               path.prefill_splits, path.ws_prefill)
        R = len(EDGES) - 1
        s.sums = torch.zeros((c["batch"], R), dtype=torch.float64, device=DEV)
        s.counts = torch.zeros((c["batch"], R), dtype=torch.int64, device=DEV)
    return s


# ------------------------------------------------------------------- one pass
def run(state):
    s, path, wl = state, state.path, state.wl
    if s.kind == "ttft":
        path.ttft_pass()
        out = {"out": path.out, "k_cache": path.k_cache, "v_cache": path.v_cache,
               "ctx_len": path.ctx_len, "inline_pos": path.inline_pos}
    elif s.kind == "served":
        path.served_pass(s.host_in, s.host_out, s.up, s.down)
        return {"out": s.host_out, "k_cache": path.k_cache, "v_cache": path.v_cache}
    elif s.kind == "prefill":
        path.prefill(0)
        out = {"out": path.out, "k_cache": path.k_cache, "v_cache": path.v_cache}
    elif s.kind == "fused":
        pic.pic_attend_prefill_fused(path.geom, 0, path.inline_pos, wl.inline_len, path.max_ctx,
                                     wl.block_table, wl.num_pages, path.k_cache, path.v_cache,
                                     wl.k_pool, wl.v_pool, path.tok_map, path.doc_delta,
                                     path.out[0], None if path.lse is None else path.lse[0],
                                     path.prefill_splits, path.ws_prefill, q=wl.q_inline[0],
                                     k_new=wl.k_inline[0], v_new=wl.v_inline[0])
        out = {"out": path.out, "k_cache": path.k_cache, "v_cache": path.v_cache}
    elif s.kind == "relocate":
        path.relocate()
        return {"k_cache": path.k_cache, "v_cache": path.v_cache}
    elif s.kind == "link":
        path.link(0)
        return {"k_cache": path.k_cache, "v_cache": path.v_cache, "doc_offset": path.doc_offset,
                "doc_delta": path.doc_delta, "slot_mapping": path.slot_mapping,
                "tok_map": path.tok_map, "inline_pos": path.inline_pos, "ctx_len": path.ctx_len}
    elif s.kind == "decode":
        path.decode_pass(0)
        out = {"out": path.dec_out, "k_cache": path.k_cache, "v_cache": path.v_cache}
        if path.dec_lse is not None:
            out["lse"] = path.dec_lse
        return out
    else:
        pic.pic_attention_deviation(path.geom, 0, path.inline_pos, wl.inline_len, wl.query_len,
                                    wl.req_doc_ids, wl.doc_len, path.doc_offset,
                                    path.slot_mapping, wl.num_pages, path.k_cache, s.k_b, s.lse_a,
                                    s.lse_b, path.ws_prefill, s.sums, s.counts, edges=EDGES,
                                    max_query_len=wl.spec.query_len)
        return {"sums": s.sums, "counts": s.counts}
    if path.lse is not None:
        out["lse"] = path.lse
    return out


# ----------------------------------------------------------------- its floor
def _positions(st, b, query):
    """Inline positions (prefix, spans, query) and document offsets of request b."""
    pos, off, offs = list(range(st.prefixes[b])), st.prefixes[b], []
    for k, i in enumerate(st.docs[b]):
        offs.append(off)
        off += int(st.lens[i])
        pos += range(off, off + st.spans[b][k])
        off += st.spans[b][k]
    pos += range(off, off + query)
    return pos, offs, off + query


def work(case):
    """Bytes: every input read once and every output written once (documents,
    inline projections, cache slots, outputs).  Flops: both contractions over
    the visible (query, key) pairs."""
    c = case
    hq, hkv, d, _ = GEOMS[c["geom"]]
    st = draw_structure(_spec(c), 1)
    row = hkv * d * 2  # one token's K (or V)
    doc_tokens = inline = pairs = ctx_total = dev_pairs = 0
    for b in range(c["batch"]):
        pos, _, ctx = _positions(st, b, c["query"])
        n = sum(int(st.lens[i]) for i in st.docs[b])
        doc_tokens += n
        inline += len(pos)
        pairs += sum(p + 1 for p in pos)
        ctx_total += ctx
        dev_pairs += c["query"] * int(0.9 * n)
    L, k = c["layers"], c["kind"]
    pool_tokens = min(int(st.lens.sum()), doc_tokens)  # a shared document counts once
    # inline q, k, v read, k and v slots and out written
    io = inline * (2 * hq * d * 2 + 4 * row)
    attn = 4.0 * d * hq * pairs
    stitch = 2 * row * (pool_tokens + doc_tokens)
    if k in ("ttft", "served"):
        return {"bytes": L * (stitch + io), "flops": L * attn}
    if k == "prefill":
        return {"bytes": 2 * row * doc_tokens + io, "flops": attn}
    if k == "fused":
        return {"bytes": 2 * row * pool_tokens + io, "flops": attn}
    if k == "relocate":
        return {"bytes": L * stitch, "flops": 0.0}
    if k == "link":
        return {"bytes": L * stitch + inline * (2 * hq * d * 2 + 4 * row), "flops": 0.0}
    if k == "decode":
        return {"bytes": L * (2 * row * ctx_total + c["batch"] * (2 * hq * d * 2 + 4 * row)),
                "flops": L * 4.0 * d * hq * ctx_total}
    return {"bytes": 2 * row * doc_tokens + c["batch"] * c["query"] * hq * d * 2,
            "flops": 2 * 2.0 * d * hq * dev_pairs}


def tolerance(case):
    """About four times the error measured against ``exact`` at these sizes
    (attention 2.3e-3 .. 4.6e-3: keys, queries, probabilities and outputs in
    bf16, sums in 32 bits; deviation sums 5e-6 here, more with fewer terms)."""
    k = case["kind"]
    if k in ("relocate", "link"):  # one bf16 rounding of a 32-bit rotation; values are copies
        return {"rel": 4e-3, "max": 8e-3}
    if k == "deviation":
        return {"rel": 2e-4}
    return {"rel": 1.5e-2, "max": 0.15}


# --------------------------------------------------------- the same in 64 bits
def _rotate(x, angle, style):
    """x [..., d] rotated pair by pair by angle [..., d/2] (broadcast over heads)."""
    cos, sin = torch.cos(angle), torch.sin(angle)
    if style == pic.ROPE_HALF:
        h = x.shape[-1] // 2
        u, w = x[..., :h], x[..., h:]
        return torch.cat([u * cos - w * sin, u * sin + w * cos], dim=-1)
    u, w = x[..., 0::2], x[..., 1::2]
    return torch.stack([u * cos - w * sin, u * sin + w * cos], dim=-1).flatten(-2)


def _attend64(q, K, V, pos):
    """q [T, Hq, d] rotated, K/V [ctx, Hkv, d]: outputs [T, Hq, d] and LSE [T, Hq]."""
    T, hq, d = q.shape
    hkv = K.shape[1]
    G = hq // hkv
    out, lse = torch.zeros_like(q), torch.zeros((T, hq), dtype=q.dtype, device=q.device)
    t0 = 0
    while t0 < T:
        step = max(1, min(T - t0, 40_000_000 // (G * (int(pos[min(T, t0 + 64) - 1]) + 1)), 64))
        t1 = t0 + step
        n = int(pos[t1 - 1]) + 1
        mask = torch.arange(n, device=q.device)[None, None, :] > pos[t0:t1, None, None]
        for g in range(hkv):
            qq = q[t0:t1, g * G:(g + 1) * G] / math.sqrt(d)
            sc = torch.matmul(qq.reshape(-1, d), K[:n, g].T).view(step, G, n)
            sc.masked_fill_(mask, -math.inf)
            m = sc.amax(-1, keepdim=True)
            sc.sub_(m).exp_()
            s = sc.sum(-1, keepdim=True)
            out[t0:t1, g * G:(g + 1) * G] = \
                torch.matmul(sc.view(-1, n), V[:n, g].contiguous()).view(step, G, d) / s
            lse[t0:t1, g * G:(g + 1) * G] = (m + s.log())[..., 0]
        t0 = t1
    return out, lse


def exact(case, seed):
    c = case
    wl = _workload(c, seed)
    st = _structure(c, seed)
    hq, hkv, d, base = GEOMS[c["geom"]]
    L, B, kind, style = c["layers"], c["batch"], c["kind"], c["rope_style"]
    f64 = torch.float64
    i = torch.arange(d // 2, dtype=f64, device=DEV)
    freqs = _layer_freqs(c) if c["layer_rope"] else \
        torch.pow(torch.tensor(base, dtype=f64, device=DEV), -2.0 * i / d).expand(L, d // 2)
    shape = (L, wl.num_pages, hkv, 16, d)
    kc, vc = torch.zeros(shape, dtype=f64, device=DEV), torch.zeros(shape, dtype=f64, device=DEV)
    T = wl.tin_max
    out = torch.zeros((L, B, T, hq, d), dtype=f64, device=DEV)
    lse = torch.zeros((L, B, T, hq), dtype=f64, device=DEV)
    dout = torch.zeros((L, B, hq, d), dtype=f64, device=DEV)
    dlse = torch.zeros((L, B, hq), dtype=f64, device=DEV)
    sums = torch.zeros((B, len(EDGES) - 1), dtype=f64, device=DEV)
    docs_in_cache = kind != "fused"
    inline_layers = {"relocate": 0, "link": 1}.get(kind, L)
    for b in range(B):
        pos_l, offs, ctx = _positions(st, b, c["query"])
        pos = torch.tensor(pos_l, device=DEV)
        n_pos = ctx + (1 if kind == "decode" else 0)
        t = torch.arange(n_pos, device=DEV)
        page = torch.as_tensor(st.block_table[b], device=DEV).long()[t // 16]
        for l in range(L):
            K = torch.zeros((n_pos, hkv, d), dtype=f64, device=DEV)
            V = torch.zeros_like(K)
            here = torch.zeros(n_pos, dtype=torch.bool, device=DEV)  # positions in the cache
            K0 = torch.zeros_like(K) if kind == "deviation" else None
            for k, o in enumerate(offs):
                j = int(st.docs[b][k])
                n, r = int(st.lens[j]), int(st.starts[j])
                kd = wl.k_pool[l, r:r + n].to(f64)
                K[o:o + n] = _rotate(kd, float(o - int(st.bases[j])) * freqs[l], style)
                if K0 is not None:
                    K0[o:o + n] = kd
                V[o:o + n] = wl.v_pool[l, r:r + n].to(f64)
                here[o:o + n] = docs_in_cache
            q = None
            if l < inline_layers:
                ang = (pos.to(f64)[:, None] * freqs[l])[:, None, :]
                n = len(pos_l)
                q = _rotate(wl.q_inline[l, b, :n].to(f64), ang, style)
                K[pos] = _rotate(wl.k_inline[l, b, :n].to(f64), ang, style)
                V[pos] = wl.v_inline[l, b, :n].to(f64)
                here[pos] = True
            if kind == "decode":
                ang = float(ctx) * freqs[l]
                K[ctx] = _rotate(wl.k_dec[0, l, b].to(f64), ang, style)
                V[ctx] = wl.v_dec[0, l, b].to(f64)
                here[ctx] = True
                qd = _rotate(wl.q_dec[0, l, b].to(f64), ang, style)
                o1, l1 = _attend64(qd[None], K, V, torch.tensor([ctx], device=DEV))
                dout[l, b], dlse[l, b] = o1[0], l1[0]
            elif kind not in ("relocate", "link", "deviation"):
                o1, l1 = _attend64(q, K, V, pos)
                out[l, b, :len(pos_l)], lse[l, b, :len(pos_l)] = o1, l1
            elif kind == "deviation":
                K0[pos] = K[pos]
                _deviation64(q[-c["query"]:], K, K0, pos[-c["query"]:], offs,
                             [int(st.lens[j]) for j in st.docs[b]], sums[b])
            at = here.nonzero()[:, 0]
            kc[l, page[at], :, at % 16] = K[at]
            vc[l, page[at], :, at % 16] = V[at]
    if kind == "deviation":
        return {"sums": sums, "counts": None}
    if kind == "relocate":
        return {"k_cache": kc, "v_cache": vc}
    if kind == "link":
        return {"k_cache": kc, "v_cache": vc, "doc_offset": None, "doc_delta": None,
                "slot_mapping": None, "tok_map": None, "inline_pos": None, "ctx_len": None}
    got = {"out": dout if kind == "decode" else out, "k_cache": kc, "v_cache": vc}
    if kind == "ttft":
        got.update(ctx_len=None, inline_pos=None)
    if c["lse"] and kind != "served":
        got["lse"] = dlse if kind == "decode" else lse
    return got


def _deviation64(q, KA, KB, pos, offs, lens, sums):
    """Adds sum |p_A - p_B| of the query rows q over each document region."""
    T, hq, d = q.shape
    hkv = KA.shape[1]
    G = hq // hkv
    n = KA.shape[0]
    region = torch.full((n,), -1, dtype=torch.long, device=q.device)
    for o, m in zip(offs, lens):
        for r in range(len(EDGES) - 1):
            region[o + math.ceil(EDGES[r] * m):o + math.ceil(EDGES[r + 1] * m)] = r
    step = max(1, 20_000_000 // (G * n))
    for t0 in range(0, T, step):
        t1 = min(T, t0 + step)
        mask = torch.arange(n, device=q.device)[None, :] > pos[t0:t1].repeat_interleave(G)[:, None]
        for g in range(hkv):
            qq = (q[t0:t1, g * G:(g + 1) * G] / math.sqrt(d)).reshape(-1, d)
            p = [torch.softmax(torch.matmul(qq, K[:, g].T).masked_fill_(mask, -math.inf), -1)
                 for K in (KA, KB)]
            diff = (p[0] - p[1]).abs_().sum(0)
            for r in range(len(EDGES) - 1):
                sums[r] += diff[region == r].sum()
