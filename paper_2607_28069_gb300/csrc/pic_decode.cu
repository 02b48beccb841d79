// pic_attend_decode: one step of plain autoregressive decoding over the
// completed stitched cache (appendix "Position-Independent Linking": after the
// first token, generation proceeds as usual on the linked cache).
//
// Decode reads every cached key and value of the request once per step and
// does 2*G*d multiply-adds per key: HBM-bound, and for few short requests
// bound by launches and dependent round trips.  Launches per call (one layer):
//  1. decode_attn_kernel: one CTA per (key split, kv head, request), four
//     warps, each warp an independent stream over the split's pages (page
//     w, w+4, ...).  Lane 0 of each warp keeps a 3-deep ring of TMA loads
//     (one 16-key K page and V page, 128-byte swizzled so the ldmatrix reads
//     below are bank-conflict free).  While the first pages are in flight the
//     CTA rotates its group's queries at the token's position; the CTA whose
//     pages hold that position also rotates the new key, writes it and the
//     new value to the cache and puts both into its copy of the page (the
//     page it loads may or may not show its own store yet).  Scores S^T = K
//     q^T come from m16n8k16 warp MMAs with the page's 16 keys as M and up to
//     8 query heads of the GQA group as N; P^T is turned into the B operand
//     of the O^T += V^T P^T MMA in registers with movmatrix.  The four warps'
//     states are merged through shared memory at the end.
//  2. decode_combine_kernel (only with several splits): log-sum-exp merge.
//     4 to 16 splits run as a thread-block cluster instead, where the GPU
//     holds all of them at once, and merge through distributed shared memory,
//     with no second launch.
#include <algorithm>
#include <mutex>

#include "pic_internal.cuh"

namespace pic {
namespace decode {

constexpr int kWarps = 4;
constexpr int kThreads = 32 * kWarps;
constexpr int NSTG = 3;
constexpr int kMaxSplits = 64;
// The splits of one (request, kv head) run as a cluster, merged through
// distributed shared memory, where there are 4 to 16 of them, the groups have up
// to 8 query heads, and the GPU holds all clusters at once (use_cluster).  us
// per layer against the merge launch: one request, 8/2 heads, 400 keys, 16 splits
// 5.27 and 6.67; over 1700 such shapes 0.96 of its time on average.  Clusters
// that wait for others to end take 1.34 to 1.88 times as long as CTAs with the
// merge launch, because a cluster needs its SMs in one GPC at once (14 clusters
// of 16 fit at d = 128, 224 CTAs of the 304 that fit without); two or three
// splits gain nothing (1.00 to 1.02), groups of more than 8 heads lose (1.01 to
// 1.17, at four splits 1.05).
constexpr int kMinCluster = 4, kMaxCluster = 16;
constexpr long long kClusterCtas = 304;  // two CTAs an SM; larger grids are not launch-bound

template <int D>
struct Layout {
  static constexpr int kPage = 16 * D * 2;        // one K (or V) page of one head
  static constexpr int kStage = 2 * kPage;        // K + V
  static constexpr int kWarpBytes = NSTG * kStage;
  static constexpr int kBar = kWarps * kWarpBytes;
  static constexpr int kCs = kBar + kWarps * NSTG * 8 + 16;  // cos/sin at the position (float2)
  static constexpr int kNew = kCs + D / 2 * 8;               // new key, new value (bf16)
  static constexpr int kQ = kNew + 2 * D * 2;                // rotated queries of the group (bf16)
  static constexpr int kBytes = kQ + 16 * D * 2;
  static constexpr int kAlloc = kBytes + 1024;
};

struct Params {
  int Hq, Hkv, G, max_pages, splits, pages_per_split, pos_offset;
  long long num_pages, layer_row0;
  int layer;
  const int32_t *pos, *block_table;
  const __nv_bfloat16 *q, *k_new, *v_new;  // un-rotated: [B][Hq][D], [B][Hkv][D]
  __nv_bfloat16 *k_cache, *v_cache;        // at the layer
  __nv_bfloat16 *out;
  float *lse, *part_o, *part_ml;
  int32_t *status;
  float scale_log2;
};

template <int D, int NT, bool kCluster>
__global__ void __launch_bounds__(kThreads)
    decode_attn_kernel(const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, Params p, RopeParams rp) {
  using L = Layout<D>;
  constexpr int PANELS = D / 64;
  constexpr int KS = D / 16;  // k-steps over d
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kBar + kWarps * NSTG * 8);

  const int split = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;

  // set-up that reads nothing another kernel writes, then wait for the
  // kernel before (programmatic dependent launch)
  if (threadIdx.x == 0) {
    for (int i = 0; i < kWarps * NSTG; ++i) mbar_init(sbase + L::kBar + 8 * i, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (lane == 0) {
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // ---- the token's projections go out before its position is known: chunk
  // (8 pairs) tid of the group's queries, and the new key and value
  constexpr int KC = D / 16, VC = D / 8;
  const int tid = threadIdx.x;
  const PairChunk pc = pair_chunk(tid % KC, D / 2, rp.style);
  const bool has_q = tid < p.G * KC;  // G <= 16: one chunk per thread
  uint4 qa = make_uint4(0, 0, 0, 0), qb2 = qa, ka = qa, kb = qa, vn = qa;
  if (has_q) {
    const __nv_bfloat16 *src = p.q + ((size_t)b * p.Hq + hk * p.G + tid / KC) * D;
    qa = ld_stream(src + pc.off_a);
    qb2 = ld_stream(src + pc.off_b);
  }
  if (tid < KC) {
    const __nv_bfloat16 *src = p.k_new + ((size_t)b * p.Hkv + hk) * D;
    ka = ld_stream(src + pc.off_a);
    kb = ld_stream(src + pc.off_b);
  } else if (tid >= 32 && tid < 32 + VC) {
    vn = ld_stream(p.v_new + ((size_t)b * p.Hkv + hk) * D + (tid - 32) * 8);
  }

  // the block-table entries of this warp's first pages do not depend on the
  // position either (lane i: its page i)
  const int32_t *bt = p.block_table + (size_t)b * p.max_pages;
  const int pg_begin = split * p.pages_per_split;
  const int my_first = pg_begin + warp;  // pages of this warp: my_first + 4 i
  const int bt_first = lane < NSTG && my_first + kWarps * lane < p.max_pages
                           ? bt[my_first + kWarps * lane] : -1;
  const int pos = p.pos[b] + p.pos_offset;
  const int npages = pos >= 0 ? pos / 16 + 1 : 0;
  // max_ctx sized the split plan: keys past the last split's pages would be
  // left out, so that is a device-checked error (the step's output for the
  // request is then incomplete)
  if (split == p.splits - 1 && threadIdx.x == 0 && npages > p.splits * p.pages_per_split)
    dev_fail(p.status, PIC_DEV_CTX_OVERFLOW, b);
  const int pg_end = min(npages, pg_begin + p.pages_per_split);

  const uint32_t wbase = sbase + warp * L::kWarpBytes;
  auto full = [&](int s) { return sbase + L::kBar + 8u * (uint32_t)(warp * NSTG + s); };
  const int cw = my_first < pg_end ? (pg_end - my_first + kWarps - 1) / kWarps : 0;

  auto issue = [&](int i, int page_first) {  // lane 0 only; page_first: entry of page i < NSTG
    const int pidx = my_first + kWarps * i;
    int y = -1;
    if (pidx < p.max_pages) {
      const int page = i < NSTG ? page_first : bt[pidx];
      if (page >= 0 && page < p.num_pages) y = (int)(p.layer_row0 + ((long long)page * p.Hkv + hk) * 16);
      else dev_fail(p.status, PIC_DEV_BAD_PAGE, b);
    } else {
      dev_fail(p.status, PIC_DEV_BLOCK_TABLE_SHORT, b);
    }
    if (y < 0) y = 0x7fffff00;  // out of the tensor: TMA fills zeros
    const int s = i % NSTG;
    const uint32_t dst = wbase + s * L::kStage;
    mbar_expect_tx(full(s), L::kStage);
    for (int pn = 0; pn < PANELS; ++pn) {
      tma_load_2d(dst + pn * 2048, &tm_k, pn * 64, y, full(s));
      tma_load_2d(dst + L::kPage + pn * 2048, &tm_v, pn * 64, y, full(s));
    }
  };
#pragma unroll
  for (int i = 0; i < NSTG; ++i) {
    const int page_first = __shfl_sync(0xffffffffu, bt_first, i);
    if (lane == 0 && i < cw) issue(i, page_first);
  }

  // ---- rotation at the position while the pages are in flight; the CTA whose
  // pages hold the position appends the new key and value
  float2 *cs = reinterpret_cast<float2 *>(smem + L::kCs);
  __nv_bfloat16 *s_new = reinterpret_cast<__nv_bfloat16 *>(smem + L::kNew);
  __nv_bfloat16 *s_q = reinterpret_cast<__nv_bfloat16 *>(smem + L::kQ);
  const int new_pg = pos >= 0 ? pos >> 4 : -1, new_row = pos & 15;
  int new_page = -1;  // the new token's page, -1: not this CTA's, or invalid
  if (new_pg < 0 || new_pg >= p.max_pages) {
    if (split == 0 && hk == 0 && tid == 0) dev_fail(p.status, PIC_DEV_BAD_POSITION, b);
  } else if (new_pg >= pg_begin && (new_pg < pg_end || split == p.splits - 1)) {
    new_page = bt[new_pg];
    if (new_page < 0 || new_page >= p.num_pages) {
      if (tid == 0) dev_fail(p.status, PIC_DEV_BAD_PAGE, b);
      new_page = -1;
    }
  }
  if (tid < D / 2) cs[tid] = rope_cos_sin(max(pos, 0), rope_theta(rp, p.layer, tid));
  __syncthreads();
  if (has_q) rotate_store_as<true>(qa, qb2, s_q + (tid / KC) * D, pc, rp.style, cs + 8 * (tid % KC));
  if (new_page >= 0) {
    const size_t row = (((size_t)new_page * p.Hkv + hk) * 16 + new_row) * D;
    if (tid < KC) {
      rotate_store_as<true>(ka, kb, s_new, pc, rp.style, cs + 8 * tid);
      rotate_store_as<false>(ka, kb, p.k_cache + row, pc, rp.style, cs + 8 * tid);
    } else if (tid >= 32 && tid < 32 + VC) {
      *reinterpret_cast<uint4 *>(s_new + D + (tid - 32) * 8) = vn;
      st_global16(p.v_cache + row + (tid - 32) * 8, vn);
    }
  }
  __syncthreads();

  // query fragments (B operand of S^T = K q^T): heads nt*8 + gid of the group
  uint32_t qb[NT][KS][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int hh = nt * 8 + gid;
    const bool hv = hh < p.G;
    const uint32_t *qr = reinterpret_cast<const uint32_t *>(s_q + (hv ? hh : 0) * D);
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      qb[nt][kk][0] = hv ? qr[(kk * 16 + 2 * tig) / 2] : 0u;
      qb[nt][kk][1] = hv ? qr[(kk * 16 + 8 + 2 * tig) / 2] : 0u;
    }
  }

  float m[NT][2], l[NT][2], o[NT][KS][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
    for (int j = 0; j < 2; ++j) { m[nt][j] = -INFINITY; l[nt][j] = 0.f; }
#pragma unroll
    for (int mt = 0; mt < KS; ++mt)
#pragma unroll
      for (int q = 0; q < 4; ++q) o[nt][mt][q] = 0.f;
  }

  int done = 0;
  for (int i = 0; i < cw; ++i) {
    const int s = i % NSTG;
    const bool ok = mbar_wait(full(s), (i / NSTG) & 1, abort_flag, p.status, b);
    if (!__all_sync(0xffffffffu, ok)) break;
    done = i + 1;
    const uint32_t ks = wbase + s * L::kStage, vs = ks + L::kPage;
    const int key0 = (my_first + kWarps * i) * 16;
    if (new_page >= 0 && my_first + kWarps * i == new_pg) {  // the new token's row of the page
      const int piece = lane % VC;
      if (lane < 2 * VC)
        sts128((lane < VC ? ks : vs) + (piece >> 3) * 2048 + sw128_offset(new_row, (piece & 7) * 8),
               *reinterpret_cast<const uint4 *>(s_new + (lane < VC ? 0 : D) + piece * 8));
      __syncwarp();
    }
    // ---- S^T[16 keys][8 heads] per n-tile
    float sacc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) sacc[nt][q] = 0.f;
    {
      const int mi = lane >> 3, rr = (mi & 1) * 8 + (lane & 7);
#pragma unroll
      for (int kk = 0; kk < KS; ++kk) {
        const int col = kk * 16 + (mi >> 1) * 8;
        uint32_t a[4];
        ldsm_x4(ks + (col >> 6) * 2048 + sw128_offset(rr, col & 63), a);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma16816(sacc[nt], a, qb[nt][kk][0], qb[nt][kk][1]);
      }
    }
    // ---- online softmax (thread: keys gid, gid+8; heads 2tig, 2tig+1 of each n-tile)
    const bool m0 = key0 + gid > pos, m1 = key0 + gid + 8 > pos;
    uint32_t pb[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float pv[2][2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float s0 = m0 ? -INFINITY : sacc[nt][j] * p.scale_log2;
        const float s1 = m1 ? -INFINITY : sacc[nt][2 + j] * p.scale_log2;
        float mx = fmaxf(s0, s1);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        const float mn = fmaxf(m[nt][j], mx);
        const float mref = mn == -INFINITY ? 0.f : mn;
        const float alpha = ex2(m[nt][j] - mref);
        m[nt][j] = mn;
        pv[0][j] = ex2(s0 - mref);
        pv[1][j] = ex2(s1 - mref);
        l[nt][j] = l[nt][j] * alpha + pv[0][j] + pv[1][j];
#pragma unroll
        for (int mt = 0; mt < KS; ++mt) {
          o[nt][mt][j] *= alpha;
          o[nt][mt][2 + j] *= alpha;
        }
      }
      pb[nt][0] = movm_t(pack2(pv[0][0], pv[0][1]));
      pb[nt][1] = movm_t(pack2(pv[1][0], pv[1][1]));
    }
    // ---- O^T[d][heads] += V^T P^T
    {
      const int mi = lane >> 3, rr = (mi >> 1) * 8 + (lane & 7);
#pragma unroll
      for (int mt = 0; mt < KS; ++mt) {
        const int col = mt * 16 + (mi & 1) * 8;
        uint32_t a[4];
        ldsm_x4_t(vs + (col >> 6) * 2048 + sw128_offset(rr, col & 63), a);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma16816(o[nt][mt], a, pb[nt][0], pb[nt][1]);
      }
    }
    __syncwarp();
    if (lane == 0 && i + NSTG < cw) issue(i + NSTG, -1);
  }

  if (done < cw) {
    // aborted: let the loads already issued land before the ring is reused
    for (int i = done; i < min(cw, done + NSTG); ++i)
      mbar_wait_no_flag(full(i % NSTG), (i / NSTG) & 1, p.status, b, kWaitLimitNs);
  }
  // ---- reduce l over the 8 key lanes, then merge the four warps
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float v = l[nt][j];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      l[nt][j] = v;
    }
  __syncthreads();  // every warp finished with its ring: reuse it for the merge
  constexpr int HMAX = NT * 8;
  float *so = reinterpret_cast<float *>(smem);                  // [warps][HMAX][D]
  float *sm = so + kWarps * HMAX * D;                            // [warps][HMAX]
  float *sl = sm + kWarps * HMAX;                                // [warps][HMAX]
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int hh = nt * 8 + 2 * tig + j;
      if (gid == 0) {
        sm[warp * HMAX + hh] = m[nt][j];
        sl[warp * HMAX + hh] = l[nt][j];
      }
#pragma unroll
      for (int mt = 0; mt < KS; ++mt) {
        so[(warp * HMAX + hh) * D + mt * 16 + gid] = o[nt][mt][j];
        so[(warp * HMAX + hh) * D + mt * 16 + gid + 8] = o[nt][mt][2 + j];
      }
    }
  __syncthreads();
  const bool single = p.splits == 1;
  float *c_acc = sl + kWarps * HMAX, *c_m = c_acc + HMAX * D, *c_l = c_m + HMAX;  // kCluster
  for (int e = threadIdx.x; e < p.G * D; e += kThreads) {
    const int hh = e / D, d = e % D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) M = fmaxf(M, sm[w * HMAX + hh]);
    float acc = 0.f, Ls = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float mw = sm[w * HMAX + hh];
      const float wt = mw == -INFINITY ? 0.f : ex2(mw - M);
      acc = fmaf(wt, so[(w * HMAX + hh) * D + d], acc);
      Ls = fmaf(wt, sl[w * HMAX + hh], Ls);
    }
    const size_t h = (size_t)b * p.Hq + hk * p.G + hh;
    if (single) {
      p.out[h * D + d] = __float2bfloat16_rn(Ls > 0.f ? acc / Ls : 0.f);
      if (d == 0 && p.lse) p.lse[h] = Ls > 0.f ? (M + __log2f(Ls)) * 0.69314718055994531f : -INFINITY;
    } else if constexpr (kCluster) {
      c_acc[e] = acc;
      if (d == 0) {
        c_m[hh] = Ls > 0.f ? M : -INFINITY;
        c_l[hh] = Ls;
      }
    } else {
      p.part_o[(h * p.splits + split) * D + d] = acc;
      if (d == 0) {
        p.part_ml[(h * p.splits + split) * 2] = Ls > 0.f ? M : -INFINITY;
        p.part_ml[(h * p.splits + split) * 2 + 1] = Ls;
      }
    }
  }
  if constexpr (kCluster) {
    // ---- the splits of this (request, kv head) are one cluster: each CTA
    // merges its share of the output elements, o = sum_s w_s O_s / sum_s w_s l_s
    // with w_s = 2^(m_s - M), from every CTA's shared memory
    cluster_sync_all();
    const int S = p.splits, per = (p.G * D + S - 1) / S;
    for (int e = split * per + (int)threadIdx.x; e < min(p.G * D, (split + 1) * per); e += kThreads) {
      const int hh = e / D, d = e % D;
      float ms[kMaxCluster], ls[kMaxCluster], os[kMaxCluster];
#pragma unroll
      for (int c = 0; c < kMaxCluster; ++c) {
        ms[c] = -INFINITY, ls[c] = 0.f, os[c] = 0.f;
        if (c < S) {
          ms[c] = ld_cluster(map_to_rank(smem_u32(c_m + hh), c));
          ls[c] = ld_cluster(map_to_rank(smem_u32(c_l + hh), c));
          os[c] = ld_cluster(map_to_rank(smem_u32(c_acc + e), c));
        }
      }
      float M = -INFINITY, acc = 0.f, Ls = 0.f;
#pragma unroll
      for (int c = 0; c < kMaxCluster; ++c) M = fmaxf(M, ms[c]);
#pragma unroll
      for (int c = 0; c < kMaxCluster; ++c) {
        const float w = ms[c] == -INFINITY ? 0.f : ex2(ms[c] - M);
        acc = fmaf(w, os[c], acc);
        Ls = fmaf(w, ls[c], Ls);
      }
      const size_t h = (size_t)b * p.Hq + hk * p.G + hh;
      p.out[h * D + d] = __float2bfloat16_rn(acc * (Ls > 0.f ? 1.f / Ls : 0.f));
      if (d == 0 && p.lse) p.lse[h] = Ls > 0.f ? (M + __log2f(Ls)) * 0.69314718055994531f : -INFINITY;
    }
  }
  // release the dependent launch (merge, or the next layer's step) last
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if constexpr (kCluster) cluster_sync_all();  // the others may still read this CTA's shared memory
}

// Merge of the split partials of one (request, query head) row by
// log-sum-exp: o = sum_s w_s O_s / sum_s w_s l_s with w_s = 2^(m_s - M).
// Lane s holds split s's (m, l) (and lane s - 32 split s >= 32), so the
// maximum and the weight sum are warp reductions, and the O rows of eight
// splits are loaded before any is used (the first sixteen together with
// the (m, l) pairs): a row costs a few L2 round trips however many splits
// it has, not one per split.
template <int D>
__global__ void decode_combine_kernel(Params p) {
  static_assert(kMaxSplits <= 64, "two (m, l) slots per lane");
  constexpr int CPL = D / 32, U = 8;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int h = blockIdx.x, b = blockIdx.y, lane = threadIdx.x;
  const size_t hrow = (size_t)b * p.Hq + h;
  const int S = p.splits;
  // the first sixteen splits' O rows go out with the (m, l) loads
  const float *src = p.part_o + hrow * S * D + lane;
  float v0[U][CPL], v1[U][CPL];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
      v0[u][q] = u < S ? src[(size_t)u * D + q * 32] : 0.f;
      v1[u][q] = U + u < S ? src[(size_t)(U + u) * D + q * 32] : 0.f;
    }
  float mA = -INFINITY, lA = 0.f, mB = -INFINITY, lB = 0.f;
  if (lane < S) {
    const float2 ml = *reinterpret_cast<const float2 *>(p.part_ml + (hrow * S + lane) * 2);
    mA = ml.x, lA = ml.y;
  }
  if (lane + 32 < S) {
    const float2 ml = *reinterpret_cast<const float2 *>(p.part_ml + (hrow * S + lane + 32) * 2);
    mB = ml.x, lB = ml.y;
  }
  float M = fmaxf(mA, mB);
#pragma unroll
  for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  const float wA = mA == -INFINITY ? 0.f : ex2(mA - M);
  const float wB = mB == -INFINITY ? 0.f : ex2(mB - M);
  float Ls = fmaf(wA, lA, wB * lB);
#pragma unroll
  for (int o = 16; o; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
  float acc[CPL];
#pragma unroll
  for (int q = 0; q < CPL; ++q) acc[q] = 0.f;
  for (int s0 = 0; s0 < S; s0 += U) {
    float v[U][CPL];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < CPL; ++q)
        v[u][q] = s0 == 0   ? v0[u][q]
                  : s0 == U ? v1[u][q]
                            : (s0 + u < S ? src[(size_t)(s0 + u) * D + q * 32] : 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int sp = s0 + u;
      if (sp >= S) break;
      const float w = __shfl_sync(0xffffffffu, sp < 32 ? wA : wB, sp & 31);
      if (w == 0.f) continue;  // an empty split; its rows were never written
#pragma unroll
      for (int q = 0; q < CPL; ++q) acc[q] = fmaf(w, v[u][q], acc[q]);
    }
  }
  const float inv = Ls > 0.f ? 1.f / Ls : 0.f;
#pragma unroll
  for (int q = 0; q < CPL; ++q) p.out[hrow * D + q * 32 + lane] = __float2bfloat16_rn(acc[q] * inv);
  if (lane == 0 && p.lse) p.lse[hrow] = Ls > 0.f ? (M + __log2f(Ls)) * 0.69314718055994531f : -INFINITY;
}

struct Plan {
  int splits, pages_per_split;
  // q_bytes: the start of the scratch, once the rotated queries, which stay in
  // shared memory now; kept so that the sizes callers have laid out still hold
  size_t q_bytes, po_bytes, pml_bytes, total;
};

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

inline Plan plan(const pic_geom_t *g, int batch, int max_ctx, int num_splits) {
  Plan pl;
  const int pages = (max_ctx + 15) / 16;
  if (num_splits <= 0) {
    // Four waves of CTAs with at least 16 pages each.  A count for whole waves of
    // resident CTAs and at most sqrt(pages) was faster by 8% on average over
    // 832 shapes (one request of 16k keys 24.1 -> 18.1 us a layer), but slower by
    // up to 46% where it chose one or two splits (12 requests of 2k keys, 12 heads
    // of 64: 15.8 -> 23.2 us, 12.4 with four), and fewer splits round more of the
    // probabilities (error against 64 bits +0.5 to 2.5%): not kept.
    const long long units = (long long)batch * g->num_kv_heads;
    int s = (int)((8LL * 152 + units - 1) / units);
    s = std::min(s, std::max(1, pages / 16));
    num_splits = std::max(1, std::min(s, kMaxSplits));
  }
  num_splits = std::min(num_splits, pages);
  pl.splits = std::max(1, num_splits);
  pl.pages_per_split = (pages + pl.splits - 1) / pl.splits;
  pl.q_bytes = align256((size_t)batch * g->num_q_heads * g->head_dim * 2);
  if (pl.splits > 1) {
    pl.po_bytes = align256((size_t)batch * g->num_q_heads * pl.splits * g->head_dim * 4);
    pl.pml_bytes = align256((size_t)batch * g->num_q_heads * pl.splits * 2 * 4);
  } else {
    pl.po_bytes = pl.pml_bytes = 0;
  }
  pl.total = pl.q_bytes + pl.po_bytes + pl.pml_bytes;
  return pl;
}

template <int D, int NT, bool kCluster>
cudaError_t allow_attn() {
  auto *kernel = decode_attn_kernel<D, NT, kCluster>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Layout<D>::kAlloc);
  if (kCluster && e == cudaSuccess)  // more than 8 CTAs
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <int D, int NT>
cudaError_t launch_attn(dim3 grid, cudaStream_t stream, const CUtensorMap &tk, const CUtensorMap &tv,
                        const Params &pp, const RopeParams &rp) {
  const cudaError_t e = allow_attn<D, NT, false>();
  if (e != cudaSuccess) return e;
  return launch_dependent(decode_attn_kernel<D, NT, false>, grid, dim3(kThreads), Layout<D>::kAlloc,
                          stream, tk, tv, pp, rp);
}

template <int D>
cudaError_t launch_attn_cluster(dim3 grid, cudaStream_t stream, const CUtensorMap &tk,
                                const CUtensorMap &tv, const Params &pp, const RopeParams &rp) {
  const cudaError_t e = allow_attn<D, 1, true>();
  if (e != cudaSuccess) return e;
  return launch_dependent_cluster(decode_attn_kernel<D, 1, true>, grid, dim3(kThreads),
                                  Layout<D>::kAlloc, stream, (int)grid.x, tk, tv, pp, rp);
}

// Clusters of `splits` CTAs that the current device holds at once; 0 also where
// it places none (a partition with few SMs a GPC) or does not say.  Asked once
// per device context and size: the answer takes the runtime 1.3 us.
template <int D>
int resident_clusters(int splits) {
  constexpr int kMaxDev = 64;
  struct Known {
    unsigned long long ctx;
    int count[kMaxCluster + 1];  // -1: not asked yet
  };
  static Known known[kMaxDev];
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  const unsigned long long id = current_context_id();
  std::lock_guard<std::mutex> lk(mu);
  Known &k = known[dev];
  if (id == 0 || id != k.ctx) {
    std::fill(k.count, k.count + kMaxCluster + 1, -1);
    k.ctx = id;
  }
  if (k.count[splits] < 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Layout<D>::kAlloc;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = allow_attn<D, 1, true>();
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveClusters(&n, decode_attn_kernel<D, 1, true>, &cfg);
    if (e != cudaSuccess) {
      cudaGetLastError();  // clear the error the failed query recorded
      n = 0;
    }
    k.count[splits] = n;
  }
  return k.count[splits];
}

inline bool use_cluster(int D, int group, int splits, long long heads) {
  if (group > 8 || splits < kMinCluster || splits > kMaxCluster || splits * heads > kClusterCtas)
    return false;
  return heads <= (D == 128 ? resident_clusters<128>(splits) : resident_clusters<64>(splits));
}

}  // namespace decode
}  // namespace pic

extern "C" size_t pic_decode_workspace_size(const pic_geom_t *geom, int32_t batch, int32_t max_ctx,
                                            int32_t num_splits) {
  if (!geom || batch <= 0 || max_ctx <= 0 || geom->num_kv_heads <= 0) return 0;
  return pic::decode::plan(geom, batch, max_ctx, num_splits).total;
}

extern "C" int32_t pic_decode_num_splits(const pic_geom_t *geom, int32_t batch, int32_t max_ctx,
                                         int32_t num_splits) {
  if (!geom || batch <= 0 || max_ctx <= 0 || geom->num_kv_heads <= 0 || num_splits < 0 ||
      num_splits > pic::decode::kMaxSplits)
    return 0;
  return pic::decode::plan(geom, batch, max_ctx, num_splits).splits;
}

namespace pic {
namespace decode {

// Host checks shared by pic_attend_decode and pic_attend_decode_noalloc
// (everything but the scratch); fills the rotary parameters.
static pic_status_t check_step(const char *who, const pic_geom_t *geom, RopeParams *rp,
                               int32_t layer, int32_t batch, const void *q, const void *k_new,
                               const void *v_new, const int32_t *pos, const int32_t *block_table,
                               int32_t max_pages, int64_t num_pages, const void *k_cache,
                               const void *v_cache, const void *out, int32_t max_ctx,
                               int32_t num_splits) {
  pic_status_t st = make_rope(geom, rp);
  if (st != PIC_OK) return st;
  if (layer < 0 || layer >= geom->num_layers)
    return fail(PIC_ERR_INVALID_ARG, "%s: layer %d outside [0, %d)", who, layer,
                geom->num_layers);
  if (batch <= 0 || max_pages <= 0 || num_pages <= 0 || max_ctx <= 0)
    return fail(PIC_ERR_INVALID_ARG, "%s: sizes must be positive", who);
  if (num_splits < 0 || num_splits > kMaxSplits)
    return fail(PIC_ERR_INVALID_ARG, "%s: num_splits %d outside [0, %d]", who, num_splits,
                kMaxSplits);
  if (geom->num_q_heads / geom->num_kv_heads > 16)
    return fail(PIC_ERR_UNSUPPORTED, "%s: more than 16 query heads per kv head", who);
  if (!q || !k_new || !v_new || !pos || !block_table || !k_cache || !v_cache || !out)
    return fail(PIC_ERR_INVALID_ARG, "%s: NULL tensor", who);
  if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k_new) |
       reinterpret_cast<uintptr_t>(v_new) | reinterpret_cast<uintptr_t>(k_cache) |
       reinterpret_cast<uintptr_t>(v_cache)) & 15)
    return fail(PIC_ERR_INVALID_ARG, "%s: bf16 tensors must be 16-byte aligned", who);
  const long long rows_total =
      (long long)geom->num_layers * num_pages * geom->num_kv_heads * 16;
  if (rows_total + 16 >= 0x7fffff00LL)
    return fail(PIC_ERR_UNSUPPORTED, "%s: cache has more than 2^31 rows", who);
  if (batch > 65535 || geom->num_kv_heads > 65535)
    return fail(PIC_ERR_UNSUPPORTED, "%s: grid too large", who);
  return PIC_OK;
}

// The launches of one decoding step of one layer (append and attention, merge
// when split) with the scratch at `ws` laid out by `pl`.
static pic_status_t launch_step(const char *who, const pic_geom_t *geom, const RopeParams &rp,
                                int32_t layer, int32_t batch, const void *q, const void *k_new,
                                const void *v_new, const int32_t *pos, int32_t pos_offset,
                                const int32_t *block_table, int32_t max_pages, int64_t num_pages,
                                void *k_cache, void *v_cache, void *out, float *lse,
                                const Plan &pl, uint8_t *ws, pic_stream_t stream) {
  int32_t *status = device_status_ptr();
  if (!status) return fail(PIC_ERR_CUDA, "%s: no device status word", who);
  const int D = geom->head_dim, Hkv = geom->num_kv_heads;
  const int G = geom->num_q_heads / Hkv;
  const long long rows_total = (long long)geom->num_layers * num_pages * Hkv * 16;
  const size_t layer_elems = (size_t)num_pages * Hkv * 16 * D;

  CUtensorMap tk, tv;
  pic_status_t st = encode_tmap_2d(&tk, k_cache, D, rows_total, (uint64_t)D * 2, 64, 16);
  if (st == PIC_OK) st = encode_tmap_2d(&tv, v_cache, D, rows_total, (uint64_t)D * 2, 64, 16);
  if (st != PIC_OK) return st;

  Params pp;
  pp.Hq = geom->num_q_heads;
  pp.Hkv = Hkv;
  pp.G = G;
  pp.max_pages = max_pages;
  pp.splits = pl.splits;
  pp.pages_per_split = pl.pages_per_split;
  pp.pos_offset = pos_offset;
  pp.num_pages = num_pages;
  pp.layer_row0 = (long long)layer * num_pages * Hkv * 16;
  pp.pos = pos;
  pp.block_table = block_table;
  pp.layer = layer;
  pp.q = static_cast<const __nv_bfloat16 *>(q);
  pp.k_new = static_cast<const __nv_bfloat16 *>(k_new);
  pp.v_new = static_cast<const __nv_bfloat16 *>(v_new);
  pp.k_cache = static_cast<__nv_bfloat16 *>(k_cache) + (size_t)layer * layer_elems;
  pp.v_cache = static_cast<__nv_bfloat16 *>(v_cache) + (size_t)layer * layer_elems;
  pp.out = static_cast<__nv_bfloat16 *>(out);
  pp.lse = lse;
  pp.part_o = pl.splits > 1 ? reinterpret_cast<float *>(ws + pl.q_bytes) : nullptr;
  pp.part_ml = pl.splits > 1 ? reinterpret_cast<float *>(ws + pl.q_bytes + pl.po_bytes) : nullptr;
  pp.status = status;
  pp.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)D));

  dim3 grid(pl.splits, Hkv, batch);
  cudaError_t e;
  const bool cluster = use_cluster(D, G, pl.splits, (long long)Hkv * batch);
  if (cluster)
    e = D == 128 ? launch_attn_cluster<128>(grid, stream, tk, tv, pp, rp)
                 : launch_attn_cluster<64>(grid, stream, tk, tv, pp, rp);
  else if (D == 128)
    e = G <= 8 ? launch_attn<128, 1>(grid, stream, tk, tv, pp, rp)
               : launch_attn<128, 2>(grid, stream, tk, tv, pp, rp);
  else
    e = G <= 8 ? launch_attn<64, 1>(grid, stream, tk, tv, pp, rp)
               : launch_attn<64, 2>(grid, stream, tk, tv, pp, rp);
  if (e != cudaSuccess) return cuda_fail(e, "decode attention launch");
  if (pl.splits > 1 && !cluster) {
    dim3 cgrid(geom->num_q_heads, batch);
    const cudaError_t ce =
        D == 128 ? launch_dependent(decode_combine_kernel<128>, cgrid, dim3(32), 0, stream, pp)
                 : launch_dependent(decode_combine_kernel<64>, cgrid, dim3(32), 0, stream, pp);
    if (ce != cudaSuccess) return cuda_fail(ce, "decode merge launch");
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "decode launch");
  return PIC_OK;
}

}  // namespace decode
}  // namespace pic

extern "C" pic_status_t pic_attend_decode(const pic_geom_t *geom, int32_t layer, int32_t batch,
                                          const void *q, const void *k_new, const void *v_new,
                                          const int32_t *pos, int32_t pos_offset,
                                          const int32_t *block_table,
                                          int32_t max_pages, int64_t num_pages, void *k_cache,
                                          void *v_cache, void *out, float *lse, int32_t max_ctx,
                                          int32_t num_splits, void *workspace,
                                          size_t workspace_bytes, pic_stream_t stream) {
  using namespace pic;
  using namespace pic::decode;
  static const char *who = "pic_attend_decode";
  RopeParams rp;
  pic_status_t st = check_step(who, geom, &rp, layer, batch, q, k_new, v_new, pos, block_table,
                               max_pages, num_pages, k_cache, v_cache, out, max_ctx, num_splits);
  if (st != PIC_OK) return st;
  const Plan pl = plan(geom, batch, max_ctx, num_splits);
  if (!workspace || workspace_bytes < pl.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return fail(PIC_ERR_WORKSPACE, "pic_attend_decode: workspace needs %zu bytes, 256-aligned",
                pl.total);
  return launch_step(who, geom, rp, layer, batch, q, k_new, v_new, pos, pos_offset, block_table,
                     max_pages, num_pages, k_cache, v_cache, out, lse, pl,
                     static_cast<uint8_t *>(workspace), stream);
}

// ---------------------------------------------------------------------------
// pic_attend_decode_noalloc: the same decoding step for callers that cannot
// allocate device memory on the step path.
//
// Some callers cannot call cudaMalloc (or any allocator) while they decode: an
// engine that has handed its whole memory budget to the KV cache, a runtime
// that forbids allocation after start-up, or an embedding that only owns the
// tensors it passes in.  For them this entry point takes no workspace: its
// scratch (the per-split partial softmax states) lives
// in the file-scope device array below, which every GPU that loads the library
// holds until the process exits.
//
// Set-up: the first call on each device (with that device current) looks up
// the array's device address with cudaGetSymbolAddress and caches it, per
// device context (a device reset replaces the context, and the address is
// looked up again); make that first call before any stream capture.  The array is shared by every
// call on the device and keeps the last call's contents: calls that overlap on
// the GPU (for example on two streams) race on it.  Nothing in it needs to
// start at zero: each call writes every scratch value before reading it.
namespace pic {
namespace decode {

constexpr size_t kNoAllocScratchBytes = 8u << 20;  // 8 MiB per device
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocScratchBytes];

static uint8_t *noalloc_scratch_ptr(pic_status_t *st) {
  constexpr int kMaxDev = 64;
  static uint8_t *ptrs[kMaxDev] = {nullptr};
  static unsigned long long ctx_ids[kMaxDev] = {0};
  static std::mutex mu;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    *st = e != cudaSuccess ? cuda_fail(e, "pic_attend_decode_noalloc: cudaGetDevice")
                           : fail(PIC_ERR_CUDA, "pic_attend_decode_noalloc: device %d", dev);
    return nullptr;
  }
  std::lock_guard<std::mutex> lk(mu);
  // Set-up once per device (per device context: after a device reset the
  // array has a new address in the new context, so it is looked up again).
  const unsigned long long id = current_context_id();
  if (!ptrs[dev] || id == 0 || id != ctx_ids[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) {
      *st = cuda_fail(e, "pic_attend_decode_noalloc: cudaGetSymbolAddress");
      return nullptr;
    }
    ptrs[dev] = static_cast<uint8_t *>(p);
    ctx_ids[dev] = current_context_id();
  }
  *st = PIC_OK;
  return ptrs[dev];
}

}  // namespace decode
}  // namespace pic

extern "C" pic_status_t pic_attend_decode_noalloc(const pic_geom_t *geom, int32_t layer,
                                                  int32_t batch, const void *q, const void *k_new,
                                                  const void *v_new, const int32_t *pos,
                                                  int32_t pos_offset, const int32_t *block_table,
                                                  int32_t max_pages, int64_t num_pages,
                                                  void *k_cache, void *v_cache, void *out,
                                                  float *lse, int32_t max_ctx, int32_t num_splits,
                                                  pic_stream_t stream) {
  using namespace pic;
  using namespace pic::decode;
  static const char *who = "pic_attend_decode_noalloc";
  RopeParams rp;
  pic_status_t st = check_step(who, geom, &rp, layer, batch, q, k_new, v_new, pos, block_table,
                               max_pages, num_pages, k_cache, v_cache, out, max_ctx, num_splits);
  if (st != PIC_OK) return st;
  // Scratch must fit the built-in array: the automatic split count is lowered
  // until it does; an explicit split count that does not fit is rejected.
  Plan pl = plan(geom, batch, max_ctx, num_splits);
  if (num_splits == 0)
    while (pl.total > kNoAllocScratchBytes && pl.splits > 1)
      pl = plan(geom, batch, max_ctx, pl.splits - 1);
  if (pl.total > kNoAllocScratchBytes)
    return fail(PIC_ERR_WORKSPACE,
                "pic_attend_decode_noalloc: needs %zu bytes of scratch, the built-in array holds "
                "%zu (fewer splits or a smaller batch may fit; pic_attend_decode takes a "
                "caller workspace instead)",
                pl.total, kNoAllocScratchBytes);
  uint8_t *ws = noalloc_scratch_ptr(&st);
  if (!ws) return st;
  return launch_step(who, geom, rp, layer, batch, q, k_new, v_new, pos, pos_offset, block_table,
                     max_pages, num_pages, k_cache, v_cache, out, lse, pl, ws, stream);
}
