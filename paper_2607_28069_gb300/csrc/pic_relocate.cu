// pic_relocate / pic_relocate_mapped: key re-rotation (Eq. 3) and stitching
// of cached documents into the paged request cache; values are copied
// unchanged (the paper rotates keys only; Background: Position-Independent
// Caching).
//
// pic_relocate takes the problem as the paper states it: per listed document
// its pool rows, base position and target position, and the request's block
// table (relocate_docs_kernel: a CTA per slice of a listed document).
// pic_relocate_mapped takes pic_compose's token and slot maps instead
// (relocate_kernel, described below); both rotate with the same operations,
// so for the same placement their caches are bit-identical.
//
// relocate_kernel: one launch, one CTA per (one or two pages of logical
// positions, request);
// the CTA moves its positions for every layer in turn, so its set-up (maps,
// cos/sin) is done once and it keeps a long stream of loads in flight.
// The CTA reads the token map and slot map of its positions (written by
// pic_compose) and evaluates cos/sin of delta_k * theta_i for the documents
// its page touches; then, per layer, it issues every K and V load of its page
// at once (16-byte streaming loads; V rows are bit copies, K rows come as the
// two 16-byte halves of 8 RoPE pairs), rotates and stores.  delta is
// constant over a document because base and target positions both advance by
// one per token, so R(b) R(a)^-1 = R(b - a) = R(delta).  The angle is formed and
// reduced in fp64, sin/cos evaluated in fp32 on the reduced angle; K is rotated
// in fp32 and rounded to bf16 (round to nearest even).  Pool rows and cache
// rows are d contiguous bf16 and consecutive threads take consecutive 16-byte
// pieces of the same row, so every warp access is fully coalesced.
// HBM-bound: 4 * Hkv * d * 2 bytes move per document token.
#include <algorithm>

#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kThreads = 256;
// Positions per CTA: one page (16) when a token carries >= 1024 K elements,
// two pages otherwise, so every CTA moves 64 KB and amortises its set-up.
constexpr int UV = 8;     // V tasks per thread per round
constexpr int UK = 4;     // K tasks per thread per round

struct RelocArgs {
  int max_docs, max_ctx, hkv, layer_begin, layer_end;
  long long pool_tokens, num_pages;
  const __nv_bfloat16 *k_pool, *v_pool;
  const int64_t *tok_map, *slots;
  const int32_t *delta;
  __nv_bfloat16 *k_cache, *v_cache;
  int32_t *status;
  // per-document form (pic_relocate): the documents' pool rows, base and
  // target positions, and the block table instead of the two maps
  int n_pool_docs, max_pages;
  const int64_t *doc_start;
  const int32_t *doc_len, *doc_base, *ids, *num_docs, *target, *block_table;
  const int32_t *prefix, *query;  // the link step's (kMapped)
  int share;  // occurrences of a document moved together, at most; 1: each by itself, no search
};

// Moves the positions a CTA of relocate_kernel set up (s_src / s_dst / s_doc,
// the documents' deltas in s_delta) for every layer of [layer_begin,
// layer_end).
template <int D, int kTok, bool kLayerRope>
__device__ __forceinline__ void move_positions(const RelocArgs &a, const RopeParams &rp, int b,
                                               const long long *s_src, const long long *s_dst,
                                               const int *s_doc, const int *s_delta,
                                               int k_first, int n_docs,
                                               float2 (*s_cs)[kTok][D / 2]);

// kLayerRope: a rotary table per layer (its cos/sin double-buffered: the next
// layer's table is computed while this layer's loads are in flight)
template <int D, int kTok, bool kLayerRope>
__global__ void __launch_bounds__(kThreads) relocate_kernel(RelocArgs a, RopeParams rp) {
  static_assert(kTok == 16 || kTok == 32, "one warp scans the positions of a CTA");
  pdl_entry();
  constexpr unsigned kMask = kTok == 32 ? 0xffffffffu : 0x0000ffffu;
  constexpr int HALF = D / 2;
  const int b = blockIdx.y;
  const long long t0 = (long long)blockIdx.x * kTok;
  const int tid = threadIdx.x;

  __shared__ long long s_src[kTok];  // pool row of position t0 + i, -1 = not a doc token
  __shared__ long long s_dst[kTok];  // cache slot
  __shared__ int s_doc[kTok];        // document index k within the request
  __shared__ int s_delta[kTok];      // delta of documents k_first .. k_first + n_docs - 1
  __shared__ int s_first, s_last;    // document range touched by this page
  __shared__ float2 s_cs[kLayerRope ? 2 : 1][kTok][HALF];

  if (tid < kTok) {
    const long long t = t0 + tid;
    long long src = -1, slot = -1;
    int k = 0;
    if (t < a.max_ctx) {
      const long long tm = a.tok_map[(size_t)b * a.max_ctx + t];
      slot = a.slots[(size_t)b * a.max_ctx + t];
      if (tm >= 0) {
        k = (int)(tm >> 40);
        src = tm & ((1LL << 40) - 1);
        if (src >= a.pool_tokens || k >= a.max_docs) {
          dev_fail(a.status, PIC_DEV_BAD_DOC_LEN, b);
          src = -1;
        } else if (slot < 0 || slot >= a.num_pages * 16) {
          dev_fail(a.status, PIC_DEV_BAD_PAGE, b);
          src = -1;
        }
      }
    }
    s_src[tid] = src;
    s_dst[tid] = slot;
    s_doc[tid] = k;
    // documents of a page are consecutive: first / last valid position's doc
    const unsigned valid = __ballot_sync(kMask, src >= 0);
    const int kf = __shfl_sync(kMask, k, valid ? __ffs(valid) - 1 : 0);
    const int kl = __shfl_sync(kMask, k, valid ? 31 - __clz(valid) : 0);
    if (tid == 0) {
      s_first = valid ? kf : -1;
      s_last = valid ? kl : -1;
    }
  }
  __syncthreads();
  if (s_first < 0) return;  // no document token on this page
  const int k_first = s_first;
  // every document between the first and last one here owns >= 1 position,
  // so at most kTok rows; anything else is a malformed token map
  const int n_docs = min(s_last - s_first + 1, kTok);
  if (tid < n_docs) s_delta[tid] = a.delta[(size_t)b * a.max_docs + k_first + tid];
  __syncthreads();
  move_positions<D, kTok, kLayerRope>(a, rp, b, s_src, s_dst, s_doc, s_delta, k_first, n_docs,
                                      s_cs);
}

// The per-document form, by pool document: a document that several listed
// occurrences share (requests of a batch that retrieved the same document, a
// boundary block repeated in one request) is read once and written to all of
// them.  CTA (k, b, slice) first finds the other occurrences of its document
// among the batch's document lists -- up to a.share of them, at most kMaxShare,
// form a group (share_limit) -- and then moves every r-th chunk of kTok tokens from its own rank on (r: the
// group's size; of those, every gridDim.z-th from its slice on) to all r
// places: token j of the document (pool row doc_start + j, compiled at base +
// j) goes to logical position target + j of each occurrence, rotated by its
// delta = target - base.  HBM-bound: 1 + r row transfers a token instead of 2r.
//
// The work of a CTA is a list of units (chunk, layer, block of kv heads) of at
// most 16 KB of K and 16 KB of V, contiguous in the pool: bulk copies bring
// them into a ring of two stages while the unit before is rotated and stored,
// so loads stay in flight whatever r is.  Three CTAs an SM (two with per-layer
// tables in chunks of 32 tokens at d = 128, for their shared memory).  Measured against
// a CTA that held 16 tokens in registers and knew one occurrence (four layers
// unless stated): 8 requests with 16 of 64 1024-token documents 720 -> 510 us
// (6.3 TB/s of the bytes that must move), 16 with 32 of 64 on 4 kv heads and
// two layers 740 -> 414, 4 with all 128 of a pool and one layer 869 -> 485;
// no document shared 275 -> 230 us (6.45 TB/s).  The same sharing with the
// chunk held in registers (two CTAs an SM) took 564, 473, 566 and 282 us.
//
// kMapped (the link step): targets are compose's doc_offset, and slots come
// from its slot map, -1 wherever its checks refused a position; it has
// reported the failures itself.
constexpr int kMaxShare = 8;      // occurrences of a document moved together
constexpr int kMaxScan = 2048;    // listed documents of a batch up to which a CTA looks for them
constexpr int kUnit = 8192;       // elements of K (and of V) in a unit
constexpr int kStageBytes = 2 * kUnit * 2;
constexpr int kRing = 2;
constexpr int kRelocSmem = kRing * kStageBytes + 128;

template <int D, int kTok, bool kLayerRope, bool kMapped>
__global__ void __launch_bounds__(kThreads, 3) relocate_docs_kernel(RelocArgs a, RopeParams rp) {
  pdl_entry();
  constexpr int HALF = D / 2, KC = D / 16, VC = D / 8;
  const int k = blockIdx.x, b = blockIdx.y, slice = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, style = rp.style;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t ring = (smem_u32(smem_raw) + 127u) & ~127u;
  __shared__ uint32_t s_mask[kMaxScan / 32];  // listed documents equal to this one
  __shared__ int s_tb[kMaxShare], s_tt[kMaxShare];  // request and target position of each
  __shared__ long long s_row[2][kMaxShare][kTok];   // cache row of head 0 of each token, -1: none
  __shared__ float2 s_cs[kLayerRope ? 2 : 1][kMaxShare][HALF];
  __shared__ __align__(8) uint64_t s_bar[kRing];
  __shared__ int s_abort;
  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) mbar_init(smem_u32(&s_bar[i]), 1);
    s_abort = 0;
    fence_mbar_init();
  }

  // ---- this occurrence, and the first 256 listed documents beside it: all
  // loads independent of one another
  const int listed = (int)gridDim.y * a.max_docs, own = b * a.max_docs + k;
  const bool scan = a.share > 1 && listed <= kMaxScan;
  auto target_ok = [&](long long t, int len) {
    return t >= 0 && (kMapped || t + len <= (long long)a.max_pages * 16);
  };
  struct Entry {
    int id, target;  // id -1: not listed
  };
  auto entry = [&](int e) -> Entry {
    Entry r{-1, -1};
    if (e < listed) {
      const int b2 = e / a.max_docs, m2 = a.num_docs[b2];
      const int id2 = a.ids[e], t2 = a.target[e];
      const bool bad = kMapped && (a.prefix[b2] < 0 || a.query[b2] < 0);
      if (m2 <= a.max_docs && e % a.max_docs < m2 && !bad) r = Entry{id2, t2};
    }
    return r;
  };
  Entry e0{-1, -1};
  if (scan) e0 = entry(tid);
  const bool report = !kMapped && tid == 0 && slice == 0;
  const int m = a.num_docs[b];
  if (m < 0 || m > a.max_docs) {
    if (report && k == 0) dev_fail(a.status, PIC_DEV_BAD_REQUEST, b);
    return;
  }
  if (k >= m) return;
  if (kMapped && (a.prefix[b] < 0 || a.query[b] < 0)) return;
  const int id = a.ids[own];
  const long long target = a.target[own];
  if (id < 0 || id >= a.n_pool_docs) {
    if (report) dev_fail(a.status, PIC_DEV_BAD_DOC_ID, b);
    return;
  }
  const int n = a.doc_len[id], base = a.doc_base[id];
  const long long start = a.doc_start[id];
  if (n <= 0 || (!kMapped && (start < 0 || start + n > a.pool_tokens))) {
    if (report) dev_fail(a.status, PIC_DEV_BAD_DOC_LEN, b);
    return;
  }
  if (!target_ok(target, n)) {
    if (report) dev_fail(a.status, target < 0 ? PIC_DEV_BAD_POSITION : PIC_DEV_BLOCK_TABLE_SHORT, b);
    return;
  }
  if (!kMapped && slice == 0 && tid < 32) {  // targets of two listed documents must not overlap
    bool clash = false;
    for (int k2 = tid; k2 < m; k2 += 32) {
      if (k2 == k) continue;
      const int id2 = a.ids[(size_t)b * a.max_docs + k2];
      if (id2 < 0 || id2 >= a.n_pool_docs) continue;
      const long long t2 = a.target[(size_t)b * a.max_docs + k2];
      const long long n2 = a.doc_len[id2];
      clash |= t2 < target + n && target < t2 + n2;
    }
    if (__any_sync(0xffffffffu, clash) && tid == 0) dev_fail(a.status, PIC_DEV_BAD_POSITION, b);
  }

  // ---- the group: the valid occurrences of the document, in list order
  int cnt = 1, rank = 0;
  if (scan) {
    if (slice >= (n + kTok - 1) / kTok) return;  // no chunk for this slice, whatever the group
    const int words = (listed + 31) / 32;
    for (int e = tid; e < words * 32; e += kThreads) {
      const Entry x = e == tid ? e0 : entry(e);
      const uint32_t w = __ballot_sync(0xffffffffu, x.id == id && target_ok(x.target, n));
      if (lane == 0) s_mask[e / 32] = w;
    }
    __syncthreads();
    // every warp: lane l the words 2l and 2l + 1, occurrences before each
    const uint32_t w0 = 2 * lane < words ? s_mask[2 * lane] : 0u;
    const uint32_t w1 = 2 * lane + 1 < words ? s_mask[2 * lane + 1] : 0u;
    int before = __popc(w0) + __popc(w1);
    const int all = before;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += v;
    }
    const int total = __shfl_sync(0xffffffffu, before, 31);
    before -= all;
    auto rank_of = [&](int e) {  // occurrences before list entry e (e / 32 uniform in the warp)
      const int w = e / 32;
      const int base_w = __shfl_sync(0xffffffffu, before + (w & 1 ? __popc(w0) : 0), w / 2);
      return base_w + __popc(s_mask[w] & ((1u << (e & 31)) - 1u));
    };
    rank = rank_of(own);
    const int first = rank / a.share * a.share;  // the group's first rank
    for (int e = tid; e < words * 32; e += kThreads) {
      const int r = rank_of(e) - first;
      if ((s_mask[e / 32] >> lane & 1u) && r >= 0 && r < a.share) {
        s_tb[r] = e / a.max_docs;
        s_tt[r] = e == tid ? e0.target : a.target[e];
      }
    }
    cnt = min(total - first, a.share);
    rank -= first;
  } else if (tid == 0) {
    s_tb[0] = b;
    s_tt[0] = (int)target;
  }
  __syncthreads();

  // ---- the units of this CTA: chunk ci of its share, layer, block of heads
  // tokens j_lo .. j_lo + n_tok - 1 have pool rows (kMapped: maybe not all do)
  const long long lo = max(0ll, -start), hi = min((long long)n, a.pool_tokens - start);
  if (lo >= hi) return;
  const int j_lo = (int)lo, n_tok = (int)(hi - lo);
  const int chunks = (n_tok + kTok - 1) / kTok;
  const int c_first = rank + cnt * slice, c_step = cnt * (int)gridDim.z;
  if (c_first >= chunks) return;
  const int my_chunks = (chunks - c_first + c_step - 1) / c_step;
  const int hkv = a.hkv, hb = min(hkv, kUnit / (kTok * D)), hblocks = (hkv + hb - 1) / hb;
  const int layers = a.layer_end - a.layer_begin, per_chunk = layers * hblocks;
  const long long units = (long long)my_chunks * per_chunk;
  auto issue = [&](long long u) {  // thread 0: the bulk copies of unit u
    const int ci = (int)(u / per_chunk), rem = (int)(u % per_chunk);
    const int layer = a.layer_begin + rem / hblocks, h0 = rem % hblocks * hb, nh = min(hb, hkv - h0);
    const int t0 = (c_first + ci * c_step) * kTok, nt = min(kTok, n_tok - t0);
    const size_t src = (((size_t)layer * a.pool_tokens + (start + j_lo + t0)) * hkv + h0) * D;
    const uint32_t st = ring + (uint32_t)(u % kRing) * kStageBytes, bar = smem_u32(&s_bar[u % kRing]);
    const uint32_t row = (uint32_t)nh * D * 2;
    mbar_expect_tx(bar, 2 * nt * row);
    if (nh == hkv) {  // whole rows: one contiguous piece
      bulk_load(st, a.k_pool + src, nt * row, bar);
      bulk_load(st + kUnit * 2, a.v_pool + src, nt * row, bar);
    } else {
      for (int i = 0; i < nt; ++i) {
        bulk_load(st + i * row, a.k_pool + src + (size_t)i * hkv * D, row, bar);
        bulk_load(st + kUnit * 2 + i * row, a.v_pool + src + (size_t)i * hkv * D, row, bar);
      }
    }
  };
  if (tid == 0)
    for (int u = 0; u < min((long long)kRing, units); ++u) issue(u);
  auto fill_rows = [&](int ci) {  // cache rows of chunk ci's tokens
    const int t0 = (c_first + ci * c_step) * kTok;
    for (int e = tid; e < cnt * kTok; e += kThreads) {
      const int q = e / kTok, i = e % kTok;
      long long slot = -1;
      if (t0 + i < n_tok) {
        const int b2 = s_tb[q];
        const long long t = (long long)s_tt[q] + j_lo + t0 + i;
        if (kMapped) {
          if (t < a.max_ctx) slot = a.slots[(size_t)b2 * a.max_ctx + t];
          if (slot >= a.num_pages * 16) slot = -1;
        } else {
          const int page = a.block_table[(size_t)b2 * a.max_pages + (t >> 4)];
          if (page < 0 || page >= a.num_pages) dev_fail(a.status, PIC_DEV_BAD_PAGE, b2);
          else slot = (long long)page * 16 + (t & 15);
        }
      }
      s_row[ci & 1][q][i] = slot < 0 ? -1 : (slot >> 4) * hkv * 16 + (slot & 15);
    }
  };
  auto fill_cs = [&](int layer, int buf) {
    for (int e = tid; e < cnt * HALF; e += kThreads) {
      const int q = e / HALF, i = e % HALF, delta = s_tt[q] - base;
      s_cs[buf][q][i] = kLayerRope ? rope_cos_sin_fast(delta, rope_theta(rp, layer, i))
                                   : rope_cos_sin(delta, rope_theta(rp, layer, i));
    }
  };
  fill_rows(0);
  fill_cs(a.layer_begin, 0);
  __syncthreads();

  const int kc = tid % KC;  // this thread's chunk of 8 pairs, the same in every row
  const PairChunk pc = pair_chunk(kc, HALF, style);
  int cur = 0;  // table buffer of the unit's layer (kLayerRope)
  long long u = 0;
  bool ok = true;
  for (int ci = 0; ok && ci < my_chunks; ++ci) {
    const int nt = min(kTok, n_tok - (c_first + ci * c_step) * kTok);
    for (int rem = 0; rem < per_chunk; ++rem, ++u) {
      const int layer = a.layer_begin + rem / hblocks, h0 = rem % hblocks * hb, nh = min(hb, hkv - h0);
      const uint32_t st = ring + (uint32_t)(u % kRing) * kStageBytes, bar = smem_u32(&s_bar[u % kRing]);
      // the next chunk's rows and the next layer's table while the copy is in flight
      if (rem == 0 && ci + 1 < my_chunks) fill_rows(ci + 1);
      bool next_table = false;
      if constexpr (kLayerRope) {
        next_table = layers > 1 && (rem + 1) % hblocks == 0;
        if (next_table) fill_cs(layer + 1 < a.layer_end ? layer + 1 : a.layer_begin, cur ^ 1);
      }
      ok = mbar_wait(bar, (u / kRing) & 1, &s_abort, a.status, b);
      ok = __syncthreads_and(ok);
      if (!ok) break;
      __nv_bfloat16 *kd = a.k_cache + ((size_t)layer * a.num_pages * hkv + h0) * 16 * D;
      __nv_bfloat16 *vd = a.v_cache + ((size_t)layer * a.num_pages * hkv + h0) * 16 * D;
      const int nv = nt * nh * VC, nk = nt * nh * KC;
#pragma unroll 1
      for (int q = 0; q < cnt; ++q) {
        const long long *rows = s_row[ci & 1][q];
        for (int t = tid; t < nv; t += kThreads) {  // values: bit copies
          const int hr = t / VC, i = hr / nh, h = hr - i * nh;
          const long long row = rows[i];
          const uint4 v = lds128(st + kUnit * 2 + t * 16);
          if (row >= 0) st_global16(vd + (row + h * 16) * D + (t % VC) * 8, v);
        }
        float2 cs[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) cs[i] = s_cs[cur][q][8 * kc + i];
        for (int t = tid; t < nk; t += kThreads) {  // keys: rotated by the occurrence's delta
          const int hr = t / KC, i = hr / nh, h = hr - i * nh;
          const long long row = rows[i];
          const uint4 x = lds128(st + (hr * D + pc.off_a) * 2), y = lds128(st + (hr * D + pc.off_b) * 2);
          if (row >= 0) rotate_store(x, y, kd + (row + h * 16) * D, pc, style, cs);
        }
      }
      fence_proxy_async();  // this thread's reads of the stage precede the next copy into it
      __syncthreads();
      if (tid == 0 && u + kRing < units) issue(u + kRing);
      if (next_table) cur ^= 1;
    }
  }
  if (!ok && tid == 0)  // aborted: let the copies already issued land before the CTA exits
    for (long long w = u; w < min(units, u + kRing); ++w)
      mbar_wait_no_flag(smem_u32(&s_bar[w % kRing]), (w / kRing) & 1, a.status, b, kWaitLimitNs);
}

template <int D, int kTok, bool kLayerRope>
__device__ __forceinline__ void move_positions(const RelocArgs &a, const RopeParams &rp, int b,
                                               const long long *s_src, const long long *s_dst,
                                               const int *s_doc, const int *s_delta,
                                               int k_first, int n_docs,
                                               float2 (*s_cs)[kTok][D / 2]) {
  constexpr int HALF = D / 2;
  constexpr int KC = D / 16;  // 8-pair chunks per K row
  constexpr int VC = D / 8;   // 16-byte pieces per V row
  const int style = rp.style;
  const int tid = threadIdx.x;
  const size_t hkv = a.hkv;
  auto fill_cs = [&](int layer, int buf) {  // cos/sin of the touched documents
    for (int e = tid; e < n_docs * HALF; e += kThreads) {
      const int j = e / HALF, i = e % HALF;
      const int delta = s_delta[j];
      s_cs[buf][j][i] = kLayerRope ? rope_cos_sin_fast(delta, rope_theta(rp, layer, i))
                                   : rope_cos_sin(delta, rope_theta(rp, layer, i));
    }
  };
  fill_cs(a.layer_begin, 0);
  __syncthreads();
  for (int layer = a.layer_begin; layer < a.layer_end; ++layer) {
  const int cur = kLayerRope ? (layer - a.layer_begin) & 1 : 0;
  const __nv_bfloat16 *kp = a.k_pool + (size_t)layer * a.pool_tokens * hkv * D;
  const __nv_bfloat16 *vp = a.v_pool + (size_t)layer * a.pool_tokens * hkv * D;
  __nv_bfloat16 *kc = a.k_cache + (size_t)layer * a.num_pages * hkv * 16 * D;
  __nv_bfloat16 *vc = a.v_cache + (size_t)layer * a.num_pages * hkv * 16 * D;
  const int nV = kTok * (int)hkv * VC, nK = kTok * (int)hkv * KC;

  for (int round = 0; round * kThreads * UV < nV || round * kThreads * UK < nK; ++round) {
    // ---- issue this round's loads
    uint4 v[UV], ka[UK], kb[UK];
    long long vdst[UV], kdst[UK];
    int kdoc[UK], kch[UK];
#pragma unroll
    for (int u = 0; u < UV; ++u) {
      const int task = (round * UV + u) * kThreads + tid;
      vdst[u] = -1;
      if (task < nV) {
        const int i = task / ((int)hkv * VC), r = task % ((int)hkv * VC);
        const int h = r / VC, c = r % VC;
        const long long src = s_src[i];
        if (src >= 0) {
          const long long slot = s_dst[i];
          v[u] = ld_stream(vp + ((size_t)src * hkv + h) * D + c * 8);
          vdst[u] = (((slot >> 4) * (long long)hkv + h) * 16 + (slot & 15)) * D + c * 8;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < UK; ++u) {
      const int task = (round * UK + u) * kThreads + tid;
      kdst[u] = -1;
      if (task < nK) {
        const int i = task / ((int)hkv * KC), r = task % ((int)hkv * KC);
        const int h = r / KC, c = r % KC;
        const long long src = s_src[i];
        if (src >= 0) {
          const long long slot = s_dst[i];
          const PairChunk pc = pair_chunk(c, HALF, style);
          const __nv_bfloat16 *sp = kp + ((size_t)src * hkv + h) * D;
          ka[u] = ld_stream(sp + pc.off_a);
          kb[u] = ld_stream(sp + pc.off_b);
          kdst[u] = (((slot >> 4) * (long long)hkv + h) * 16 + (slot & 15)) * D;
          kdoc[u] = s_doc[i] - k_first;
          kch[u] = c;
          if (kdoc[u] >= n_docs) kdst[u] = -1;
        }
      }
    }
    if constexpr (kLayerRope) {  // next layer's table while the loads are in flight
      if (round == 0 && layer + 1 < a.layer_end) fill_cs(layer + 1, cur ^ 1);
    }
    // ---- V: bit copy
#pragma unroll
    for (int u = 0; u < UV; ++u)
      if (vdst[u] >= 0) st_global16(vc + vdst[u], v[u]);
    // ---- K: rotate 8 pairs and store
#pragma unroll
    for (int u = 0; u < UK; ++u) {
      if (kdst[u] < 0) continue;
      const int c = kch[u];
      float2 cs[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) cs[q] = s_cs[cur][kdoc[u]][8 * c + q];
      float x[8], y[8], uu[8], ww[8];
      unpack8(ka[u], x);
      unpack8(kb[u], y);
      if (style == PIC_ROPE_HALF) {
#pragma unroll
        for (int q = 0; q < 8; ++q) { uu[q] = x[q]; ww[q] = y[q]; }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uu[q] = x[2 * q]; ww[q] = x[2 * q + 1];
          uu[4 + q] = y[2 * q]; ww[4 + q] = y[2 * q + 1];
        }
      }
      rotate8(uu, ww, cs);
      if (style == PIC_ROPE_HALF) {
#pragma unroll
        for (int q = 0; q < 8; ++q) { x[q] = uu[q]; y[q] = ww[q]; }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          x[2 * q] = uu[q]; x[2 * q + 1] = ww[q];
          y[2 * q] = uu[4 + q]; y[2 * q + 1] = ww[4 + q];
        }
      }
      const PairChunk pc = pair_chunk(c, HALF, style);
      st_global16(kc + kdst[u] + pc.off_a, pack8(x));
      st_global16(kc + kdst[u] + pc.off_b, pack8(y));
    }
  }
  if constexpr (kLayerRope) __syncthreads();  // next table written; this one read
  }
}

// Tokens of a chunk, by the elements of a token's K row (units of at most 16 KB).
constexpr int chunk_tokens(int row) { return row >= 1024 ? 8 : row >= 512 ? 16 : 32; }

// Occurrences of a document that are moved together, at most (1: no search), for
// a relocation of `tokens` listed document tokens (host estimate: the pool's mean
// length) that moves `bytes`.  The search costs a CTA about a microsecond before
// its first copy, which pays from kShareBytes on (2 requests of 8 documents of
// 512 tokens, 67 MB: 24 us with it, 19 without).  And a chunk that r occurrences
// share is one CTA's work instead of r CTAs', so groups stay small enough that
// two waves of chunks are left if every document has r occurrences: with groups
// of up to 8 in any case, 16 requests listing the same two documents of 64 tokens,
// 16 layers, took 4.4 times as long as without sharing, and 84 of 153 shapes with
// shared documents from 128 MB on got slower by it (1.21 times as long on average);
// with this limit five, by up to 16% (640 listed documents of 100 tokens), and 0.94
// on average (8 requests with 16 documents of 1024 tokens, one layer 147 -> 108 us).
constexpr double kShareBytes = 128e6;
constexpr int kWave = 3 * 152;  // CTAs resident at once
inline int share_limit(double tokens, int row, double bytes) {
  if (bytes < kShareBytes) return 1;
  return (int)std::max(1.0, std::min<double>(kMaxShare, tokens / chunk_tokens(row) / (2 * kWave)));
}

// Launch of the per-document form.  Slices per listed document: each CTA
// walks every slices-th chunk of its share of the document; few documents get
// more slices (up to one chunk per CTA), so that a small request still fills
// the GPU, but no more than a document of twice the pool's mean length has
// chunks.  The slices come last in the launch order: CTAs past a document's
// last chunk exit, and among working ones they left the SMs unevenly filled (one
// request of 8 documents of 512 tokens, 16/2 heads of 64, 16 layers: 47% of the SM
// cycles active, 37 us; in this order 30; 720 relocations 0.70 of the time before
// the bulk copies on average, 0.78 with the slices first).
template <int D, int kTok, bool kMapped>
cudaError_t launch_docs_as(const RelocArgs &a, const RopeParams &rp, const dim3 &grid,
                           cudaStream_t stream) {
  auto *kernel = rp.layer_theta ? relocate_docs_kernel<D, kTok, true, kMapped>
                                : relocate_docs_kernel<D, kTok, false, kMapped>;
  const cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRelocSmem);
  if (e != cudaSuccess) return e;
  return launch_dependent(kernel, grid, dim3(kThreads), kRelocSmem, stream, a, rp);
}
template <bool kMapped>
cudaError_t launch_docs(const pic_geom_t *geom, const RelocArgs &a, const RopeParams &rp, int batch,
                        cudaStream_t stream) {
  const int row = geom->num_kv_heads * geom->head_dim;
  const long long docs_total = (long long)batch * a.max_docs;
  const int tok = chunk_tokens(row);
  const double mean_chunks = (double)a.pool_tokens / std::max(a.n_pool_docs, 1) / tok;
  const long long most = std::max(1ll, (long long)std::ceil(2.0 * std::min(mean_chunks, 1e6)));
  const long long want = std::max<long long>(16, (8 * 152 + docs_total - 1) / docs_total);
  const int slices = (int)std::min({128ll, want, most});
  const dim3 grid(a.max_docs, batch, slices);
  if (geom->head_dim == 128)
    return tok == 8    ? launch_docs_as<128, 8, kMapped>(a, rp, grid, stream)
           : tok == 16 ? launch_docs_as<128, 16, kMapped>(a, rp, grid, stream)
                       : launch_docs_as<128, 32, kMapped>(a, rp, grid, stream);
  return tok == 8    ? launch_docs_as<64, 8, kMapped>(a, rp, grid, stream)
         : tok == 16 ? launch_docs_as<64, 16, kMapped>(a, rp, grid, stream)
                     : launch_docs_as<64, 32, kMapped>(a, rp, grid, stream);
}

}  // namespace

cudaError_t launch_link_relocation(const pic_geom_t *geom, const RopeParams &rp, int batch,
                                   int max_docs, int n_pool_docs, const void *k_pool,
                                   const void *v_pool, int64_t pool_tokens,
                                   const int64_t *doc_token_start, const int32_t *doc_len,
                                   const int32_t *doc_base_pos, const int32_t *req_doc_ids,
                                   const int32_t *req_num_docs, const int32_t *prefix_len,
                                   const int32_t *query_len, const int32_t *doc_offset,
                                   const int64_t *slot_mapping, int max_ctx, int64_t num_pages,
                                   void *k_cache, void *v_cache, int layer_begin, int layer_end,
                                   int32_t *status, cudaStream_t stream) {
  RelocArgs a = {};
  a.max_docs = max_docs;
  a.max_ctx = max_ctx;
  a.hkv = geom->num_kv_heads;
  a.layer_begin = layer_begin;
  a.layer_end = layer_end;
  a.pool_tokens = pool_tokens;
  a.num_pages = num_pages;
  a.k_pool = static_cast<const __nv_bfloat16 *>(k_pool);
  a.v_pool = static_cast<const __nv_bfloat16 *>(v_pool);
  a.slots = slot_mapping;
  a.k_cache = static_cast<__nv_bfloat16 *>(k_cache);
  a.v_cache = static_cast<__nv_bfloat16 *>(v_cache);
  a.status = status;
  a.n_pool_docs = n_pool_docs;
  a.doc_start = doc_token_start;
  a.doc_len = doc_len;
  a.doc_base = doc_base_pos;
  a.ids = req_doc_ids;
  a.num_docs = req_num_docs;
  a.target = doc_offset;
  a.prefix = prefix_len;
  a.query = query_len;
  const double tokens = listed_tokens(batch, max_docs, n_pool_docs, pool_tokens, max_ctx);
  const int row = geom->num_kv_heads * geom->head_dim;
  a.share = share_limit(tokens, row, 8.0 * tokens * row * (layer_end - layer_begin));
  return launch_docs<true>(geom, a, rp, batch, stream);
}

// One launch derives the layout in every CTA, empty ones included, and reads a
// shared document once per occurrence; three launches cost about 10 us of
// launches and dependencies.  Measured over 1140 shapes of 1 to 16 requests (1,
// 4, 16 layers; capacity max_ctx one and four times the context): from 600 MB in
// two waves of chunks, or from 2200 CTAs on, the three launches are faster (8 requests with 16 of 64 documents
// of 1024 tokens, four layers 740 -> 533 us; 4 with 16 of 1024 tokens, one layer
// 131 -> 89; one of 8 documents of 512 tokens, capacity 131k, one layer 60 -> 22),
// but for three shapes, by 7 to 16%.  Below, one launch is (one request of 8
// documents of 512 tokens, one layer, capacity 16k: 14.4 us against 21.6).  A line
// at 128 MB of capacity made 105 of them up to 52% slower than one launch.
bool link_relocation_apart(double tokens, int row, int layers, long long ctas) {
  return (8.0 * tokens * row * layers >= 600e6 && tokens / chunk_tokens(row) >= 2 * kWave) || ctas >= 2200;
}

double listed_tokens(int batch, int max_docs, int n_pool_docs, int64_t pool_tokens, double max_ctx) {
  return batch * std::min((double)max_docs * pool_tokens / std::max(n_pool_docs, 1), max_ctx);
}
}  // namespace pic

extern "C" pic_status_t pic_relocate_mapped(const pic_geom_t *geom, int32_t batch,
                                            int32_t max_docs, const void *k_pool,
                                            const void *v_pool, int64_t pool_tokens,
                                            const int64_t *tok_map, const int32_t *doc_delta,
                                            const int64_t *slot_mapping, int32_t max_ctx,
                                            int64_t num_pages, void *k_cache, void *v_cache,
                                            int32_t layer_begin, int32_t layer_end,
                                            pic_stream_t stream) {
  using namespace pic;
  RopeParams rp;
  pic_status_t st = make_rope(geom, &rp);
  if (st != PIC_OK) return st;
  if (max_docs == 0 && batch > 0) return PIC_OK;  // no document to move
  if (batch <= 0 || max_docs < 0 || pool_tokens <= 0 || max_ctx <= 0 || num_pages <= 0)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate_mapped: sizes must be positive");
  if (pool_tokens >= (1LL << 40))
    return fail(PIC_ERR_UNSUPPORTED, "pic_relocate_mapped: pool has 2^40 rows or more");
  if (layer_begin < 0 || layer_end > geom->num_layers || layer_begin >= layer_end)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate_mapped: layer range [%d, %d) outside [0, %d)",
                layer_begin, layer_end, geom->num_layers);
  if (layer_end - layer_begin > 65535 || batch > 65535)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate_mapped: grid too large");
  if (!k_pool || !v_pool || !tok_map || !doc_delta || !slot_mapping || !k_cache || !v_cache)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate_mapped: NULL tensor");
  if ((reinterpret_cast<uintptr_t>(k_pool) | reinterpret_cast<uintptr_t>(v_pool) |
       reinterpret_cast<uintptr_t>(k_cache) | reinterpret_cast<uintptr_t>(v_cache)) & 15)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate_mapped: K/V tensors must be 16-byte aligned");
  int32_t *status = device_status_ptr();
  if (!status) return fail(PIC_ERR_CUDA, "pic_relocate_mapped: no device status word");

  RelocArgs a;
  a.max_docs = max_docs;
  a.max_ctx = max_ctx;
  a.hkv = geom->num_kv_heads;
  a.layer_begin = layer_begin;
  a.layer_end = layer_end;
  a.pool_tokens = pool_tokens;
  a.num_pages = num_pages;
  a.k_pool = static_cast<const __nv_bfloat16 *>(k_pool);
  a.v_pool = static_cast<const __nv_bfloat16 *>(v_pool);
  a.tok_map = tok_map;
  a.slots = slot_mapping;
  a.delta = doc_delta;
  a.k_cache = static_cast<__nv_bfloat16 *>(k_cache);
  a.v_cache = static_cast<__nv_bfloat16 *>(v_cache);
  a.status = status;
  const bool wide = geom->num_kv_heads * geom->head_dim >= 1024;
  const int tok = wide ? 16 : 32;
  dim3 grid((max_ctx + tok - 1) / tok, batch);
  const dim3 block(kThreads);
  cudaError_t e;
  if (geom->head_dim == 128)
    e = rp.layer_theta
            ? (wide ? launch_dependent(relocate_kernel<128, 16, true>, grid, block, 0, stream, a, rp)
                    : launch_dependent(relocate_kernel<128, 32, true>, grid, block, 0, stream, a, rp))
            : (wide ? launch_dependent(relocate_kernel<128, 16, false>, grid, block, 0, stream, a, rp)
                    : launch_dependent(relocate_kernel<128, 32, false>, grid, block, 0, stream, a, rp));
  else
    e = rp.layer_theta
            ? (wide ? launch_dependent(relocate_kernel<64, 16, true>, grid, block, 0, stream, a, rp)
                    : launch_dependent(relocate_kernel<64, 32, true>, grid, block, 0, stream, a, rp))
            : (wide ? launch_dependent(relocate_kernel<64, 16, false>, grid, block, 0, stream, a, rp)
                    : launch_dependent(relocate_kernel<64, 32, false>, grid, block, 0, stream, a, rp));
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "pic_relocate_mapped launch");
  return PIC_OK;
}

extern "C" pic_status_t pic_relocate(const pic_geom_t *geom, int32_t batch, int32_t max_docs,
                                     int32_t n_pool_docs, const void *k_pool, const void *v_pool,
                                     int64_t pool_tokens, const int64_t *doc_token_start,
                                     const int32_t *doc_len, const int32_t *doc_base_pos,
                                     const int32_t *req_doc_ids, const int32_t *req_num_docs,
                                     const int32_t *doc_target, const int32_t *block_table,
                                     int32_t max_pages, int64_t num_pages, void *k_cache,
                                     void *v_cache, int32_t layer_begin, int32_t layer_end,
                                     pic_stream_t stream) {
  using namespace pic;
  RopeParams rp;
  pic_status_t st = make_rope(geom, &rp);
  if (st != PIC_OK) return st;
  if (max_docs == 0 && batch > 0) return PIC_OK;  // no document to move
  if (batch <= 0 || max_docs < 0 || n_pool_docs <= 0 || pool_tokens <= 0 || max_pages <= 0 ||
      num_pages <= 0)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate: sizes must be positive");
  if (layer_begin < 0 || layer_end > geom->num_layers || layer_begin >= layer_end)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate: layer range [%d, %d) outside [0, %d)",
                layer_begin, layer_end, geom->num_layers);
  if (max_docs > 65535 || batch > 65535)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate: grid too large");
  if ((long long)max_pages * 16 >= (1LL << 31))
    return fail(PIC_ERR_UNSUPPORTED, "pic_relocate: block table longer than 2^27 pages");
  if (!k_pool || !v_pool || !doc_token_start || !doc_len || !doc_base_pos || !req_doc_ids ||
      !req_num_docs || !doc_target || !block_table || !k_cache || !v_cache)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate: NULL tensor");
  if ((reinterpret_cast<uintptr_t>(k_pool) | reinterpret_cast<uintptr_t>(v_pool) |
       reinterpret_cast<uintptr_t>(k_cache) | reinterpret_cast<uintptr_t>(v_cache)) & 15)
    return fail(PIC_ERR_INVALID_ARG, "pic_relocate: K/V tensors must be 16-byte aligned");
  int32_t *status = device_status_ptr();
  if (!status) return fail(PIC_ERR_CUDA, "pic_relocate: no device status word");

  RelocArgs a = {};
  a.max_docs = max_docs;
  a.hkv = geom->num_kv_heads;
  a.layer_begin = layer_begin;
  a.layer_end = layer_end;
  a.pool_tokens = pool_tokens;
  a.num_pages = num_pages;
  a.k_pool = static_cast<const __nv_bfloat16 *>(k_pool);
  a.v_pool = static_cast<const __nv_bfloat16 *>(v_pool);
  a.k_cache = static_cast<__nv_bfloat16 *>(k_cache);
  a.v_cache = static_cast<__nv_bfloat16 *>(v_cache);
  a.status = status;
  a.n_pool_docs = n_pool_docs;
  a.max_pages = max_pages;
  a.doc_start = doc_token_start;
  a.doc_len = doc_len;
  a.doc_base = doc_base_pos;
  a.ids = req_doc_ids;
  a.num_docs = req_num_docs;
  a.target = doc_target;
  a.block_table = block_table;
  const double tokens = listed_tokens(batch, max_docs, n_pool_docs, pool_tokens, 16.0 * max_pages);
  const int row = geom->num_kv_heads * geom->head_dim;
  a.share = share_limit(tokens, row, 8.0 * tokens * row * (layer_end - layer_begin));
  cudaError_t e = launch_docs<false>(geom, a, rp, batch, stream);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "pic_relocate launch");
  return PIC_OK;
}
