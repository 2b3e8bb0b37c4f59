// k_attn.cu -- grouped-query attention of a verification block over the
// retained prefix (Section 3.2: one causal pass over the root and the
// candidates; App. C.4: rows attend to the committed prefix and to the
// block's own earlier rows).
//
// Row i of request b sits at position L_b + i and attends to keys [0, L_b + i].
// All G = n_q / n_kv query heads of a key/value head, for all rows of the
// request, form one query matrix of M * G rows, so each key/value entry is
// read from HBM once per block (twice when a request has more than 64 query
// rows, the second time from L2).
//
// qkv_finish_kernel: the QKV projection arrives as split-K partial sums
// (TC_PART); half a warp per (token row, head) adds them in rank order, scales by
// the row's 1 / rms and rotates (RoPE).  Keys and values are appended to the
// cache; queries, scaled by log2(e) / sqrt(d), are written as bf16 hi and lo
// parts straight into the tensor-core operand image of their (request, kv
// head, 64-query tile): 128 rows (hi_row: of every 16 rows 8 hi parts, then the
// lo parts of the same queries) of d elements in the 128-byte-swizzled K-major
// layout, one 16 KB region per 64 columns.
//
// attn_tc_kernel: one CTA per 128-key tile of one (request, kv head, query
// tile); a cluster of 8 CTAs covers one chunk of 1024 keys.  Per CTA:
//   * the tile's keys and values arrive by TMA (3D map over the cache, 128-
//     byte swizzle; tiles holding only entries older than this call are
//     requested before the wait for the finishing kernel), the query image
//     by one bulk copy;
//   * S = Q K^T on tcgen05 (M = 128: the hi and lo rows of 64 queries, N = 128
//     keys) into TMEM; 16-lane loads (tcgen05.ld.16x256b) bring both parts of
//     the same scores to one thread, which adds them (TileThread); masking
//     (causal, and keys past the call's end) and P = 2^(S - m) with the tile's
//     own maximum m and sum l;
//   * O = P V on tcgen05 (P's hi and lo rows stored the same way, as the A
//     operand in TMEM over S, or in the narrow layout as a shared-memory
//     image over Q; B = V read MN-major from the TMA image), hi + lo added in
//     the thread that loads them;
//   * the tile partials (m, l, O) are pushed through distributed shared
//     memory to the CTA that folds their query rows (CTA r: rows 8r..8r+7),
//     which folds the chunk's 8 tiles in tile order.  With one chunk the
//     result is normalised and written (bf16 hi, lo).  With two chunks in a
//     cluster of 16 (PAIR), CTA r receives rows 4r..4r+3 from all 16 tiles
//     and folds each chunk's tiles, then the two chunks.  Otherwise the
//     CTA's rows of the chunk partial go to memory and the last CTA of those
//     rows to arrive, over the chunks of the (request, kv head, query tile),
//     folds them in chunk order (9 to 15 chunks staged in shared memory).
// Shared-memory layouts (the same arithmetic): wide, K and V in their own
// images, two CTAs per SM; NARROW, V loaded over K once the first product is
// done (from L2, where the launch is small enough to prefetch it) and O
// accumulated over S in TMEM, three CTAs per SM, for launches of more
// clusters than the wide layout serves well; and attn_tc4_kernel, four CTAs
// per SM in 48 KB, for launches of more clusters than the narrow layout
// keeps resident.
// Bound by latency: each CTA is one dependent chain, of which an SM overlaps
// two to four.  With both parts of a query in one thread a pass takes 1079 us
// (1.5B, k = 0) and 2692 (7B, k = 8), with the parts in adjacent lanes,
// exchanged by shuffles, 1111 and 2749.
// Every fold boundary is a fixed absolute key position (128-key tiles,
// 1024-key chunks), and a fold with a part a row cannot see (fully masked:
// m = -inf, l = 0, O = 0) leaves it bitwise unchanged, so a row's result does
// not depend on the other rows of the call (batch invariance).
#include "as2d_internal.h"
#include "ptx_sm100.cuh"
#include "quotient.cuh"

namespace as2d {
namespace {

constexpr int kTile = 128;    // keys per CTA
constexpr int kCluster = 8;   // CTAs per cluster
constexpr int kChunk = kTile * kCluster;
constexpr int kQT = 64;       // queries per query tile (hi and lo rows interleaved)
constexpr uint32_t kRegion = 128 * 128;  // one 64-column region of 128 rows, bytes
// chunks whose partial rows the last arriver stages in shared memory: [15][8
// rows][128] floats and [15][8] (max, sum) within the first two 32 KB images
constexpr int kStage = 15;
static_assert(kStage * 8 * 128 * 4 + kStage * 8 * 8 <= 2 * 32768, "staging fits two images");
// Shared memory: the Q / P image, then the K and V tiles.  Wide (launches of
// up to kWideClusters clusters of 8): K and V in separate images, both
// requested at the start.  Narrow (larger launches): V is loaded over K once
// the first product has consumed it, so that three CTAs fit on an SM.
// Pair (wide only): clusters of 16 CTAs over two chunks, each CTA folding 4
// query rows of both, so that the chunks fold without going through global
// memory.
template <bool NARROW, bool PAIR>
constexpr uint32_t attn_smem() {
  return (NARROW ? 2 : 3) * 32768 + 64 * 8 + 5 * 8 + 16 + 1024;
}
static_assert(3 * (attn_smem<true, false>() + 1024) <= 228 * 1024, "three narrow CTAs per SM");
static_assert(2 * (attn_smem<false, true>() + 1024) <= 228 * 1024, "two wide CTAs per SM");
// A launch of more clusters of 8 than this takes the narrow layout.  The wide
// kernel's shared memory allows 36 clusters of 8 at two CTAs per SM.  Passes,
// us, wide / narrow: 7B, k = 8 with 32 clusters 2834 / 2860, 36 2847 / 2872,
// 40 3009 / 2880; blocks of the 1.5B with 32 1420 / 1464, 36 1472 / 1500, 40
// 1663 / 1520.
constexpr int kWideClusters = 32;
// Clusters of 8 the narrow layout keeps resident (three CTAs per SM, residency
// probe); larger launches take four CTAs per SM.  Passes, us, narrow / four:
// 7B, k = 8 with 48 clusters 2918 / 2938, 52 3029 / 2949, 60 3081 / 2978; blocks
// of the 1.5B with 48 1624 / 1638, 52 1772 / 1685.
constexpr int kNarrowClusters = 51;

struct AttnArgs {
  RowMap rm;
  const int32_t* len;
  int layer, batch, cap, nq, nkv;
  float qscale;  // log2(e) / sqrt(d), folded into the stored queries
  // split-K sums of the QKV projection (TC_PART)
  const float* qkv_part;  // [tile][split][qkv_ld][128], tile = column / 128
  const float* qkv_rinv;  // [qkv_ld] 1 / rms of each token row
  const float2* rope;     // [rows][d / 2] (cos, sin)
  int qkv_split, qkv_ld;
  bf16* kc;
  bf16* vc;
  uint8_t* qimg;          // [batch][nkv][qt_max] operand images, 256 d bytes each
  int qt_max;
  float* ws_o;            // [batch][nkv][qt_max][chunks_max][64][d] chunk partials
  float2* ws_ml;          // [batch][nkv][qt_max][chunks_max][64] (max, sum), base 2
  int chunks_max;
  int* cnt;               // [batch][nkv][qt_max][8] chunks arrived per 8-row group
  bf16* ao;               // [2 rows][nq d]: hi rows, then lo rows from lo_row
  int lo_row;
  int32_t* err;
  unsigned long long timeout_ns;
  int fold_later;         // chunk partials are folded by attn_fold_kernel
  int v_prefetch;         // narrow and quad: bring each tile's V into L2 with its K
  // clusters of request b: [cl_start[b], cl_start[b + 1]); n_ch[b] of them per
  // query tile (chunks covering the host's bound of the request's keys)
  int32_t cl_start[kMaxBatch + 1];
  int32_t n_ch[kMaxBatch];
};

// ---- finishing the QKV projection from its split-K sums ----------------------

// Byte offset of element (row r, column e) in a 128-row operand image of
// 128-byte-swizzled K-major bf16: 64-column regions of kRegion bytes, 16-byte
// chunk j of row r stored at chunk j ^ (r mod 8).
__device__ __forceinline__ uint32_t img_off(int r, int e) {
  const int reg = e >> 6, j = (e & 63) >> 3;
  return (uint32_t)reg * kRegion + (uint32_t)r * 128u + (uint32_t)((j ^ (r & 7)) << 4) +
         (uint32_t)((e & 7) << 1);
}

// Query q of a tile: its hi part is row hi_row(q) of the operand image and of
// the products, its lo part row hi_row(q) + 8.  Of every 16 rows the first 8
// are the hi parts of eight queries, the others their lo parts: the layout in
// which a 16-lane TMEM load gives a thread both parts of the same columns.
__device__ __forceinline__ int hi_row(int q) { return (q >> 3) * 16 + (q & 7); }

// Half a warp per (token row, head); lane l of it forms the pairs (e, e + D/2)
// of e = V l .. V l + V - 1.  Rotate-half RoPE: x' = x cos - x_p sin at e, x_p cos +
// x sin at e + D/2.  Bound by latency, as the residual projections' finishing
// kernel is (whose comment has the figures of both): addresses before the
// wait, every load issued before any is used, 16 bytes a lane (D = 128): with a
// warp to a head and 8 bytes a lane 64 requests of the 1.5B (576 rows) took 6962
// us, now 6859.  The
// dependent launch is triggered after the wait: attention CTAs that start
// before it read the requests' lengths (and measured slower: 7B k = 8 2784 ->
// 2810 us).
constexpr int kQkvWarps = 8;  // warps of one CTA, two heads each
template <int D>
__global__ void __launch_bounds__(32 * kQkvWarps) qkv_finish_kernel(const __grid_constant__ AttnArgs a) {
  constexpr int H2 = D / 2, V = H2 / 16;
  const int gm = blockIdx.x, head = 2 * (blockIdx.y * kQkvWarps + threadIdx.y) + (threadIdx.x >> 4);
  const int e = V * (threadIdx.x & 15);
  const int b = row_request(a.rm, gm), r0 = a.rm.start[b], i = gm - r0, rows = a.rm.start[b + 1] - r0;
  const bool live = head < a.nq + 2 * a.nkv;
  const bool is_q = head < a.nq, rotate = head < a.nq + a.nkv;
  // the split parts of columns head D + e .. and head D + e + H2 ..
  const int c0 = head * D + e, c1 = c0 + H2;
  const size_t part = (size_t)a.qkv_ld * 128;
  const float* s0 = a.qkv_part + ((size_t)(c0 >> 7) * a.qkv_split * a.qkv_ld + gm) * 128 + (c0 & 127);
  const float* s1 = a.qkv_part + ((size_t)(c1 >> 7) * a.qkv_split * a.qkv_ld + gm) * 128 + (c1 & 127);
  const float2* csp = a.rope + (size_t)gm * H2 + e;
  // where the results go: the query image's two rows of q, or
  // the cache entry at the request's length + i
  const int G = a.nq / a.nkv;
  const int g = is_q ? head / G : (rotate ? head - a.nq : head - a.nq - a.nkv);
  const int qg = i * G + (head - g * G), qt = qg / kQT, q = qg - qt * kQT;
  uint8_t* img = a.qimg + ((size_t)(b * a.nkv + g) * a.qt_max + qt) * (size_t)(256 * D);
  bf16* dst = (rotate ? a.kc : a.vc) + (((size_t)a.layer * a.batch + b) * a.nkv + g) * a.cap * D + e;
  ptx::griddep_wait();
  ptx::griddep_launch_dependents();
  if (!live) return;
  const int len_b = a.len[b];
  const float rinv = a.qkv_rinv[gm];
  float x[V], xp[V];
  float2 cs[V];
  {
    float v0[8][V], v1[8][V];
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r < a.qkv_split) {
        if constexpr (V == 4) {
          const float4 t0 = __ldcg(reinterpret_cast<const float4*>(s0 + r * part));
          const float4 t1 = __ldcg(reinterpret_cast<const float4*>(s1 + r * part));
          v0[r][0] = t0.x, v0[r][1] = t0.y, v0[r][2] = t0.z, v0[r][3] = t0.w;
          v1[r][0] = t1.x, v1[r][1] = t1.y, v1[r][2] = t1.z, v1[r][3] = t1.w;
        } else {
          const float2 t0 = __ldcg(reinterpret_cast<const float2*>(s0 + r * part));
          const float2 t1 = __ldcg(reinterpret_cast<const float2*>(s1 + r * part));
          v0[r][0] = t0.x, v0[r][1] = t0.y;
          v1[r][0] = t1.x, v1[r][1] = t1.y;
        }
      }
#pragma unroll
    for (int u = 0; u < V; ++u) cs[u] = rotate ? csp[u] : make_float2(1.f, 0.f);
    // the parts in rank order, times the row's 1 / rms
#pragma unroll
    for (int u = 0; u < V; ++u) {
      float t0 = 0.f, t1 = 0.f;
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < a.qkv_split) {
          t0 += v0[r][u];
          t1 += v1[r][u];
        }
      x[u] = t0 * rinv;
      xp[u] = t1 * rinv;
    }
  }
  if (!rows_fit(len_b, rows, a.cap)) return;  // flagged
  float y0[V], y1[V];
#pragma unroll
  for (int u = 0; u < V; ++u) {
    y0[u] = rotate ? fmaf(x[u], cs[u].x, -(xp[u] * cs[u].y)) : x[u];
    y1[u] = rotate ? fmaf(xp[u], cs[u].x, x[u] * cs[u].y) : xp[u];
  }
  // V consecutive bf16 (8- or 4-byte aligned)
  auto put = [](void* to, const float* v) {
    uint32_t w[V / 2];
#pragma unroll
    for (int u = 0; u < V / 2; ++u) {
      const __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * u], v[2 * u + 1]);
      w[u] = *reinterpret_cast<const uint32_t*>(&t);
    }
    if constexpr (V == 4)
      *reinterpret_cast<uint2*>(to) = make_uint2(w[0], w[1]);
    else
      *reinterpret_cast<uint32_t*>(to) = w[0];
  };
  if (is_q) {
    // hi parts, and what they leave (exact) as lo parts
    float l0[V], l1[V];
#pragma unroll
    for (int u = 0; u < V; ++u) {
      y0[u] *= a.qscale;
      y1[u] *= a.qscale;
      l0[u] = y0[u] - __bfloat162float(__float2bfloat16_rn(y0[u]));
      l1[u] = y1[u] - __bfloat162float(__float2bfloat16_rn(y1[u]));
    }
    const int row = hi_row(q);
    put(img + img_off(row, e), y0);
    put(img + img_off(row, e + H2), y1);
    put(img + img_off(row + 8, e), l0);
    put(img + img_off(row + 8, e + H2), l1);
  } else {
    dst += (size_t)(len_b + i) * D;
    put(dst, y0);
    put(dst + H2, y1);
  }
}

// ---- attention over 128-key tiles on the tensor cores ------------------------

// 2^x on the special-function unit (ftz: results below 2^-126 are 0).
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void dsmem_st_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}

__device__ __forceinline__ void dsmem_st_f2(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y)
               : "memory");
}

// A thread's share of a tile.  The four warps that read a tile's products
// cover 16 queries each: warp w, lane 4r + c holds queries 16w + r and 16w + 8
// + r (i = 0, 1), and of each the keys (dims) 8j + 2c + u, u < 2, as element 2j
// + u.  Hi and lo parts come to the same thread, so they are added without an
// exchange between lanes: with the parts in adjacent lanes (two selects and a
// shuffle an element) a tile took some 1500 instructions a warp, now 700, and
// the rows of P need no exchange either.
struct TileThread {
  int w, r, c;
  __device__ __forceinline__ TileThread(int warp, int lane) : w(warp & 3), r(lane >> 2), c(lane & 3) {}
  __device__ __forceinline__ int query(int i) const { return 16 * w + 8 * i + r; }
};
// Columns [0, 32 NCH) of one of the thread's queries (hi + lo) from the 16 TMEM
// lanes at taddr: every load issued before the wait.
template <int NCH>
__device__ __forceinline__ void tile_load(uint32_t taddr, float (&x)[8 * NCH]) {
  uint32_t v[NCH][16];
#pragma unroll
  for (int ch = 0; ch < NCH; ++ch) ptx::tmem_ld_16x256b_x4(taddr + 32 * ch, v[ch]);
  ptx::tmem_ld_wait();
#pragma unroll
  for (int ch = 0; ch < NCH; ++ch)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        x[8 * ch + 2 * j + u] =
            __uint_as_float(v[ch][4 * j + u]) + __uint_as_float(v[ch][4 * j + 2 + u]);
}

// P (>= 0) as bf16 pairs of keys: hi = P with its low 16 bits cleared (exact
// in bf16), lo = bf16(P - hi), so that hi + lo matches P to about 17 bits.
__device__ __forceinline__ void hi_lo(float x0, float x1, uint32_t& h, uint32_t& l) {
  const uint32_t b0 = __float_as_uint(x0), b1 = __float_as_uint(x1);
  h = __byte_perm(b0, b1, 0x7632);
  const __nv_bfloat162 lv = __floats2bfloat162_rn(x0 - __uint_as_float(b0 & 0xFFFF0000u),
                                                  x1 - __uint_as_float(b1 & 0xFFFF0000u));
  l = *reinterpret_cast<const uint32_t*>(&lv);
}

// P of one query into the 16 TMEM lanes at taddr (over S), where the second
// product reads its A operand: two keys a column, rows as the queries' rows.
// The caller waits for the stores (ptx::tmem_st_wait).
__device__ __forceinline__ void tile_store_p(uint32_t taddr, const float (&x)[32]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t v[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) hi_lo(x[16 * h + 2 * j], x[16 * h + 2 * j + 1], v[2 * j], v[2 * j + 1]);
    ptx::tmem_st_16x128b_x8(taddr + 32 * h, v);
  }
}
constexpr uint32_t kLane16 = 16u << 16;  // TMEM address of the upper 16 lanes of a warp's 32


// A partial row of O as the threads pass it on: position 16v + 4c + 2w + u
// holds dim 16v + 8w + 2c + u (each thread's four consecutive elements as one
// float4, the four threads of a row side by side).  The folds keep that order
// and write_rows undoes it.
__device__ __forceinline__ int part_pos(int c) { return 4 * c; }  // of thread c; + 16 v

// The weight of a part (max m) in a fold whose maximum is M: 2^(m - M), 0
// where m = -inf (nothing of the part is visible to the row), exactly 1 for
// the part holding the maximum.  Parts of weight 0 are skipped by the folds,
// so a part a row cannot see leaves its result bitwise unchanged.
__device__ __forceinline__ float part_weight(float m, float M) {
  return m == -INFINITY ? 0.f : (m == M ? 1.f : ex2(m - M));
}

// The tile's scores of one query (this thread's 32 keys p0 + 8j + 2c + u, in sv)
// -> P = 2^(S - m) in sv (visible keys: key <= lim; a masked key gets 0), with
// the tile's maximum m (-inf where nothing is visible) and sum l over the four
// threads of the query.
__device__ __forceinline__ void softmax_tail(float (&sv)[32], int c, int p0, int lim, float& m, float& l) {
  // (a tile wholly at or below the row's limit needs no mask)
  if (p0 + kTile - 1 > lim) {
    const int k0 = p0 + 2 * c;
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if (k0 + 8 * (t >> 1) + (t & 1) > lim) sv[t] = -INFINITY;
  }
  float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int t = 0; t < 32; ++t) mx4[t & 3] = fmaxf(mx4[t & 3], sv[t]);
  float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
  mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
  m = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
  const float ref = m == -INFINITY ? 0.f : m;  // (2^(-inf - 0) = 0)
  // sums in four interleaved parts, then ((0 + 1) + (2 + 3)), then over the
  // threads in pairs: a fixed order
  float ls4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int t = 0; t < 32; ++t) {
    sv[t] = ex2(sv[t] - ref);
    ls4[t & 3] += sv[t];
  }
  float ls = (ls4[0] + ls4[1]) + (ls4[2] + ls4[3]);
  ls += __shfl_xor_sync(0xFFFFFFFFu, ls, 1);
  l = ls + __shfl_xor_sync(0xFFFFFFFFu, ls, 2);
}

// Positions [fd, fd + DT) (fd a multiple of DT) of row fr of query tile qt,
// normalised (o / l), as bf16 hi and lo parts into the attention output; rows
// past the call's queries are skipped.  One reciprocal serves the row
// (quotient.cuh), as eight divisions in a row would hold up the chain.
template <int D, int DT>
__device__ __forceinline__ void write_rows(const AttnArgs& a, const float* o_, float Ls, int fr,
                                           int fd, int qt, int qn, int G, int g, int r0) {
  static_assert(DT == 4 || DT == 8, "one or two threads' elements");
  const int fqg = qt * kQT + fr;
  if (fqg >= qn) return;
  const int i = fqg / G, hq = g * G + (fqg - i * G);
  const float inv = 1.f / Ls;
  uint32_t hw[2][DT / 4], lw[2][DT / 4];  // [dims 2c .., dims 8 + 2c ..]
#pragma unroll
  for (int e = 0; e < DT / 2; ++e) {
    float v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) v[u] = quotient(o_[2 * e + u], Ls, inv);
    const __nv_bfloat162 hv = __floats2bfloat162_rn(v[0], v[1]);
    const float2 hf = __bfloat1622float2(hv);
    const __nv_bfloat162 lv = __floats2bfloat162_rn(v[0] - hf.x, v[1] - hf.y);
    hw[e & 1][e >> 1] = *reinterpret_cast<const uint32_t*>(&hv);
    lw[e & 1][e >> 1] = *reinterpret_cast<const uint32_t*>(&lv);
  }
  const size_t at = (size_t)(r0 + i) * a.nq * D + (size_t)hq * D + (fd & ~15) + ((fd & 15) >> 1);
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    bf16* hi = a.ao + at + 8 * w;
    bf16* lo = hi + (size_t)a.lo_row * a.nq * D;
    if constexpr (DT == 8) {
      *reinterpret_cast<uint2*>(hi) = make_uint2(hw[w][0], hw[w][1]);
      *reinterpret_cast<uint2*>(lo) = make_uint2(lw[w][0], lw[w][1]);
    } else {
      *reinterpret_cast<uint32_t*>(hi) = hw[w][0];
      *reinterpret_cast<uint32_t*>(lo) = lw[w][0];
    }
  }
}

// The fold of NT tile partials (rows at o, `stride` floats apart; their
// maxima m, -inf for none): o and l relative to the largest, fm.  Every load is
// issued before the first is used, and parts of weight 0 are dropped by
// selection (what lies in their place is not read into the sums).  The fold
// stands at the end of every layer's chain: with a branch for each part and
// eight divisions it took 1.5 us (1.5B, k = 8 1142 us a pass, now 1115).
template <int NT, int DT>
__device__ __forceinline__ void fold_tiles(const float* o, int stride, const float2 (&ml)[NT], float& fm,
                                           float& fl, float (&fo)[DT]) {
  float4 v[NT][DT / 4];
#pragma unroll
  for (int i = 0; i < NT; ++i)
#pragma unroll
    for (int u = 0; u < DT / 4; ++u) v[i][u] = reinterpret_cast<const float4*>(o + i * stride)[u];
  fm = -INFINITY;
#pragma unroll
  for (int i = 0; i < NT; ++i) fm = fmaxf(fm, ml[i].x);
  fl = 0.f;
#pragma unroll
  for (int e = 0; e < DT; ++e) fo[e] = 0.f;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const float w = part_weight(ml[i].x, fm);
    const bool on = w != 0.f;
    fl = on ? fmaf(ml[i].y, w, fl) : fl;
#pragma unroll
    for (int u = 0; u < DT / 4; ++u) {
      fo[4 * u] = on ? fmaf(v[i][u].x, w, fo[4 * u]) : fo[4 * u];
      fo[4 * u + 1] = on ? fmaf(v[i][u].y, w, fo[4 * u + 1]) : fo[4 * u + 1];
      fo[4 * u + 2] = on ? fmaf(v[i][u].z, w, fo[4 * u + 2]) : fo[4 * u + 2];
      fo[4 * u + 3] = on ? fmaf(v[i][u].w, w, fo[4 * u + 3]) : fo[4 * u + 3];
    }
  }
}

// The fold of a chunk's 8 tile partials for query rows 8 rank .. 8 rank + 7
// (received into s_rml [8 tiles][8 rows] and recv [8 tiles][8 rows][D]) and
// what follows it: with one chunk the rows are normalised and written; with
// several, the rows of the chunk partial go to memory, for attn_fold_kernel
// (fold_later) or for the last CTA of these rows to arrive, which folds the
// chunks in chunk order (9 to STAGE chunks staged in shared memory at sm,
// whose images are no longer read; none with STAGE 0).
template <int D, int STAGE>
__device__ __forceinline__ void fold_chunk8(const AttnArgs& a, const float* recv,
                                            const float2* s_rml, int* s_flag, uint8_t* sm,
                                            uint32_t rank, int c, int n_tiles, int n_chunks, int b,
                                            int g, int qt, int qn, int G, int r0) {
  constexpr int DT = D / 16;  // dims per thread (8 rows x 16 threads)
  const int tid = threadIdx.x;
  // ---- fold (thread: query row 8 rank + fj, positions [fd, fd + DT)) ----------
  const int n_here = min(kCluster, n_tiles - c * kCluster);  // tiles of this chunk with keys
  const int fj = tid >> 4, fr = 8 * (int)rank + fj, fd = DT * (tid & 15);
  float fm, fl, fo[DT];
  {
    float2 pml[kCluster];
#pragma unroll
    for (int i = 0; i < kCluster; ++i)
      pml[i] = (i < n_here) ? s_rml[i * 8 + fj] : make_float2(-INFINITY, 0.f);
    fold_tiles<kCluster, DT>(recv + fj * D + fd, 8 * D, pml, fm, fl, fo);
  }
  // normalise and write the row's positions (o / l as bf16 hi, lo)
  auto write_out = [&](const float* o_, float Ls) {
    write_rows<D, DT>(a, o_, Ls, fr, fd, qt, qn, G, g, r0);
  };
  if (n_chunks == 1) {
    write_out(fo, fl);
    return;
  }
  // ---- several chunks: this CTA's rows of the chunk partial go to memory;
  // the last chunk's CTA of these rows to arrive folds them in chunk order
  const size_t item = (size_t)(b * a.nkv + g) * a.qt_max + qt;
  {
    const size_t pc = item * a.chunks_max + c;
    float4* dst = reinterpret_cast<float4*>(a.ws_o + (pc * kQT + fr) * D + fd);
#pragma unroll
    for (int u = 0; u < DT / 4; ++u)
      dst[u] = make_float4(fo[4 * u], fo[4 * u + 1], fo[4 * u + 2], fo[4 * u + 3]);
    if ((tid & 15) == 0) a.ws_ml[pc * kQT + fr] = make_float2(fm, fl);
  }
  if (a.fold_later) return;
  __syncthreads();
  int* cnt = a.cnt + item * kCluster + rank;
  if (tid == 0) {
    // the arrival releases the CTA's writes above (ordered before it by the
    // barrier) and acquires the other chunks' partials for the last arriver
    int prev;
    asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], 1;" : "=r"(prev) : "l"(cnt) : "memory");
    const int last = prev == n_chunks - 1;
    if (last) *cnt = 0;  // every chunk of these rows has arrived
    *s_flag = last;
  }
  __syncthreads();
  if (!*s_flag) return;
  float cl_ = 0.f, co[DT];
#pragma unroll
  for (int e = 0; e < DT; ++e) co[e] = 0.f;
  if constexpr (STAGE > 0) {
    if (n_chunks > 8 && n_chunks <= STAGE) {
      // nine or more chunks: every chunk's rows come into shared memory (over
      // the Q / P and K images, no longer read) by copies issued together, one
      // memory round trip instead of two through registers
      float* st_o = reinterpret_cast<float*>(sm);                          // [chunk][8 rows][D]
      float2* st_ml = reinterpret_cast<float2*>(sm + STAGE * 8 * D * 4);  // [chunk][8 rows]
      for (int cc = 0; cc < n_chunks; ++cc) {
        const size_t pc = item * a.chunks_max + cc;
        const float* src = a.ws_o + (pc * kQT + fr) * D + fd;
        float* dst = st_o + (cc * 8 + fj) * D + fd;
  #pragma unroll
        for (int u = 0; u < DT / 4; ++u) ptx::cp_async16(dst + 4 * u, src + 4 * u);
        // (max, sum) of rows fj and fj + 1 in one copy
        if ((tid & 15) == 0 && (fj & 1) == 0) ptx::cp_async16(st_ml + cc * 8 + fj, a.ws_ml + pc * kQT + fr);
      }
      ptx::cp_async_wait_all();
      __syncthreads();
      float cm = -INFINITY;
      for (int cc = 0; cc < n_chunks; ++cc) cm = fmaxf(cm, st_ml[cc * 8 + fj].x);
      for (int cc = 0; cc < n_chunks; ++cc) {
        const float2 ml = st_ml[cc * 8 + fj];
        const float w = part_weight(ml.x, cm);
        if (w != 0.f) {
          cl_ += ml.y * w;
          const float4* src = reinterpret_cast<const float4*>(st_o + (cc * 8 + fj) * D + fd);
  #pragma unroll
          for (int u = 0; u < DT / 4; ++u) {
            const float4 v = src[u];
            co[4 * u + 0] += v.x * w;
            co[4 * u + 1] += v.y * w;
            co[4 * u + 2] += v.z * w;
            co[4 * u + 3] += v.w * w;
          }
        }
      }
      write_out(co, cl_);
      return;
    }
  }
  // eight chunks' values in flight at a time; the first eight are requested
  // together with every chunk's maximum, so that up to eight chunks take one
  // memory round trip
  float4 v[8][DT / 4];
  float2 ml[8];
  auto load8 = [&](int c0) {
#pragma unroll
    for (int u8 = 0; u8 < 8; ++u8)
      if (c0 + u8 < n_chunks) {
        const size_t pc = item * a.chunks_max + c0 + u8;
        ml[u8] = __ldcg(a.ws_ml + pc * kQT + fr);
        const float4* src = reinterpret_cast<const float4*>(a.ws_o + (pc * kQT + fr) * D + fd);
#pragma unroll
        for (int u = 0; u < DT / 4; ++u) v[u8][u] = __ldcg(src + u);
      }
  };
  // more chunks than shared memory holds, but no more than eight plus that:
  // chunks 8.. come into shared memory by copies issued together with the
  // first eight's loads, so that all of them take one memory round trip
  const bool hybrid = STAGE > 0 && n_chunks > 8 && n_chunks - 8 <= STAGE;
  float* st_o = reinterpret_cast<float*>(sm);                          // [chunk - 8][8 rows][D]
  float2* st_ml = reinterpret_cast<float2*>(sm + STAGE * 8 * D * 4);  // [chunk - 8][8 rows]
  if (hybrid) {
    for (int cc = 8; cc < n_chunks; ++cc) {
      const size_t pc = item * a.chunks_max + cc;
      const float* src = a.ws_o + (pc * kQT + fr) * D + fd;
      float* dst = st_o + ((cc - 8) * 8 + fj) * D + fd;
#pragma unroll
      for (int u = 0; u < DT / 4; ++u) ptx::cp_async16(dst + 4 * u, src + 4 * u);
      if ((tid & 15) == 0 && (fj & 1) == 0)
        ptx::cp_async16(st_ml + (cc - 8) * 8 + fj, a.ws_ml + pc * kQT + fr);
    }
  }
  load8(0);
  float cm = -INFINITY;
  for (int cc = 8; cc < n_chunks; ++cc)
    cm = fmaxf(cm, __ldcg(a.ws_ml + (item * a.chunks_max + cc) * kQT + fr).x);
#pragma unroll
  for (int u8 = 0; u8 < 8; ++u8)
    if (u8 < n_chunks) cm = fmaxf(cm, ml[u8].x);
  for (int c0 = 0; c0 < n_chunks; c0 += 8) {
    if (hybrid && c0 == 8) {
      ptx::cp_async_wait_all();
      __syncthreads();
      for (int cc = 8; cc < n_chunks; ++cc) {
        const float2 mlc = st_ml[(cc - 8) * 8 + fj];
        const float w = part_weight(mlc.x, cm);
        if (w != 0.f) {
          cl_ += mlc.y * w;
          const float4* src = reinterpret_cast<const float4*>(st_o + ((cc - 8) * 8 + fj) * D + fd);
#pragma unroll
          for (int u = 0; u < DT / 4; ++u) {
            const float4 vv = src[u];
            co[4 * u + 0] += vv.x * w;
            co[4 * u + 1] += vv.y * w;
            co[4 * u + 2] += vv.z * w;
            co[4 * u + 3] += vv.w * w;
          }
        }
      }
      break;
    }
    if (c0 > 0) load8(c0);
#pragma unroll
    for (int u8 = 0; u8 < 8; ++u8)
      if (c0 + u8 < n_chunks) {
        const float w = part_weight(ml[u8].x, cm);
        if (w != 0.f) {
          cl_ += ml[u8].y * w;
#pragma unroll
          for (int u = 0; u < DT / 4; ++u) {
            co[4 * u + 0] += v[u8][u].x * w;
            co[4 * u + 1] += v[u8][u].y * w;
            co[4 * u + 2] += v[u8][u].z * w;
            co[4 * u + 3] += v[u8][u].w * w;
          }
        }
      }
  }
  write_out(co, cl_);
}

template <int D, bool NARROW, bool PAIR>
__global__ void __launch_bounds__(128, NARROW ? 3 : 2)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ AttnArgs a) {
  constexpr int NR = D / 64;          // 64-column regions of a K / V tile
  constexpr uint32_t K_BYTES = NR * kRegion;            // one K or V tile
  constexpr uint32_t TMEM_COLS = NARROW ? 128 : 256;   // narrow: O over S
  constexpr uint32_t Q_BYTES = 2u * kQT * D * 2;
  constexpr int DQ = D / 4;           // dims of a query that a thread holds
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* R0 = sm;            // Q image -> P image
  uint8_t* R1 = sm + 32768;    // K tile -> the partials received from the cluster
  uint8_t* R2 = NARROW ? R1 : sm + 65536;  // V tile (narrow: over K, after the first product)
  float* recv = reinterpret_cast<float*>(R1);  // [8 tiles][8 rows][D] received
  // [tiles of the cluster][rows folded here] (max, sum): [8][8], pair [16][4]
  float2* s_rml = reinterpret_cast<float2*>(sm + (NARROW ? 2 : 3) * 32768);
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_rml + 64);  // q, k (wide: and v), mma1, mma2, v
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 5);
  int* s_flag = reinterpret_cast<int*>(tslot + 1);

  const int tid = threadIdx.x, warp = tid >> 5;
  // a cluster covers HALVES chunks of 8 tiles; half: this CTA's chunk of
  // them, rank: its tile within the chunk
  constexpr int HALVES = PAIR ? 2 : 1;
  const uint32_t crank = ptx::cluster_rank();
  const int half = (int)(crank >> 3);
  const uint32_t rank = crank & 7u;
  const int cl = (int)(blockIdx.x / (kCluster * HALVES)), g = blockIdx.y;
  int b = 0;
  while (b + 1 < a.rm.batch && a.cl_start[b + 1] <= cl) ++b;
  const int ci = cl - a.cl_start[b];
  const int ncl = (a.n_ch[b] + HALVES - 1) / HALVES;  // clusters per query tile
  const int qt = ci / ncl, c2 = ci - qt * ncl;
  const int c = c2 * HALVES + half;  // this CTA's chunk
  const int t = c * kCluster + (int)rank, p0 = t * kTile;
  const int r0 = a.rm.start[b], M = a.rm.start[b + 1] - r0;
  const int G = a.nq / a.nkv, qn = M * G;
  const int L = a.len[b];
  const bool fits = rows_fit(L, M, a.cap);
  const int kend = L + M;
  const int n_tiles = fits ? (kend + kTile - 1) / kTile : 0;
  const int n_chunks = (n_tiles + kCluster - 1) / kCluster;
  const bool active = t < n_tiles;      // this CTA's tile holds keys
  const bool cl_active = c2 * HALVES < n_chunks;  // uniform over the cluster
  if (!cl_active) return;               // the whole cluster holds no keys of this request
  const int z = (a.layer * a.batch + b) * a.nkv + g;
  const uint8_t* qsrc = a.qimg + ((size_t)(b * a.nkv + g) * a.qt_max + qt) * (size_t)Q_BYTES;

  if (tid == 0) {
    for (int i = 0; i < 5; ++i) ptx::mbar_init(&bars[i], 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) ptx::tmem_alloc(tslot, TMEM_COLS);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t lane_base = (uint32_t)(32 * warp) << 16;

  // a tile of entries older than this call does not depend on the finishing
  // kernel: request it before the wait
  const bool early = active && p0 + kTile <= L;
  const uint64_t pol = ptx::policy_evict_first();
  auto load_kv = [&]() {
    ptx::mbar_arrive_expect_tx(&bars[1], NARROW ? K_BYTES : 2 * K_BYTES);
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      ptx::tma_load_3d(R1 + h * kRegion, &tmK, &bars[1], 64 * h, p0, z, pol);
      // narrow: V is loaded once the first product has consumed the keys;
      // in launches of a few waves it is brought into L2 now
      if (!NARROW)
        ptx::tma_load_3d(R2 + h * kRegion, &tmV, &bars[1], 64 * h, p0, z, pol);
      else if (a.v_prefetch)
        ptx::tma_prefetch_3d(&tmV, 64 * h, p0, z);
    }
  };
  auto load_v = [&]() {  // narrow: into the K image, once the first product is done
    ptx::mbar_arrive_expect_tx(&bars[4], K_BYTES);
#pragma unroll
    for (int h = 0; h < NR; ++h) ptx::tma_load_3d(R2 + h * kRegion, &tmV, &bars[4], 64 * h, p0, z, pol);
  };
  if (tid == 0 && early) {
    ptx::prefetch_tmap(&tmK);
    ptx::prefetch_tmap(&tmV);
    load_kv();
  }
  ptx::griddep_wait();
  if (tid == 0 && active) {
    if (!early) load_kv();
    ptx::mbar_arrive_expect_tx(&bars[0], Q_BYTES);
    ptx::bulk_load(R0, qsrc, Q_BYTES, &bars[0], ptx::policy_evict_last());
  }

  const TileThread me(warp, tid & 31);
  int lim[2];                                              // each query's last visible key
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // the tile partials
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int qg = qt * kQT + me.query(i);
    lim[i] = qg < qn ? L + qg / G : -1;
  }
  float o[2][DQ];
#pragma unroll
  for (int j = 0; j < DQ; ++j) o[0][j] = o[1][j] = 0.f;
  bool ok = true;
  if (active) {
    ok = ptx::mbar_wait(&bars[0], 0, a.timeout_ns) && ptx::mbar_wait(&bars[1], 0, a.timeout_ns);
    ok = ptx::group_all(ok, 1, 128);
    if (!ok) {
      if (tid == 0) {
        atomicOr(a.err, kErrTimeout);
        // the copies may still be in flight: wait for them before the CTA ends
        ptx::mbar_wait(&bars[0], 0, ptx::kDrainNs);
        ptx::mbar_wait(&bars[1], 0, ptx::kDrainNs);
      }
      __syncthreads();
    }
  }
  // values past the call's last key (stale entries, or NaN in a poisoned
  // cache) would reach O through 0 * V: those rows of the V tile are zeroed
  auto zero_v_tail = [&]() {
    const int z0 = kend - p0;
    if (z0 < kTile) {
      for (int idx = tid; idx < (kTile - z0) * NR * 8; idx += 128) {
        const int r = z0 + idx / (NR * 8), rest = idx - (idx / (NR * 8)) * (NR * 8);
        *reinterpret_cast<uint4*>(R2 + (rest >> 3) * kRegion + r * 128 + (rest & 7) * 16) =
            make_uint4(0, 0, 0, 0);
      }
      ptx::fence_proxy_async_smem();
    }
  };
  // Every thread arrives once at the split cluster barrier, when its CTA no
  // longer reads the image the cluster's partials are received into (the K
  // image: wide after the first product, narrow after the second, V being
  // loaded there): the product's completion, observed on its mbarrier, means
  // its operand reads are done, so the arrival needs no release.  The others
  // wait for the arrival only when they push.
  if (active && ok) {
    if (tid == 0) {
      ptx::tc_fence_after();
      constexpr uint32_t IDESC1 = ptx::idesc_bf16_f32(128, kTile);
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const uint64_t ad = ptx::sdesc_sw128(ptx::smem_u32(R0 + (kk >> 2) * kRegion)) + 2 * (kk & 3);
        const uint64_t bd = ptx::sdesc_sw128(ptx::smem_u32(R1 + (kk >> 2) * kRegion)) + 2 * (kk & 3);
        ptx::mma_bf16(tmem, ad, bd, IDESC1, kk > 0 ? 1u : 0u);
      }
      ptx::mma_commit(&bars[2]);
    }
    if (!NARROW) zero_v_tail();  // while the first product runs
    const bool ok1 = ptx::group_all(ptx::mbar_wait(&bars[2], 0, a.timeout_ns), 1, 128);
    // (after a timeout: once the product has drained)
    if (!ok1 && tid == 0) ptx::mbar_wait(&bars[2], 0, ptx::kDrainNs);
    if (!NARROW || !ok1) ptx::cluster_arrive_relaxed();
    // narrow: the keys are consumed; V comes into their image during the softmax
    if (NARROW && ok1 && tid == 0) load_v();
    ptx::tc_fence_after();
    bool ok2 = ok1, vok = ok1;
    if (ok1) {
      // S = hi + lo, masked; the tile's maximum and P = 2^(S - m).  P's hi
      // and lo parts: wide, into TMEM over S; narrow, into the operand image in
      // shared memory, K-major by key (the same values)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float sv[32];
        tile_load<4>(tmem + lane_base + i * kLane16, sv);
        softmax_tail(sv, me.c, p0, lim[i], m[i], l[i]);
        if (!NARROW) {
          tile_store_p(tmem + lane_base + i * kLane16, sv);
        } else {
          const int row = hi_row(me.query(i));
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            uint32_t h, lo;
            hi_lo(sv[2 * j], sv[2 * j + 1], h, lo);
            *reinterpret_cast<uint32_t*>(R0 + img_off(row, 8 * j + 2 * me.c)) = h;
            *reinterpret_cast<uint32_t*>(R0 + img_off(row + 8, 8 * j + 2 * me.c)) = lo;
          }
        }
      }
      if (!NARROW) ptx::tmem_st_wait();
      if (NARROW) {
        vok = ptx::group_all(ptx::mbar_wait(&bars[4], 0, a.timeout_ns), 1, 128);
        if (vok) zero_v_tail();
      }
      ptx::fence_proxy_async_smem();
      // (narrow: the second product writes O over S, read out above)
      ptx::tc_fence_before();
      __syncthreads();
      if (tid == 0 && vok) {
        ptx::tc_fence_after();
        constexpr uint32_t IDESC2 = ptx::idesc_bf16_f32(128, D, true);
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          const uint64_t bd = ptx::sdesc_sw128_mn(ptx::smem_u32(R2) + kk * 2048u, kRegion, 1024u);
          if (NARROW) {
            const uint64_t ad = ptx::sdesc_sw128(ptx::smem_u32(R0 + (kk >> 2) * kRegion)) + 2 * (kk & 3);
            ptx::mma_bf16(tmem, ad, bd, IDESC2, kk > 0 ? 1u : 0u);
          } else {
            // A: 16 keys = 8 columns per k-step
            ptx::mma_bf16_ta(tmem + 128, tmem + 8u * kk, bd, IDESC2, kk > 0 ? 1u : 0u);
          }
        }
        ptx::mma_commit(&bars[3]);
      }
      ok2 = vok && ptx::group_all(ptx::mbar_wait(&bars[3], 0, a.timeout_ns), 1, 128);
      if (NARROW) {
        // (after a timeout: once the copy and the product have drained)
        if (!ok2 && tid == 0) {
          ptx::mbar_wait(&bars[4], 0, ptx::kDrainNs);
          if (vok) ptx::mbar_wait(&bars[3], 0, ptx::kDrainNs);
        }
        ptx::cluster_arrive_relaxed();
      }
      ptx::tc_fence_after();
      if (ok2) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
          tile_load<D / 32>(tmem + lane_base + i * kLane16 + (NARROW ? 0 : 128), o[i]);
      }
    }
    if (!(ok1 && ok2)) {
      if (tid == 0) {
        atomicOr(a.err, kErrTimeout);
        // no MMA may still run when TMEM is freed
        ptx::mbar_wait(&bars[2], 0, ptx::kDrainNs);
        if (vok) ptx::mbar_wait(&bars[3], 0, ptx::kDrainNs);
      }
      m[0] = m[1] = -INFINITY;  // nothing of this tile is passed on
    }
  } else {
    ptx::cluster_arrive_relaxed();  // no keys of this CTA's tile are read
  }
  // the tile's products are done: the next kernel (the O projection) may
  // start and stream its first weight tiles now (earlier, they would compete
  // with this kernel's own loads)
  ptx::griddep_launch_dependents();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) ptx::tmem_dealloc(tmem, TMEM_COLS);

  // ---- the cluster's tile partials, pushed to the CTA that folds them ----
  // CTA r folds query rows RPC r .. RPC r + RPC - 1 (RPC: 8 in a cluster of
  // 8, 4 in a cluster of 16); it receives, from the CTA of every tile i of
  // the cluster, rows (max, sum) into s_rml[i][row] and O into
  // recv[i][row][d], over its K image (every CTA's is consumed once all have
  // arrived)
  constexpr int RPC = PAIR ? 4 : 8;
  ptx::cluster_wait();
  if (active) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int q = me.query(i);
      const uint32_t dst_rank = (uint32_t)(q / RPC), row = (uint32_t)(q % RPC);
      if (me.c == 0)
        dsmem_st_f2(ptx::dsmem_map(ptx::smem_u32(s_rml + crank * RPC + row), dst_rank),
                    make_float2(m[i], l[i]));
      if (m[i] != -INFINITY) {
        const uint32_t dst =
            ptx::dsmem_map(ptx::smem_u32(recv + (crank * RPC + row) * D + part_pos(me.c)), dst_rank);
#pragma unroll
        for (int u = 0; u < DQ / 4; ++u)
          dsmem_st_f4(dst + 64u * u, make_float4(o[i][4 * u], o[i][4 * u + 1], o[i][4 * u + 2], o[i][4 * u + 3]));
      }
    }
  }
  ptx::cluster_sync();

  if (PAIR) {
    // ---- two chunks in one cluster: CTA r folds rows 4r..4r+3, each
    // chunk's 8 tiles in tile order, then the two chunk partials in chunk
    // order: the arithmetic of the one-chunk fold and of the fold through
    // memory below (thread: row fj, positions [fd, fd + 4))
    constexpr int TPR = D / 4 < 32 ? D / 4 : 32;  // threads per row
    if (tid < 4 * TPR) {
      const int fj = tid / TPR, fr = 4 * (int)crank + fj, fd = 4 * (tid % TPR);
      float cmx[2], cls[2], cfo[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int nh = min(kCluster, n_tiles - (c2 * 2 + h) * kCluster);  // may be <= 0
        float2 pml[kCluster];
#pragma unroll
        for (int i = 0; i < kCluster; ++i)
          pml[i] = (i < nh) ? s_rml[(h * kCluster + i) * 4 + fj] : make_float2(-INFINITY, 0.f);
        fold_tiles<kCluster, 4>(recv + (h * kCluster * 4 + fj) * D + fd, 4 * D, pml, cmx[h], cls[h], cfo[h]);
      }
      if (n_chunks == 1) {
        write_rows<D, 4>(a, cfo[0], cls[0], fr, fd, qt, qn, G, g, r0);
      } else {
        float cm = -INFINITY;
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) cm = fmaxf(cm, cmx[cc]);
        float cl_ = 0.f, co[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const float w = part_weight(cmx[cc], cm);
          if (w != 0.f) {
            cl_ += cls[cc] * w;
#pragma unroll
            for (int e = 0; e < 4; ++e) co[e] += cfo[cc][e] * w;
          }
        }
        write_rows<D, 4>(a, co, cl_, fr, fd, qt, qn, G, g, r0);
      }
    }
    return;
  }

  fold_chunk8<D, kStage>(a, recv, s_rml, s_flag, sm, rank, c, n_tiles, n_chunks, b, g, qt, qn, G, r0);
}

// Four CTAs per SM (QUAD), for launches of more clusters than the narrow
// layout keeps resident: the narrow layout's tiles, arithmetic and fold in
// 48 KB of shared memory, 128 TMEM columns and at most 128 registers a
// thread.  The first product runs in halves of d (the whole Q image, one
// 16 KB region of the K tile at a time); V is loaded over Q; P goes to TMEM
// over S, and the second product runs in 64-dim halves of O over S's second
// half, each read out before the next.  S is read and P written in 16-key
// chunks, so that no thread holds a whole row of either.
constexpr uint32_t attn4_smem() { return 32768 + 16384 + 64 * 8 + 8 * 8 + 16 + 1024; }
static_assert(4 * (attn4_smem() + 1024) <= 228 * 1024, "four CTAs per SM");
template <int D>
__global__ void __launch_bounds__(128, 4)
    attn_tc4_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ AttnArgs a) {
  constexpr int NR = D / 64;          // 64-column regions of a K / V tile
  constexpr uint32_t Q_BYTES = 2u * kQT * D * 2;
  constexpr int DQ = D / 4;           // dims of a query that a thread holds
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* R0 = sm;            // Q image -> V tile -> the partials received from the cluster
  uint8_t* RK = sm + 32768;    // one 64-column region of the K tile
  float* recv = reinterpret_cast<float*>(R0);                // [8 tiles][8 rows][D]
  float2* s_rml = reinterpret_cast<float2*>(sm + 49152);    // [8][8] (max, sum)
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_rml + 64);  // q, k0, s0, k1, s1, v, o0, o1
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 8);
  int* s_flag = reinterpret_cast<int*>(tslot + 1);

  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t rank = ptx::cluster_rank();
  const int cl = (int)(blockIdx.x / kCluster), g = blockIdx.y;
  int b = 0;
  while (b + 1 < a.rm.batch && a.cl_start[b + 1] <= cl) ++b;
  const int ci = cl - a.cl_start[b];
  const int ncl = a.n_ch[b];  // clusters per query tile
  const int qt = ci / ncl, c = ci - qt * ncl;
  const int t = c * kCluster + (int)rank, p0 = t * kTile;
  const int r0 = a.rm.start[b], M = a.rm.start[b + 1] - r0;
  const int G = a.nq / a.nkv, qn = M * G;
  const int L = a.len[b];
  const bool fits = rows_fit(L, M, a.cap);
  const int kend = L + M;
  const int n_tiles = fits ? (kend + kTile - 1) / kTile : 0;
  const int n_chunks = (n_tiles + kCluster - 1) / kCluster;
  const bool active = t < n_tiles;
  if (c >= n_chunks) return;  // the whole cluster holds no keys of this request
  const int z = (a.layer * a.batch + b) * a.nkv + g;
  const uint8_t* qsrc = a.qimg + ((size_t)(b * a.nkv + g) * a.qt_max + qt) * (size_t)Q_BYTES;

  if (tid == 0) {
    for (int i = 0; i < 8; ++i) ptx::mbar_init(&bars[i], 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) ptx::tmem_alloc(tslot, 128);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t lane_base = (uint32_t)(32 * warp) << 16;

  const uint64_t pol = ptx::policy_evict_first();
  uint32_t issued = 0;  // (thread 0) barriers with a copy or product outstanding
  auto load_k = [&](int h, int bar) {  // region h of the K tile into RK
    ptx::mbar_arrive_expect_tx(&bars[bar], kRegion);
    ptx::tma_load_3d(RK, &tmK, &bars[bar], 64 * h, p0, z, pol);
    issued |= 1u << bar;
  };
  auto prefetch_rest = [&]() {  // the other K regions (and V, in launches of a few waves) into L2
#pragma unroll
    for (int h = 1; h < NR; ++h) ptx::tma_prefetch_3d(&tmK, 64 * h, p0, z);
    if (a.v_prefetch)
      for (int h = 0; h < NR; ++h) ptx::tma_prefetch_3d(&tmV, 64 * h, p0, z);
  };
  // a tile of entries older than this call does not depend on the finishing
  // kernel: request it before the wait
  const bool early = active && p0 + kTile <= L;
  if (tid == 0 && early) {
    ptx::prefetch_tmap(&tmK);
    ptx::prefetch_tmap(&tmV);
    load_k(0, 1);
    prefetch_rest();
  }
  ptx::griddep_wait();
  if (tid == 0 && active) {
    if (!early) {
      load_k(0, 1);
      prefetch_rest();
    }
    ptx::mbar_arrive_expect_tx(&bars[0], Q_BYTES);
    ptx::bulk_load(R0, qsrc, Q_BYTES, &bars[0], ptx::policy_evict_last());
    issued |= 1u;
  }

  const TileThread me(warp, tid & 31);
  int lim[2];                                              // each query's last visible key
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // the tile partials
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int qg = qt * kQT + me.query(i);
    lim[i] = qg < qn ? L + qg / G : -1;
  }
  float o[2][DQ];  // written by the second product's read-out; pushed only then
  auto wait_all = [&](bool ok, int bar) {
    return ptx::group_all(ok && ptx::mbar_wait(&bars[bar], 0, a.timeout_ns), 1, 128);
  };
  bool ok = true;
  if (active) {
    ok = wait_all(wait_all(true, 0), 1);
    // S = Q K^T in halves of d: region h of Q and of K, one accumulation chain
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      if (h > 0) {
        if (ok && tid == 0) load_k(h, 3);  // over the region the first half consumed
        ok = wait_all(ok, 3);
      }
      if (ok && tid == 0) {
        ptx::tc_fence_after();
        constexpr uint32_t IDESC1 = ptx::idesc_bf16_f32(128, kTile);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
          const int kk = 4 * h + k4;
          const uint64_t ad = ptx::sdesc_sw128(ptx::smem_u32(R0 + h * kRegion)) + 2 * k4;
          const uint64_t bd = ptx::sdesc_sw128(ptx::smem_u32(RK)) + 2 * k4;
          ptx::mma_bf16(tmem, ad, bd, IDESC1, kk > 0 ? 1u : 0u);
        }
        ptx::mma_commit(&bars[2 + 2 * h]);
        issued |= 1u << (2 + 2 * h);
      }
      ok = wait_all(ok, 2 + 2 * h);
    }
    // Q and K are consumed: V comes over Q (from L2) during the softmax
    if (ok && tid == 0) {
      ptx::mbar_arrive_expect_tx(&bars[5], NR * kRegion);
#pragma unroll
      for (int h = 0; h < NR; ++h) ptx::tma_load_3d(R0 + h * kRegion, &tmV, &bars[5], 64 * h, p0, z, pol);
      issued |= 1u << 5;
    }
    ptx::tc_fence_after();
    if (ok) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float sv[32];
        tile_load<4>(tmem + lane_base + i * kLane16, sv);
        softmax_tail(sv, me.c, p0, lim[i], m[i], l[i]);
        tile_store_p(tmem + lane_base + i * kLane16, sv);
      }
      ptx::tmem_st_wait();
    }
    ok = wait_all(ok, 5);
    // values past the call's last key would reach O through 0 * V
    if (ok) {
      const int z0 = kend - p0;
      if (z0 < kTile) {
        for (int idx = tid; idx < (kTile - z0) * NR * 8; idx += 128) {
          const int r = z0 + idx / (NR * 8), rest = idx - (idx / (NR * 8)) * (NR * 8);
          *reinterpret_cast<uint4*>(R0 + (rest >> 3) * kRegion + r * 128 + (rest & 7) * 16) =
              make_uint4(0, 0, 0, 0);
        }
      }
    }
    ptx::fence_proxy_async_smem();
    // O = P V in 64-dim halves into TMEM columns 64..127 (S's second half,
    // read out above), each read out before the next is written
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      ptx::tc_fence_before();
      __syncthreads();
      if (ok && tid == 0) {
        ptx::tc_fence_after();
        constexpr uint32_t IDESC2 = ptx::idesc_bf16_f32(128, 64, true);
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          const uint64_t bd =
              ptx::sdesc_sw128_mn(ptx::smem_u32(R0 + h * kRegion) + kk * 2048u, kRegion, 1024u);
          ptx::mma_bf16_ta(tmem + 64, tmem + 8u * kk, bd, IDESC2, kk > 0 ? 1u : 0u);
        }
        ptx::mma_commit(&bars[6 + h]);
        issued |= 1u << (6 + h);
      }
      ok = wait_all(ok, 6 + h);
      ptx::tc_fence_after();
      if (ok) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
          tile_load<2>(tmem + lane_base + i * kLane16 + 64, *reinterpret_cast<float(*)[16]>(&o[i][16 * h]));
      }
    }
    if (!ok) {
      if (tid == 0) {
        atomicOr(a.err, kErrTimeout);
        // no copy or product may still run when TMEM is freed and the CTA ends
        for (int i = 0; i < 8; ++i)
          if (issued & (1u << i)) ptx::mbar_wait(&bars[i], 0, ptx::kDrainNs);
      }
      m[0] = m[1] = -INFINITY;  // nothing of this tile is passed on
    }
  }
  // the V image is consumed: the cluster's partials may come into it
  ptx::cluster_arrive_relaxed();
  ptx::griddep_launch_dependents();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) ptx::tmem_dealloc(tmem, 128);

  // ---- the tile partials, pushed to the CTA that folds their rows ----------
  ptx::cluster_wait();
  if (active) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int q = me.query(i);
      const uint32_t dst_rank = (uint32_t)(q / 8), row = (uint32_t)(q % 8);
      if (me.c == 0)
        dsmem_st_f2(ptx::dsmem_map(ptx::smem_u32(s_rml + rank * 8 + row), dst_rank),
                    make_float2(m[i], l[i]));
      if (m[i] != -INFINITY) {
        const uint32_t dst =
            ptx::dsmem_map(ptx::smem_u32(recv + (rank * 8 + row) * D + part_pos(me.c)), dst_rank);
#pragma unroll
        for (int u = 0; u < DQ / 4; ++u)
          dsmem_st_f4(dst + 64u * u, make_float4(o[i][4 * u], o[i][4 * u + 1], o[i][4 * u + 2], o[i][4 * u + 3]));
      }
    }
  }
  ptx::cluster_sync();
  fold_chunk8<D, 0>(a, recv, s_rml, s_flag, sm, rank, c, n_tiles, n_chunks, b, g, qt, qn, G, r0);
}

// The chunk partials of attn_tc4_kernel's requests of several chunks, folded in
// chunk order (the arithmetic of fold_chunk8's last arriver), normalised and
// written: one CTA per (query tile, kv head, 8 rows), 16 threads a row, one
// memory round trip for up to 16 chunks.  With many chunks it costs less than an
// acquiring arrival at the end of every CTA and a long last one
// (launch_attention_split has the figures).
template <int D>
__global__ void __launch_bounds__(128) attn_fold_kernel(const __grid_constant__ AttnArgs a) {
  constexpr int DT = D / 16, U = 16;  // positions per thread, chunks in flight
  const int tid = threadIdx.x, fr = 8 * blockIdx.z + (tid >> 4), fd = DT * (tid & 15);
  const int G = a.nq / a.nkv, g = blockIdx.y;
  int b = 0, qt = blockIdx.x;
  for (;; ++b) {
    const int tiles = ((a.rm.start[b + 1] - a.rm.start[b]) * G + kQT - 1) / kQT;
    if (qt < tiles) break;
    qt -= tiles;
  }
  const int r0 = a.rm.start[b], M = a.rm.start[b + 1] - r0, qn = M * G;
  const size_t pc0 = ((size_t)(b * a.nkv + g) * a.qt_max + qt) * a.chunks_max;
  const float2* mlp = a.ws_ml + pc0 * kQT + fr;
  const float* op = a.ws_o + (pc0 * kQT + fr) * D + fd;
  ptx::griddep_launch_dependents();
  ptx::griddep_wait();
  const int L = a.len[b];
  const int n_tiles = rows_fit(L, M, a.cap) ? (L + M + kTile - 1) / kTile : 0;
  const int n_chunks = (n_tiles + kCluster - 1) / kCluster;
  if (n_chunks <= 1 || qt * kQT + fr >= qn) return;
  float cm = -INFINITY, cl = 0.f, co[DT];
#pragma unroll
  for (int i = 0; i < DT; ++i) co[i] = 0.f;
  for (int c = U; c < n_chunks; ++c) cm = fmaxf(cm, __ldcg(mlp + (size_t)c * kQT).x);
  for (int c0 = 0; c0 < n_chunks; c0 += U) {
    float2 ml[U];
    float4 v[U][DT / 4];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (c0 + u < n_chunks) {
        ml[u] = __ldcg(mlp + (size_t)(c0 + u) * kQT);
#pragma unroll
        for (int i = 0; i < DT / 4; ++i)
          v[u][i] = __ldcg(reinterpret_cast<const float4*>(op + (size_t)(c0 + u) * kQT * D) + i);
      }
    if (c0 == 0) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u < n_chunks) cm = fmaxf(cm, ml[u].x);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (c0 + u < n_chunks) {
        const float w = part_weight(ml[u].x, cm);
        if (w != 0.f) {
          cl += ml[u].y * w;
#pragma unroll
          for (int i = 0; i < DT / 4; ++i) {
            co[4 * i] += v[u][i].x * w;
            co[4 * i + 1] += v[u][i].y * w;
            co[4 * i + 2] += v[u][i].z * w;
            co[4 * i + 3] += v[u][i].w * w;
          }
        }
      }
  }
  write_rows<D, DT>(a, co, cl, fr, fd, qt, qn, G, g, r0);
}

// Clusters of 16 resident at once, two CTAs per SM: 14 in a residency probe
// (the occupancy calculator reports 7).
constexpr int kPairClusters = 14;

// How many clusters of 16 of the pair kernel the occupancy calculator allows
// (0 if none fits, or the launch attributes are refused); queried once per
// head size.
template <int D>
int pair_clusters_max() {
  static const int n = [] {
    constexpr uint32_t smem = attn_smem<false, true>();
    if (cudaFuncSetAttribute(attn_tc_kernel<D, false, true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(attn_tc_kernel<D, false, true>,
                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16 * 16, 1);
    cfg.blockDim = dim3(128);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, attn_tc_kernel<D, false, true>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      return 0;
    }
    return nc;
  }();
  return n;
}

template <int D, bool NARROW, bool PAIR>
cudaError_t launch_attn(const CUtensorMap& tk, const CUtensorMap& tv, const AttnArgs& a,
                        int clusters, cudaStream_t st) {
  constexpr uint32_t smem = attn_smem<NARROW, PAIR>();
  constexpr int CL = PAIR ? 2 * kCluster : kCluster;
  static const cudaError_t attr = cudaFuncSetAttribute(
      attn_tc_kernel<D, NARROW, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (attr != cudaSuccess) return attr;
  // clusters of 16 are beyond the portable size of 8
  static const cudaError_t attr16 =
      PAIR ? cudaFuncSetAttribute(attn_tc_kernel<D, NARROW, PAIR>,
                                  cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
           : cudaSuccess;
  if (attr16 != cudaSuccess) return attr16;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * CL, a.nkv);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr2[2];
  attr2[0].id = cudaLaunchAttributeClusterDimension;
  attr2[0].val.clusterDim.x = CL;
  attr2[0].val.clusterDim.y = 1;
  attr2[0].val.clusterDim.z = 1;
  attr2[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr2[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr2;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, attn_tc_kernel<D, NARROW, PAIR>, tk, tv, a);
}

template <int D>
cudaError_t launch_attn4(const CUtensorMap& tk, const CUtensorMap& tv, const AttnArgs& a,
                         int clusters, int q_tiles, bool fold, cudaStream_t st) {
  constexpr uint32_t smem = attn4_smem();
  static const cudaError_t attr = cudaFuncSetAttribute(
      attn_tc4_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (attr != cudaSuccess) return attr;
  const cudaError_t e = launch_pdl(attn_tc4_kernel<D>, dim3(clusters * kCluster, a.nkv), dim3(128), smem,
                                   st, kCluster, tk, tv, a);
  if (e != cudaSuccess || !fold) return e;
  return launch_pdl(attn_fold_kernel<D>, dim3(q_tiles, a.nkv, kQT / 8), dim3(128), 0, st, 1, a);
}

}  // namespace

int attn_q_tiles(int rows_per_request, int group) {
  return (rows_per_request * group + kQT - 1) / kQT;
}
int attn_chunks(int capacity) { return (capacity + kChunk - 1) / kChunk; }
size_t attn_qimg_bytes(int head_dim) { return (size_t)256 * head_dim; }

cudaError_t launch_attention_split(const RowMap& m, const Model& md, KvState& kv, int layer,
                                   cudaStream_t st) {
  const as2d_config& c = md.cfg;
  AttnArgs a;
  a.rm = m;
  a.len = kv.d_len;
  a.layer = layer;
  a.batch = kv.batch;
  a.cap = kv.capacity;
  a.nq = c.n_q_heads;
  a.nkv = c.n_kv_heads;
  a.qscale = 1.4426950408889634f / sqrtf((float)c.head_dim);
  a.qkv_part = kv.qkv_part;
  a.qkv_rinv = kv.qkv_rinv;
  a.rope = kv.rope;
  a.qkv_split = kv.qkv_split;
  a.qkv_ld = kv.rows_alloc;
  a.kc = kv.k_cache;
  a.vc = kv.v_cache;
  a.qimg = kv.qimg;
  a.qt_max = kv.attn_qt;
  a.ws_o = kv.attn_o;
  a.ws_ml = kv.attn_ml;
  a.chunks_max = kv.attn_chunks;
  a.cnt = kv.attn_cnt;
  a.ao = kv.ao;
  a.lo_row = kv.rows_alloc;
  a.err = kv.d_err;
  a.timeout_ns = kv.wait_ns;
  const int G = c.n_q_heads / c.n_kv_heads;
  int clusters8 = 0, max_nch = 0;
  for (int b = 0; b < kv.batch; ++b) {
    const int rows = m.start[b + 1] - m.start[b];
    const int64_t keys = kv.len_upper[b] + rows;
    int nch = (int)((keys + kChunk - 1) / kChunk);
    if (nch > kv.attn_chunks) nch = kv.attn_chunks;
    a.n_ch[b] = nch;
    if (nch > max_nch) max_nch = nch;
    clusters8 += attn_q_tiles(rows, G) * nch;
  }
  // The same arithmetic whichever way the launch runs; the layout decides
  // how many CTAs an SM holds and whether two chunks fold in one cluster.
  // Narrow: more than kWideClusters clusters of 8.  Pair: every request has
  // at most two chunks, and the clusters of 16 run at once.
  const bool narrow = clusters8 * c.n_kv_heads > kWideClusters;
  const bool quad = clusters8 * c.n_kv_heads > kNarrowClusters;
  // Passes, us, without / with the prefetch of V: 36 clusters of 8 on the 7B
  // 2877 / 2872, on the 1.5B 1509 / 1500; 60 (7B) 2972 / 2978; 128 3392 / 3400;
  // 144 3447 / 3460; 16 ragged requests (about 440) 6127 / 6180.
  a.v_prefetch = clusters8 * c.n_kv_heads <= 128;
  int clusters16 = 0;
  for (int b = 0; b < kv.batch; ++b)
    clusters16 += attn_q_tiles(m.start[b + 1] - m.start[b], G) * ((a.n_ch[b] + 1) / 2);
  const bool pair_fits =
      (c.head_dim == 128 ? pair_clusters_max<128>() : pair_clusters_max<64>()) > 0;
  const bool pair = !narrow && pair_fits && max_nch == 2 && clusters16 * c.n_kv_heads <= kPairClusters;
  const int halves = pair ? 2 : 1;
  a.cl_start[0] = 0;
  for (int b = 0; b < kv.batch; ++b)
    a.cl_start[b + 1] = a.cl_start[b] + attn_q_tiles(m.start[b + 1] - m.start[b], G) *
                                            ((a.n_ch[b] + halves - 1) / halves);
  const int clusters = a.cl_start[kv.batch];
  // a four-per-SM launch in which a request may have more than four chunks is
  // followed by the fold of its chunk partials.  Measured, the last arriver's
  // fold against the kernel, 7B, k = 16: requests of 3500 positions (4 chunks)
  // 3669 / 3700 us, 5500 (6) 3576 / 3518, 7500 (8) 3423 / 3390, 15128 (15) 3376 /
  // 3295; 64 requests of the 1.5B of up to two chunks 7213 / 7505.
  const bool fold = quad && max_nch > 4;
  a.fold_later = fold ? 1 : 0;
  int q_tiles = 0;
  for (int b = 0; b < kv.batch; ++b) q_tiles += attn_q_tiles(m.start[b + 1] - m.start[b], G);
  const dim3 gf(m.rows, (c.n_q_heads + 2 * c.n_kv_heads + 2 * kQkvWarps - 1) / (2 * kQkvWarps));
  const dim3 bf(32, kQkvWarps);
  cudaError_t e;
  kv.launches += fold ? 3 : 2;
  if (c.head_dim == 128) {
    e = launch_pdl(qkv_finish_kernel<128>, gf, bf, 0, st, 1, a);
    if (e == cudaSuccess)
      e = quad     ? launch_attn4<128>(kv.tm_kc, kv.tm_vc, a, clusters, q_tiles, fold, st)
          : narrow ? launch_attn<128, true, false>(kv.tm_kc, kv.tm_vc, a, clusters, st)
          : pair ? launch_attn<128, false, true>(kv.tm_kc, kv.tm_vc, a, clusters, st)
                 : launch_attn<128, false, false>(kv.tm_kc, kv.tm_vc, a, clusters, st);
  } else {
    e = launch_pdl(qkv_finish_kernel<64>, gf, bf, 0, st, 1, a);
    if (e == cudaSuccess)
      e = quad     ? launch_attn4<64>(kv.tm_kc, kv.tm_vc, a, clusters, q_tiles, fold, st)
          : narrow ? launch_attn<64, true, false>(kv.tm_kc, kv.tm_vc, a, clusters, st)
          : pair ? launch_attn<64, false, true>(kv.tm_kc, kv.tm_vc, a, clusters, st)
                 : launch_attn<64, false, false>(kv.tm_kc, kv.tm_vc, a, clusters, st);
  }
  return e;
}

}  // namespace as2d
