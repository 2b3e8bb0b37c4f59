// small_dev.cuh -- device functions of the embedding gather and the accept
// scan (k_basic.cu).
#pragma once

#include "as2d_internal.h"

namespace as2d {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;  // identical in every lane: each butterfly step is commutative
}

// Residual stream row r = the embedding row e; the first projection's operand
// h * g0 as bf16 hi + lo parts (lo rows start at ss_ld, the rows allocated);
// the row's sum of squares in tile slot 0 of ss (slots 1.. = 0).  Run by nthr
// threads (128 in every caller, which fixes the summation order); red holds
// nthr / 32 floats of shared memory; bar_id is the group's barrier.
__device__ __forceinline__ void embed_row_body(const bf16* __restrict__ e,
                                               const float* __restrict__ g0, int H, int r,
                                               int ss_ld, float* __restrict__ h,
                                               bf16* __restrict__ xn, float* __restrict__ ss,
                                               int tid, int nthr, float* red, int bar_id) {
  // Bound by the latency of the table row's load from HBM: up to kBatch columns
  // a thread are requested before the first is used, so that the 12 of the 1.5B
  // take one memory round trip and the 28 of the 7B two.  With 7 / 14 / 28 a
  // pass takes 1075 / 1069 / 1072 us (1.5B, k = 0), 1110 / 1108 / 1111 (k = 8),
  // 2613 / 2610 / 2608 (7B, k = 0), 2680 / 2681 / 2689 (k = 8).
  constexpr int kBatch = 14;
  float sq = 0.f;
  for (int c0 = tid; c0 < H; c0 += kBatch * nthr) {
    bf16 v[kBatch];
    float g[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      if (c0 + i * nthr < H) {
        v[i] = e[c0 + i * nthr];
        g[i] = g0[c0 + i * nthr];
      }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int c = c0 + i * nthr;
      if (c < H) {
        const float x = __bfloat162float(v[i]);
        h[(size_t)r * H + c] = x;
        const float xv = x * g[i];
        const bf16 xh = __float2bfloat16_rn(xv);
        xn[(size_t)r * H + c] = xh;
        xn[(size_t)(ss_ld + r) * H + c] = __float2bfloat16_rn(xv - __bfloat162float(xh));
        sq = fmaf(x, x, sq);
      }
    }
  }
  sq = warp_sum(sq);
  if ((tid & 31) == 0) red[tid >> 5] = sq;
  asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(nthr) : "memory");
  const int nt = H / 128;
  for (int t = tid; t < nt; t += nthr) {
    float tot = 0.f;
    if (t == 0)
      for (int w = 0; w < nthr / 32; ++w) tot += red[w];
    ss[(size_t)t * ss_ld + r] = tot;
  }
  asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(nthr) : "memory");
}

struct AcceptArgs {
  RowMap rm;
  const int32_t* cand;
  unsigned long long* best;
  int32_t* len;
  int32_t* root;
  int32_t* bad;
  int32_t* n_out;
  int32_t* corr_out;
  int32_t* greedy_out;
  int32_t mode;  // AcceptMode
  // kAcceptAll, nullable: whether an earlier pass of the prefill was kept (the
  // greedy token of a flagged pass is then the one after the last row kept)
  const int32_t* kept;
};

// Accept scan of request b by one warp (App. C.2): g_i from the packed maxima,
// the number of leading candidates equal to the greedy tokens by ballot, the
// correction by shuffle, then L += n + 1 and root = correction.
__device__ __forceinline__ void accept_request(const AcceptArgs& a, int b, int lane) {
  const RowMap& m = a.rm;
  const int r0 = m.start[b];
  const int k = m.start[b + 1] - r0 - 1;
  if (a.mode != kAcceptVerify) {
    // every row kept (prefill, up to kPrefillMaxRows rows): the maxima cleared
    // 32 rows at a time, the root is the greedy token after the last row (in
    // the pass that runs the LM head)
    int g_last = 0;
    for (int i = lane; i <= k; i += 32) {
      const unsigned long long v = a.best[r0 + i];
      const int g = (int)(0xFFFFFFFFu - (uint32_t)(v & 0xFFFFFFFFull));
      a.best[r0 + i] = 0ull;
      if (a.greedy_out) a.greedy_out[r0 + i] = g;
      if (i == k) g_last = g;
    }
    g_last = __shfl_sync(0xFFFFFFFFu, g_last, k & 31);
    if (lane == 0) {
      if (a.bad[b]) {
        a.n_out[b] = -1;
        a.corr_out[b] = -1;
        a.bad[b] = 0;
        if (a.kept && *a.kept) a.root[b] = g_last;
      } else {
        a.n_out[b] = k;
        a.len[b] += k + 1;
        if (a.mode == kAcceptAll) {
          a.corr_out[b] = g_last;
          a.root[b] = g_last;
        }
      }
    }
    return;
  }
  // every load before the first use: one memory round trip
  const unsigned long long v = lane <= k ? a.best[r0 + lane] : 0ull;
  const int cand = lane < k ? a.cand[r0 - b + lane] : -1;
  const int bad = a.bad[b], len = a.len[b];
  const int g = (int)(0xFFFFFFFFu - (uint32_t)(v & 0xFFFFFFFFull));
  if (lane <= k) {
    a.best[r0 + lane] = 0ull;
    if (a.greedy_out) a.greedy_out[r0 + lane] = g;
  }
  const bool match = (lane < k) && (cand == g);
  const unsigned mm = __ballot_sync(0xFFFFFFFFu, match);
  const int n = __ffs(~mm) - 1;  // bit k of mm is clear, so n <= k
  const int corr = __shfl_sync(0xFFFFFFFFu, g, n);
  if (lane == 0) {
    if (bad) {
      a.n_out[b] = -1;
      a.corr_out[b] = -1;
      a.bad[b] = 0;
    } else {
      a.n_out[b] = n;
      a.corr_out[b] = corr;
      a.len[b] = len + n + 1;
      a.root[b] = corr;
    }
  }
}

}  // namespace as2d
