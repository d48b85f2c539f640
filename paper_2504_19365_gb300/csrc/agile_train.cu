// Backward of the cache-backed embedding bag with a fused SGD step written into the
// cached pages (the differentiable extension of the Sec. 4.4 lookups).
//
// G[r, :] = sum over every index position i with idx[i] = r of gout[bag(i), :], added in
// increasing i (= increasing (bag, i)) in FP32, one accumulator per element starting at
// +0.  With lr != 0 every touched row becomes T[r, :] - (lr * G[r, :]) (product rounded
// first, no fused multiply-add) in its cache line, which turns MODIFIED; such lines reach
// the store through the queues when they are evicted or flushed (Sec. 3.4 case (d)).
//
// Grouping the positions by row in increasing position order: a stable radix sort of the
// keys (row << 32 | bag of the position) by row.  Rows that take part often (Zipf
// indices: the hottest row of an 82 k-position batch has 10 k positions) are summed by a
// light kernel of their own first; the engine sums the others and applies the step.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>

#include "agile.h"
#include "agile_ctx.cuh"
#include "agile_dev.cuh"

using namespace agile;

namespace {

constexpr int kMaxF4 = 8;  // dim <= 1024

// bag of every index position
__global__ void bag_of_kernel(const int64_t *off, uint32_t n_bags, int32_t *bag_of) {
  uint64_t w = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  unsigned l = threadIdx.x & 31;
  if (w >= n_bags) return;
  for (int64_t i = off[w] + l; i < off[w + 1]; i += 32) bag_of[i] = (int32_t)w;
}

// ---------------------------------------------------------------- stable radix sort by row
// Least significant digit first, at most 8 bits of the row a pass (as many passes as the
// table's row count needs, digits of equal width).  A pass is three launches: digit
// counts of every tile, one scan per digit over the tiles, and the scatter.  Within a
// tile a warp owns a contiguous run of keys and ranks 32 at a time with
// __match_any_sync, so equal digits keep their order: no key needs its position to be
// told apart, and the low word carries the bag instead.  Bound by launch latency at a
// training batch's size (three passes of ~2 us a launch): 81,920 positions of 2^18 rows
// take 25 us of kernels; the bitonic network it replaces took 153 launches, 263 us.
constexpr int kSortThreads = 256, kSortWarps = kSortThreads / 32;

struct SortIn {  // where a pass reads its keys: the caller's indices (first pass) or the last pass's output
  const int64_t *idx;
  const int32_t *bag_of;
  const uint64_t *keys;
  uint32_t rows;
  int32_t *err;
  __device__ __forceinline__ uint64_t load(uint64_t i, bool report) const {
    if (keys) return keys[i];
    int64_t r = idx[i];
    if (r < 0 || (uint64_t)r >= rows) {  // reported; summed as row 0
      if (report) atomicCAS(err, 0, 22);
      r = 0;
    }
    return ((uint64_t)r << 32) | (uint32_t)bag_of[i];
  }
};

template <int IPT>  // keys a thread
__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(SortIn in, uint64_t n, uint32_t shift, uint32_t digits,
                                                                  uint32_t *hist) {
  __shared__ uint32_t h[256];
  for (uint32_t d = threadIdx.x; d < digits; d += kSortThreads) h[d] = 0;
  __syncthreads();
  const uint64_t t0 = (uint64_t)blockIdx.x * kSortThreads * IPT;
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    uint64_t i = t0 + k * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(uint32_t)(in.load(i, true) >> shift) & (digits - 1)], 1u);
  }
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < digits; d += kSortThreads) hist[(uint64_t)d * gridDim.x + blockIdx.x] = h[d];
}

// exclusive scan of one digit's counts over the tiles (a CTA per digit), and its total
__global__ void __launch_bounds__(kSortThreads) sort_scan_kernel(uint32_t *hist, uint32_t tiles, uint32_t *total) {
  __shared__ uint32_t wsum[kSortWarps];
  uint32_t *row = hist + (uint64_t)blockIdx.x * tiles;
  const unsigned l = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0;
  for (uint32_t t0 = 0; t0 < tiles; t0 += kSortThreads) {
    uint32_t t = t0 + threadIdx.x;
    uint32_t v = t < tiles ? row[t] : 0, incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t u = __shfl_up_sync(kFull, incl, o);
      if (l >= (unsigned)o) incl += u;
    }
    if (l == 31) wsum[w] = incl;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < kSortWarps; ++k) {
      if (k < (int)w) before += wsum[k];
      all += wsum[k];
    }
    if (t < tiles) row[t] = carry + before + incl - v;
    carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

template <int IPT>
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(SortIn in, uint64_t n, uint32_t shift, uint32_t digits,
                                                                    const uint32_t *hist, const uint32_t *total,
                                                                    uint64_t *out) {
  __shared__ uint32_t cnt[kSortWarps][256];  // keys of each digit per warp, then where the warp's first one goes
  __shared__ uint32_t dsum[kSortWarps];
  const unsigned l = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t d = l; d < digits; d += 32) cnt[w][d] = 0;
  __syncwarp();
  const uint64_t t0 = ((uint64_t)blockIdx.x * kSortWarps + w) * 32 * IPT;
  uint64_t key[IPT];
  uint32_t rank[IPT];
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    uint64_t i = t0 + k * 32 + l;
    key[k] = i < n ? in.load(i, false) : 0;
  }
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    bool have = t0 + k * 32 + l < n;
    uint32_t dg = (uint32_t)(key[k] >> shift) & (digits - 1);
    unsigned m = __match_any_sync(kFull, have ? dg : 0xFFFFFFFFu);
    uint32_t before = have ? cnt[w][dg] : 0;
    rank[k] = before + __popc(m & ((1u << l) - 1));
    __syncwarp();
    if (have && (m >> l) == 1u) cnt[w][dg] = rank[k] + 1;  // the group's last lane
    __syncwarp();
  }
  __syncthreads();
  // first place of each digit: the totals of smaller digits, this tile's share of the
  // digit, the warps before
  {
    const uint32_t d = threadIdx.x;
    uint32_t v = d < digits ? total[d] : 0, incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t u = __shfl_up_sync(kFull, incl, o);
      if (l >= (unsigned)o) incl += u;
    }
    if (l == 31) dsum[w] = incl;
    __syncthreads();
    uint32_t at = incl - v;
#pragma unroll
    for (int k = 0; k < kSortWarps; ++k)
      if (k < (int)w) at += dsum[k];
    if (d < digits) {
      at += hist[(uint64_t)d * gridDim.x + blockIdx.x];
#pragma unroll
      for (int k = 0; k < kSortWarps; ++k) {
        uint32_t c = cnt[k][d];
        cnt[k][d] = at;
        at += c;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    if (t0 + k * 32 + l >= n) continue;
    uint32_t dg = (uint32_t)(key[k] >> shift) & (digits - 1);
    out[cnt[w][dg] + rank[k]] = key[k];
  }
}

// ---------------------------------------------------------------- rows of many positions
// A row with at least `span` positions (span = kLong positions, more for wide rows) is
// summed before the engine starts: a warp per (window of `span` sorted positions, 32
// columns).  At most one such row starts in a window, so its sum has a place of its own:
// G[window][dim].  The sum of a column is one chain of dependent adds, so what the split
// can hide is the loads: the warp stages its 128-byte pieces of 32 gradient rows at a time
// in shared memory with cp.async, three stages ahead of the adds (the keys one more), and
// a wide row is shared by dim / 32 warps.  The 10 k positions of the hottest row (2^18
// rows, Zipf 1.1, batch 4096 x 20) were 4.1 ms of serial load latency in one engine warp and
// take 119 us here; the bound that is left is the chain (4 cycles an add, 20 us).
constexpr uint32_t kLong = 64;
constexpr int kStages = 4, kLongWarps = 2;

__host__ __device__ __forceinline__ uint32_t long_span(uint32_t dim) { return dim / 4 > kLong ? dim / 4 : kLong; }

__device__ __forceinline__ bool starts_row(const uint64_t *keys, uint64_t j) {
  return j == 0 || (uint32_t)(keys[j] >> 32) != (uint32_t)(keys[j - 1] >> 32);
}
__device__ __forceinline__ bool is_long(const uint64_t *keys, uint64_t n, uint64_t j, uint32_t span) {
  return j + span <= n && (uint32_t)(keys[j + span - 1] >> 32) == (uint32_t)(keys[j] >> 32);
}

__global__ void __launch_bounds__(32 * kLongWarps) long_rows_kernel(const uint64_t *keys, uint64_t n, const float *gout,
                                                                    uint32_t dim, uint32_t span, uint32_t groups,
                                                                    float *G, float *grad_table) {
  __shared__ __align__(16) float stage[kLongWarps][kStages][32 * 32];
  const unsigned l = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t unit = (uint64_t)blockIdx.x * kLongWarps + w;
  const uint64_t win = unit / groups;
  const uint32_t col0 = (uint32_t)(unit % groups) * 32, wide = min(32u, dim - col0), nc = wide / 4;
  uint64_t j0 = ~0ull;
  for (uint32_t o = 0; o < span && j0 == ~0ull; o += 32) {
    uint64_t j = win * span + o + l;
    unsigned m = __ballot_sync(kFull, o + l < span && j < n && starts_row(keys, j) && is_long(keys, n, j, span));
    if (m) j0 = win * span + o + (__ffs(m) - 1);
  }
  if (j0 == ~0ull) return;
  const uint32_t r = (uint32_t)(keys[j0] >> 32);
  const uint32_t per = 32 / nc;  // rows one warp-wide copy brings
  // a batch is 32 positions; those of the row are a prefix of it (the keys are sorted).
  // Its keys are loaded one batch before they are looked at, so that no load is waited for
  // in the loop.
  auto keys_of = [&](uint64_t b) -> uint64_t {
    uint64_t j = j0 + 32 * b + l;
    return j < n ? keys[j] : ~((uint64_t)r << 32);  // past the end: another row
  };
  auto count = [&](uint64_t key) -> uint32_t { return __popc(__ballot_sync(kFull, (uint32_t)(key >> 32) == r)); };
  auto copy = [&](uint64_t b, uint32_t bag, uint32_t c) {
    float *s = stage[w][b % kStages];
    if (c == 32 && nc == 8) {  // a whole batch of 128-byte pieces: four rows a copy, no loop
      const float *src = gout + col0 + 4 * (l & 7);
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s + (l >> 3) * 32 + 4 * (l & 7));
      uint32_t bi[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) bi[t] = __shfl_sync(kFull, bag, 4 * t + (l >> 3));
#pragma unroll
      for (int t = 0; t < 8; ++t)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * t), "l"(src + (uint64_t)bi[t] * dim)
                     : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
      return;
    }
    for (uint32_t i0 = 0; i0 < c; i0 += per) {
      uint32_t i = i0 + l / nc;
      uint32_t bi = __shfl_sync(kFull, bag, i & 31);
      if (i < c) {
        const float *src = gout + (uint64_t)bi * dim + col0 + 4 * (l % nc);
        uint32_t dst = (uint32_t)__cvta_generic_to_shared(s + i * wide + 4 * (l % nc));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  uint32_t cnt[kStages];
  uint64_t key[kStages];
#pragma unroll
  for (int b = 0; b < kStages; ++b) key[b] = keys_of(b);
#pragma unroll
  for (int b = 0; b < kStages - 1; ++b) {
    cnt[b] = count(key[b]);
    copy(b, (uint32_t)key[b], cnt[b]);
  }
  uint64_t next = key[kStages - 1];
  float acc = 0.0f;
  for (uint64_t b0 = 0;; b0 += kStages) {
#pragma unroll
    for (int k = 0; k < kStages; ++k) {
      const uint64_t b = b0 + k;
      const int ahead = (k + kStages - 1) % kStages;
      // the stage being refilled was summed one batch ago
      const uint64_t now = next;
      next = keys_of(b + kStages);
      cnt[ahead] = count(now);
      copy(b + kStages - 1, (uint32_t)now, cnt[ahead]);
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
      __syncwarp();
      const float *s = stage[w][k] + (l < wide ? l : 0);
      if (cnt[k] == 32 && nc == 8) {
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = s[i * 32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc = __fadd_rn(acc, v[i]);
      } else {
        for (uint32_t i = 0; i < cnt[k]; ++i) acc = __fadd_rn(acc, s[i * wide]);
      }
      __syncwarp();
      if (cnt[k] < 32) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (l < wide) {
          if (G) G[win * dim + col0 + l] = acc;
          if (grad_table) grad_table[(uint64_t)r * dim + col0 + l] = acc;
        }
        return;
      }
    }
  }
}

// Sum of the gradient rows of the positions j0, j0 + 1, ... of row r, in that order: the
// bags of 32 positions are read at once, the rows of several in flight together.
template <int MF4>
__device__ __forceinline__ void sum_positions(const uint64_t *keys, uint64_t n, uint64_t j0, uint32_t r,
                                              const float *gout, uint32_t dim, float4 (&acc)[MF4]) {
  const unsigned l = lane_id();
  const uint32_t nf4 = dim / 4;
  constexpr int RB = MF4 >= 8 ? 1 : 8 / MF4;
#pragma unroll
  for (int k = 0; k < MF4; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (;; j0 += 32) {
    uint64_t j = j0 + l;
    uint64_t key = j < n ? keys[j] : ~0ull;
    const uint32_t c = __popc(__ballot_sync(kFull, j < n && (uint32_t)(key >> 32) == r));
    for (uint32_t i0 = 0; i0 < c; i0 += RB) {
      float4 v[RB][MF4];
#pragma unroll
      for (int ii = 0; ii < RB; ++ii) {
        const float4 *g = (const float4 *)(gout + (uint64_t)__shfl_sync(kFull, (uint32_t)key, (i0 + ii) & 31) * dim);
#pragma unroll
        for (int k = 0; k < MF4; ++k)
          v[ii][k] = i0 + ii < c && l + 32 * k < nf4 ? g[l + 32 * k] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int ii = 0; ii < RB; ++ii) {
        if (i0 + ii >= c) break;
#pragma unroll
        for (int k = 0; k < MF4; ++k) {
          acc[k].x = __fadd_rn(acc[k].x, v[ii][k].x);
          acc[k].y = __fadd_rn(acc[k].y, v[ii][k].y);
          acc[k].z = __fadd_rn(acc[k].z, v[ii][k].z);
          acc[k].w = __fadd_rn(acc[k].w, v[ii][k].w);
        }
      }
    }
    if (c < 32) return;
  }
}

template <int MF4>
__device__ __forceinline__ void store_row(float *grad_table, uint32_t r, uint32_t dim, const float4 (&acc)[MF4]) {
  float4 *o = (float4 *)(grad_table + (uint64_t)r * dim);
#pragma unroll
  for (int k = 0; k < MF4; ++k)
    if (lane_id() + 32 * k < dim / 4) o[lane_id() + 32 * k] = acc[k];
}

// The gradient table alone (lr = 0): the table's pages are not touched, so no engine is
// launched; a warp per 32 sorted positions sums the rows that start among them and are
// not long_rows_kernel's.
template <int MF4>
__global__ void __launch_bounds__(256) short_rows_kernel(const uint64_t *keys, uint64_t n, const float *gout, uint32_t dim,
                                                         uint32_t span, float *grad_table) {
  const uint64_t base = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * 32, j = base + lane_id();
  unsigned m = __ballot_sync(kFull, j < n && starts_row(keys, j) && !is_long(keys, n, j, span));
  for (; m; m &= m - 1) {
    const uint64_t j0 = base + (__ffs(m) - 1);
    const uint32_t r = (uint32_t)(keys[j0] >> 32);
    float4 acc[MF4];
    sum_positions<MF4>(keys, n, j0, r, gout, dim, acc);
    store_row<MF4>(grad_table, r, dim, acc);
  }
}

// The engine part (lr != 0): per distinct row (a segment of the sorted keys) the gradient
// row in fixed order, applied to the cached page and written out if asked for.  The rows
// of one page follow each other in the sorted keys: a warp pins the page once for all of
// those that start in its 32 positions.
//   SYNC : the row's page is requested when the warp gets to the row.
//   ASYNC: the pages of the rows of the warp's next 32 sorted positions are requested
//          before the rows of the current 32 are processed.
template <int MF4>
struct BackwardApp {
  uint64_t page0;
  uint32_t rows, dim;
  const uint64_t *keys;
  uint64_t n;
  const float *gout;
  const float *G;  // sums of the rows of many positions
  uint32_t span;
  float lr;
  float *grad_table;
  uint32_t mode;
  // no request ahead of need: the launch uses every queue pair for demand
  bool demand_only() const { return mode == AGILE_SYNC; }

  __device__ __forceinline__ uint32_t row_at(uint64_t j) const { return (uint32_t)(keys[j] >> 32); }

  __device__ bool prefetch(const Dev &d, const AppCtx &a, uint64_t base) const {
    uint64_t j = base + lane_id();
    bool head = j < n && starts_row(keys, j);
    uint64_t pg = head ? page0 + ((uint64_t)row_at(j) * dim * 4) / kPage : 0;
    return warp_request(d, head, pg, a.q0, false, a.deadline, nullptr, nullptr, nullptr, true, true);
  }

  __device__ void run(const Dev &d, const AppCtx &a) const {
    const unsigned l = lane_id();
    const uint32_t nf4 = dim / 4;
    const bool async = mode == AGILE_ASYNC;
    const uint64_t stride = (uint64_t)a.n_warps * 32;
    if (async && (uint64_t)a.warp * 32 < n && !prefetch(d, a, (uint64_t)a.warp * 32)) return;
    for (uint64_t base = (uint64_t)a.warp * 32; base < n; base += stride) {
      if (async && base + stride < n && !prefetch(d, a, base + stride)) return;
      const uint64_t j = base + l;
      const bool head = j < n && starts_row(keys, j);
      const uint32_t row = j < n ? row_at(j) : 0;
      const uint64_t page = page0 + ((uint64_t)row * dim * 4) / kPage;
      const unsigned longs = __ballot_sync(kFull, head && is_long(keys, n, j, span));
      unsigned m = __ballot_sync(kFull, head);
      while (m) {
        const uint64_t pg = __shfl_sync(kFull, page, __ffs(m) - 1);
        unsigned same = __ballot_sync(kFull, head && page == pg);
        m &= ~same;
        uint32_t line = 0;
        for (bool pinned = false; same; same &= same - 1) {
          const int t = __ffs(same) - 1;
          const uint32_t r = __shfl_sync(kFull, row, t);
          float4 acc[MF4];
          if ((longs >> t) & 1u) {
            const float4 *g = (const float4 *)(G + (base + t) / span * dim);
#pragma unroll
            for (int k = 0; k < MF4; ++k)
              acc[k] = l + 32 * k < nf4 ? g[l + 32 * k] : make_float4(0.f, 0.f, 0.f, 0.f);
          } else {
            sum_positions<MF4>(keys, n, base + t, r, gout, dim, acc);
            if (grad_table) store_row<MF4>(grad_table, r, dim, acc);
          }
          // the first wait for the page comes with nothing pinned
          if (!pinned && !warp_pin_page(d, pg, a.q0, a.deadline, line)) return;
          pinned = true;
          uint8_t *rowp = line_ptr(d, line) + ((uint64_t)r * dim * 4) % kPage;
#pragma unroll
          for (int k = 0; k < MF4; ++k) {
            uint32_t c = l + 32 * k;
            if (c < nf4) {
              float4 t4 = ld_cg_f4(rowp + 16 * c);
              t4.x = __fsub_rn(t4.x, __fmul_rn(lr, acc[k].x));
              t4.y = __fsub_rn(t4.y, __fmul_rn(lr, acc[k].y));
              t4.z = __fsub_rn(t4.z, __fmul_rn(lr, acc[k].z));
              t4.w = __fsub_rn(t4.w, __fmul_rn(lr, acc[k].w));
              st_cg16(rowp + 16 * c,
                      make_int4(__float_as_int(t4.x), __float_as_int(t4.y), __float_as_int(t4.z), __float_as_int(t4.w)));
            }
          }
        }
        __threadfence();
        __syncwarp();
        if (l == 0) {
          uint64_t old = atomicOr(&d.tag[line], 1ull);  // READY (2) -> MODIFIED (3)
          if (tag_state(old) == ST_READY) note_dirty(d, pg);
          cache_unpin(d, line);
        }
      }
    }
  }
};

}  // namespace

extern "C" {

int agile_embedding_bag_backward(agile_ctx *c, uint64_t table_byte0, uint32_t rows, uint32_t dim,
                                 const int64_t *d_idx, const int64_t *d_offsets, uint32_t n_bags,
                                 uint32_t n_indices, const float *d_grad_out, float lr, float *d_grad_table,
                                 uint32_t mode, void *stream) {
  if (!c || mode > 1) return AGILE_EINVAL;
  if (n_bags == 0 || n_indices == 0) return AGILE_OK;
  if (!d_idx || !d_offsets || !d_grad_out) return AGILE_EINVAL;
  if (dim == 0 || dim % 4 || dim * 4 > kPage || dim > 32 * 4 * kMaxF4 || kPage % (dim * 4)) return AGILE_EINVAL;
  if (table_byte0 % kPage || table_byte0 + (uint64_t)rows * dim * 4 > c->cfg.store_bytes) return AGILE_EINVAL;
  if (((uintptr_t)d_grad_out) & 15 || ((uintptr_t)d_grad_table) & 15) return AGILE_EINVAL;
  AGILE_CUDA_TRY(cudaSetDevice(c->device));
  cudaStream_t s = as_stream(stream);
  const uint64_t n = n_indices;
  // digits of the row number: equal widths of at most 8 bits
  uint32_t bits = 1;
  while (bits < 32 && (1ull << bits) < rows) ++bits;
  const uint32_t passes = (bits + 7) / 8, width = (bits + passes - 1) / passes, digits = 1u << width;
  // tiles of 1,024 keys while they are few (more CTAs in flight), else of 4,096 (fewer counts to scan)
  const uint32_t ipt = n <= (1u << 20) ? 4 : 16;
  const uint64_t tiles = (n + (uint64_t)kSortThreads * ipt - 1) / ((uint64_t)kSortThreads * ipt);
  const uint32_t span = long_span(dim);
  const uint64_t windows = (n + span - 1) / span;
  // scratch: keys before and after a pass, sums of the rows of many positions (16-byte
  // aligned: n is rounded up to a multiple of 4), counts, totals, bag of each position
  const uint64_t n2 = (n + 3) & ~3ull;
  const uint64_t g_floats = lr != 0.0f ? windows * dim : 0;
  size_t need = n2 * 16 + g_floats * 4 + (size_t)digits * tiles * 4 + 1024 + n2 * 4;
  if (c->train_scratch_bytes < need) {
    if (c->train_scratch) cudaFree(c->train_scratch);
    c->train_scratch = nullptr;
    c->train_scratch_bytes = 0;
    AGILE_CUDA_TRY(cudaMalloc(&c->train_scratch, need));
    c->train_scratch_bytes = need;
  }
  uint64_t *keys = (uint64_t *)c->train_scratch, *keys_out = keys + n2;
  float *G = (float *)(keys_out + n2);
  uint32_t *hist = (uint32_t *)(G + g_floats), *total = hist + (uint64_t)digits * tiles;
  int32_t *bag_of = (int32_t *)(total + 256);
  bag_of_kernel<<<(unsigned)((n_bags * 32ull + 255) / 256), 256, 0, s>>>(d_offsets, n_bags, bag_of);
  SortIn in{d_idx, bag_of, nullptr, rows, c->dev.err_sticky};
  for (uint32_t p = 0; p < passes; ++p) {
    const uint32_t shift = 32 + p * width;
    auto pass = [&](auto count, auto scatter) {
      count<<<(unsigned)tiles, kSortThreads, 0, s>>>(in, n, shift, digits, hist);
      sort_scan_kernel<<<digits, kSortThreads, 0, s>>>(hist, (uint32_t)tiles, total);
      scatter<<<(unsigned)tiles, kSortThreads, 0, s>>>(in, n, shift, digits, hist, total, keys_out);
    };
    if (ipt == 4) pass(sort_count_kernel<4>, sort_scatter_kernel<4>);
    else pass(sort_count_kernel<16>, sort_scatter_kernel<16>);
    in.keys = keys_out;
    std::swap(keys, keys_out);
  }
  AGILE_CUDA_TRY(cudaGetLastError());
  if (d_grad_table) AGILE_CUDA_TRY(cudaMemsetAsync(d_grad_table, 0, (size_t)rows * dim * 4, s));
  if (lr == 0.0f && !d_grad_table) return AGILE_OK;
  const uint32_t groups = (dim + 31) / 32;
  long_rows_kernel<<<(unsigned)((windows * groups + kLongWarps - 1) / kLongWarps), 32 * kLongWarps, 0, s>>>(
      keys, n, d_grad_out, dim, span, groups, lr != 0.0f ? G : nullptr, d_grad_table);
  AGILE_CUDA_TRY(cudaGetLastError());
  auto go = [&](auto app) {
    constexpr int MF4 = decltype(app)::value;
    if (lr == 0.0f) {
      short_rows_kernel<MF4><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(keys, n, d_grad_out, dim, span, d_grad_table);
      AGILE_CUDA_TRY(cudaGetLastError());
      return (int)AGILE_OK;
    }
    uint32_t warps = warps_for_cache(c, mode == AGILE_ASYNC ? 8 : 4, 32);
    BackwardApp<MF4> b{table_byte0 / kPage, rows, dim, keys, n, d_grad_out, G, span, lr, d_grad_table, mode};
    return launch_engine(c, b, stream, warps);
  };
  return dim <= 128 ? go(std::integral_constant<int, 1>{}) : go(std::integral_constant<int, kMaxF4>{});
}

}  // extern "C"
