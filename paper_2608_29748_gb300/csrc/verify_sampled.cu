// Stochastic verification of a draft block (speculative sampling) at
// temperature T with top-k / top-p filtering (Appendix "Evaluation Protocol":
// T = 1, top_p = 0.95, top_k = 20).  The paper keeps the underlying
// verification unchanged; the rule implemented is standard speculative
// sampling on the filtered distributions p (target) and q (drafter):
// accept x_i iff u_i q_i(x_i) < p_i(x_i); at the first rejection A draw the
// appended token from max(0, p_A - q_A) (renormalised; p_A if that is zero),
// else the bonus from p_K; draws are inverse-CDF in the filtered order.
//
// Only the top_k logits of a row enter its filtered distribution, so the
// row's full softmax is never formed:
//   sampled_topk_kernel      one CTA, or a cluster, per row (target rows, then
//                            drafter rows): one branch-free pass for maxima,
//                            from them a proven lower bound of the row's k-th
//                            largest, then the few elements above it, ranked;
//   sampled_finalize_kernel  one CTA per sequence: the filtered
//                            probabilities of the draft tokens from the sorted
//                            lists (16 positions at a time, one per warp),
//                            the accept tests in order, the draw, and for a
//                            round the copies and packing of e~ and [m; u].
// The outputs depend only on the target rows 0..A_b and the drafter rows
// 0..min(A_b, K-1).  In the windowed schedule the pair of kernels runs once
// per row window, over the sequences that accepted every earlier draft (live
// lists in the workspace); the copies and packing then follow in the greedy
// path's copy kernel.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cfloat>
#include <cstddef>

#include "common.cuh"
#include "internal.h"
#include "tc_pair.cuh"

namespace retrace {
namespace {

constexpr int kThreads = 512;
constexpr int kUnroll = 4;    // 16-byte loads in flight per thread
constexpr int kCells = 16;    // most cells per thread
constexpr int kBuf = 1024;    // candidates a CTA keeps without the slow path
constexpr int kTieThreads = 128;  // threads that reach the bound from which a row counts as tied there
constexpr int kMaxParts = 8;  // most CTAs (a cluster) per row
constexpr int kPrefetchVectors = 4096;  // 64 KB of the next row: two batches of every thread

struct TopkParams {
  const void* tlogits;
  long long t_row, t_batch;
  const void* dlogits;
  long long d_row, d_batch;
  int B, K, V, k;
  unsigned long long* keys;  // [B (2K+1), kMaxTopK]: target rows b*(K+1)+i, then drafter rows
  // Row window of this pass ([0, K+1) in one pass): target rows [i0, i1) and
  // drafter rows [i0, min(i1, K)) of the listed sequences (NULL: 0..B-1;
  // count_in NULL: B of them, else written by the previous pass).
  int i0, i1;
  const int32_t* live_in;
  const uint32_t* count_in;
  int parts;  // CTAs of a cluster, which share a row (or take a row each when there are many)
};

// One lane's 16 bytes of a row.
template <typename T>
struct Chunk;
template <>
struct Chunk<__nv_bfloat16> {
  static constexpr int E = 8;
  using Part = __nv_bfloat162;  // two running maxima
  uint4 w;
  __device__ Part part() const {
    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&w.x);
    const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&w.y);
    const __nv_bfloat162 c = *reinterpret_cast<const __nv_bfloat162*>(&w.z);
    const __nv_bfloat162 d = *reinterpret_cast<const __nv_bfloat162*>(&w.w);
    return __hmax2(__hmax2(a, b), __hmax2(c, d));
  }
  static __device__ Part combine(Part a, Part b) { return __hmax2(a, b); }
  static __device__ float finish(Part m) { return fmaxf(__low2float(m), __high2float(m)); }
  static __device__ Part lowest() { return __floats2bfloat162_rn(-INFINITY, -INFINITY); }
  __device__ float value(int e) const {
    const uint32_t x = e < 2 ? w.x : e < 4 ? w.y : e < 6 ? w.z : w.w;
    return (e & 1) ? bf16_hi(x) : bf16_lo(x);
  }
};
template <>
struct Chunk<float> {
  static constexpr int E = 4;
  using Part = float;
  uint4 w;
  __device__ Part part() const {
    return fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)), fmaxf(__uint_as_float(w.z), __uint_as_float(w.w)));
  }
  static __device__ Part combine(Part a, Part b) { return fmaxf(a, b); }
  static __device__ float finish(Part m) { return m; }
  static __device__ Part lowest() { return -INFINITY; }
  __device__ float value(int e) const { return __uint_as_float(e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w); }
};

// Shared memory of a top-k CTA.  The slow path and topk_tied use buf and cell
// together as one array of kSlowBuf keys.
struct TopkSmem {
  unsigned long long buf[kBuf];
  float cell[kCells][kThreads];
  unsigned long long top[kMaxTopK];  // this CTA's part of the row, in descending order
  float thr;
  int warp_n[kThreads / 32];
  int n;      // candidates in buf
  int n_top;  // keys in top
};
constexpr int kSlowBuf = kBuf + kCells * kThreads / 2;
static_assert(offsetof(TopkSmem, cell) == sizeof(unsigned long long) * kBuf, "the slow path's array is contiguous");
static_assert(kSlowBuf >= kBuf + kThreads * 8, "a slow-path round fits behind kBuf keys");

// Cells of the vectors [v0, v1): batches of kUnroll * kThreads per cell, and cells.
__device__ __forceinline__ int cell_batches(int v0, int v1) {
  const int batches = (v1 - v0 + kUnroll * kThreads - 1) / (kUnroll * kThreads);
  return (batches + kCells - 1) / kCells;
}
__device__ __forceinline__ int cell_count(int v0, int v1) {
  const int batches = (v1 - v0 + kUnroll * kThreads - 1) / (kUnroll * kThreads), per = cell_batches(v0, v1);
  return per > 0 ? (batches + per - 1) / per : 0;
}

// Moves the largest min(n, k) of `keys` (distinct) to `top` in descending
// order, by rank counting; returns their count.  Called by the whole CTA,
// after a barrier; ends before one.
__device__ __forceinline__ int rank_top(const unsigned long long* keys, int n, int k, unsigned long long* top) {
  for (int a = threadIdx.x; a < n; a += kThreads) {
    const unsigned long long x = keys[a];
    int rank = 0;
    for (int c = 0; c < n; ++c) rank += keys[c] > x ? 1 : 0;
    if (rank < k) top[rank] = x;
  }
  return n < k ? n : k;
}

// The k largest keys of row elements >= t when they are too many for buf: rounds
// of one vector per thread, the keys cut to the k largest whenever they pass kBuf.
// Fills sm.top; returns the count.
template <typename T>
__device__ __noinline__ int topk_slow(const T* x, int head, int v0, int v1, int edge_n, int full, float t, int k,
                                      TopkSmem& sm) {
  constexpr int E = Chunk<T>::E;
  unsigned long long* keys = sm.buf;
  if (threadIdx.x == 0) sm.n = 0;
  __syncthreads();
  unsigned long long least = 0ull;  // keys up to this one are not among the k largest
  auto add = [&](float v, int idx) {
    const unsigned long long key = make_key(v, (uint32_t)idx);
    if (v >= t && key > least) keys[atomicAdd(&sm.n, 1)] = key;
  };
  if ((int)threadIdx.x < edge_n) {
    const int i = (int)threadIdx.x < head ? (int)threadIdx.x : (int)threadIdx.x + full * E;
    add(to_f32(x[i]), i);
  }
  for (int b = v0;; b += kThreads) {
    const int v = b + (int)threadIdx.x;
    if (v < v1) {
      Chunk<T> c;
      c.w = __ldg(reinterpret_cast<const uint4*>(x + head) + v);
#pragma unroll
      for (int e = 0; e < E; ++e) add(c.value(e), head + v * E + e);
    }
    __syncthreads();
    const int n = sm.n;
    const bool done = b + kThreads >= v1;
    if (n > kBuf || done) {
      const int m = rank_top(keys, n, k, sm.top);
      __syncthreads();
      for (int a = threadIdx.x; a < m; a += kThreads) keys[a] = sm.top[a];
      if (threadIdx.x == 0) sm.n = m;
      least = m == k ? sm.top[k - 1] : 0ull;
      __syncthreads();
      if (done) return m;
    }
    __syncthreads();
  }
}

// The top-k keys of a part where many threads' maxima are the bound t itself: a
// row masked with a finite value that leaves fewer than k tokens, or coarse
// logits.  At most k - 1 threads hold anything larger, and of the elements equal
// to t the first by index are enough, which a scan in index order finds in its
// first rounds.  A verification of 1056 rows of 151936 bf16 masked so takes 109 us
// (where nothing ties 88; with every masked element a candidate for topk_slow
// 2585).  Nothing here is unrolled: with unrolled loops in this function the
// kernel's rows that never call it took 2 % longer.  Fills sm.top; returns the
// count.
template <typename T>
__device__ __noinline__ int topk_tied(const T* x, int head, int v0, int v1, int edge_n, int full, float t, int k,
                                      TopkSmem& sm) {
  using CT = Chunk<T>;
  constexpr int E = CT::E;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint4* vp = reinterpret_cast<const uint4*>(x + head);
  const int per = cell_batches(v0, v1), cells = cell_count(v0, v1);
  const int edge_i = tid < head ? tid : tid + full * E;
  float tm = tid < edge_n ? to_f32(x[edge_i]) : -INFINITY;  // this thread's maximum
  for (int j = 0; j < cells; ++j) tm = fmaxf(tm, sm.cell[j][tid]);
  if (tid == 0) sm.n = 0;
  __syncthreads();
  if constexpr (sizeof(T) == 4) {  // the bound's other 16 bits
    const unsigned h = ordered_bits(tm);
    unsigned b = ordered_bits(t) & 0xFFFF0000u;
#pragma unroll 1
    for (int bit = 15; bit >= 0; --bit) {
      const unsigned c = b | (1u << bit);
      if (__syncthreads_count(h >= c) >= k) b = c;
    }
    t = fmaxf(t, key_value((unsigned long long)b << 32));
  }
  // the elements > t
  auto above = [&](float v, int idx) {
    if (v > t) {
      const int at = atomicAdd(&sm.n, 1);
      if (at < kBuf) sm.buf[at] = make_key(v, (uint32_t)idx);
    }
  };
  if (tm > t) {
    if (tid < edge_n) above(to_f32(x[edge_i]), edge_i);
    for (int j = 0; j < cells; ++j) {
      if (!(sm.cell[j][tid] > t)) continue;
      for (int c = j * per; c < (j + 1) * per; ++c)
        for (int u = 0; u < kUnroll; ++u) {
          const int v = v0 + (c * kUnroll + u) * kThreads + tid;
          if (v >= v1) continue;
          CT ch;
          ch.w = __ldg(vp + v);
#pragma unroll 1
          for (int e = 0; e < E; ++e) above(ch.value(e), head + v * E + e);
        }
    }
  }
  __syncthreads();
  const int n_above = sm.n;
  __syncthreads();
  if (n_above > kBuf) return topk_slow<T>(x, head, v0, v1, edge_n, full, t, k, sm);
  // the elements equal to t in index order: before the vectors, the vectors, after them
  const int limit = max(n_above, k);
  int have = n_above;
  for (int b = v0 - kThreads; have < limit; b += kThreads) {
    unsigned equal = 0u;
    int idx = 0;
    if (b < v0) {
      if (edge_n > 0 && tid < head) {
        idx = tid;
        equal = to_f32(x[idx]) == t ? 1u : 0u;
      }
    } else if (b < v1) {
      const int v = b + tid;
      if (v < v1) {
        CT ch;
        ch.w = __ldg(vp + v);
        idx = head + v * E;
#pragma unroll 1
        for (int e = 0; e < E; ++e) equal |= ch.value(e) == t ? 1u << e : 0u;
      }
    } else if (tid < edge_n - head) {
      idx = head + full * E + tid;
      equal = to_f32(x[idx]) == t ? 1u : 0u;
    }
    const int count = __popc(equal);
    int incl = count;
#pragma unroll 1
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += y;
    }
    if (lane == 31) sm.warp_n[warp] = incl;
    __syncthreads();
    int at = have + incl - count;
#pragma unroll 1
    for (int w = 0; w < kThreads / 32; ++w) {
      const int n = sm.warp_n[w];
      at += w < warp ? n : 0;
      have += n;
    }
    for (; equal != 0u && at < limit; equal &= equal - 1u, ++at)
      sm.buf[at] = make_key(t, (uint32_t)(idx + __ffs((int)equal) - 1));
    __syncthreads();
    if (b >= v1) break;
  }
  return rank_top(sm.buf, min(have, limit), k, sm.top);
}

// The top-k keys of part `part` of `parts` of row x, into sm.top (whole CTA).
// Elements at -infinity carry no weight and get no key.
//
// Every thread streams its vectors once and keeps only maxima: one per cell
// (a few batches of kUnroll vectors) in shared memory and one overall.  The
// k-th largest of the threads' maxima is a lower bound t of the part's k-th
// largest element (each is an element), and a close one: with 512 threads and
// k = 20 a part has about 21 elements above it.  With several parts the
// largest of their bounds serves all.  Then the few threads whose maxima
// reach t reload the cells that do, and their elements >= t are ranked.  The
// stream itself has no branch on the data; a scan that compared each vector
// with a bound sampled from the row's start spent most of its time on the
// vectors that passed it (one pass over 1056 rows of 151936 bf16: 84 us, now
// 74).
template <typename T>
__device__ __forceinline__ void topk_part(const T* x, int V, int k, int parts, int part, TopkSmem& sm) {
  using CT = Chunk<T>;
  constexpr int E = CT::E;
  const int tid = threadIdx.x;
  const int head = min(V, (int)((16u - (uint32_t)((uintptr_t)x & 15u)) & 15u) / (int)sizeof(T));
  const int full = (V - head) / E;  // aligned vectors inside the row
  const int v0 = (int)((long long)part * full / parts), v1 = (int)((long long)(part + 1) * full / parts);
  // the elements before and after the vectors (fewer than 2 E), one per thread of part 0
  const int edge_n = part == 0 ? V - full * E : 0;
  const int per = cell_batches(v0, v1), cells = cell_count(v0, v1);
  const int edge_i = tid < head ? tid : tid + full * E;
  const uint4* vp = reinterpret_cast<const uint4*>(x + head);
  if (tid == 0) sm.n = 0;
  float edge_v = -INFINITY;
  if (tid < edge_n) edge_v = to_f32(x[edge_i]);
  float tm = edge_v;
  for (int j = 0; j < cells; ++j) {
    typename CT::Part m = CT::lowest();
    for (int c = j * per; c < (j + 1) * per; ++c) {
      const int b = v0 + c * kUnroll * kThreads + tid;
      CT ch[kUnroll];
      if (b + (kUnroll - 1) * kThreads < v1) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) ch[u].w = __ldcs(vp + b + u * kThreads);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) m = CT::combine(m, ch[u].part());
      } else {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          if (b + u * kThreads < v1) {
            ch[u].w = __ldcs(vp + b + u * kThreads);
            m = CT::combine(m, ch[u].part());
          }
        }
      }
    }
    const float mv = CT::finish(m);
    sm.cell[j][tid] = mv;
    tm = fmaxf(tm, mv);
  }
  // t: the largest value of 16 leading key bits that at least k threads'
  // maxima reach (all bits of a bf16 value; an fp32 bound is rounded down)
  const unsigned h = ordered_bits(tm) >> 16;
  unsigned lo = 0u;
#pragma unroll 1
  for (int bit = 15; bit >= 0; --bit) {
    const unsigned c = lo | (1u << bit);
    if (__syncthreads_count(h >= c) >= k) lo = c;
  }
  const unsigned minus_inf = ordered_bits(-INFINITY) >> 16;
  // (a negative value's key has its low bits set)
  const unsigned low = sizeof(T) == 2 && !(lo & 0x8000u) ? 0xFFFFu : 0u;
  float t = lo <= minus_inf ? -FLT_MAX : key_value((unsigned long long)(lo << 16 | low) << 32);
  if (parts > 1) {
    if (tid == 0) sm.thr = t;
    cluster_sync_all();
    for (int q = 0; q < parts; ++q) t = fmaxf(t, ld_cluster_f1(map_rank(smem_u32(&sm.thr), (uint32_t)q)));
  }
  // the elements >= t
  auto add = [&](float v, int idx) {
    if (v >= t) {
      const int at = atomicAdd(&sm.n, 1);
      if (at < kBuf) sm.buf[at] = make_key(v, (uint32_t)idx);
    }
  };
  if (__syncthreads_count(h >= lo) > kTieThreads && lo > minus_inf) {
    sm.n = kBuf + 1;  // for topk_tied
  } else if (tm >= t) {
    if (tid < edge_n) add(edge_v, edge_i);
    for (int j = 0; j < cells; ++j) {
      if (!(sm.cell[j][tid] >= t)) continue;
      for (int c = j * per; c < (j + 1) * per; ++c) {
        const int b = v0 + c * kUnroll * kThreads + tid;
        CT ch[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
          if (b + u * kThreads < v1) ch[u].w = __ldg(vp + b + u * kThreads);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
          if (b + u * kThreads < v1) {
            const int v = b + u * kThreads;
#pragma unroll
            for (int e = 0; e < E; ++e) add(ch[u].value(e), head + v * E + e);
          }
      }
    }
  }
  __syncthreads();
  int n = sm.n;
  __syncthreads();  // topk_tied reuses sm.n
  if (n > kBuf) n = topk_tied<T>(x, head, v0, v1, edge_n, full, t, k, sm);
  else n = rank_top(sm.buf, n, k, sm.top);
  if (tid == 0) sm.n_top = n;
  __syncthreads();
}

// Clusters of p.parts CTAs.  The rows of a pass: the window's target rows of
// each listed sequence, then its drafter rows (`row` is the row's slot in
// p.keys).  A cluster takes one row, each CTA a part of it, and CTA 0 merges
// the parts; when a pass has more rows than clusters, each CTA takes whole rows
// instead (rounds, V = 151936, d = 2560, of which a later pass has 192 / 228 / 432
// rows for 114 clusters of four: 173 / 193 / 185 us, with up to two rows per
// cluster 183 / 224 / 192, with up to four 182 / 222 / 236).  The live count of a later pass is known on the device
// only, so its grid is resident CTAs that loop over the rows (LOOP; in the first
// pass a CTA per row, which measured 158 us per round of 32 sequences, was
// faster than resident ones, 165).
template <typename T, bool LOOP>
__global__ void __launch_bounds__(kThreads, 3) sampled_topk_kernel(const TopkParams p) {
  __shared__ TopkSmem sm;
  pdl_launch_dependents();  // the finalize kernel may take SMs as these CTAs finish
  int n_live = p.B;
  if (p.count_in) {  // a later pass: the previous finalize wrote the live list
    pdl_wait();
    n_live = (int)__ldcg(p.count_in);
  }
  const int wt = p.i1 - p.i0, wd = min(p.i1, p.K) - p.i0;
  const int rows = n_live * (wt + wd);  // B (2K+1) at most, below 2^31
  const int parts = rows > (int)gridDim.x / p.parts ? 1 : p.parts;
  const int part = parts > 1 ? (int)cluster_rank() : 0;
  const int step = (int)gridDim.x / parts;
  auto row_of = [&](int r0, const T*& x) -> int {
    if (r0 < n_live * wt) {
      const int l = r0 / wt, i = p.i0 + (r0 - l * wt);
      const int b = p.live_in ? __ldg(p.live_in + l) : l;
      x = reinterpret_cast<const T*>(p.tlogits) + b * p.t_batch + i * p.t_row;
      return b * (p.K + 1) + i;
    }
    const int r = r0 - n_live * wt, l = r / wd, i = p.i0 + (r - l * wd);
    const int b = p.live_in ? __ldg(p.live_in + l) : l;
    x = reinterpret_cast<const T*>(p.dlogits) + b * p.d_batch + i * p.d_row;
    return p.B * (p.K + 1) + b * p.K + i;
  };
  for (int r0 = (int)blockIdx.x / parts; r0 < rows; r0 += step) {
    const T* x;
    if (LOOP && threadIdx.x == 0 && r0 + step < rows) {
      // the stream pauses between rows: the first vectors of this CTA's next
      // part (inside the row, 16-byte aligned) go to L2 meanwhile
      row_of(r0 + step, x);
      const int h = min(p.V, (int)((16u - (uint32_t)((uintptr_t)x & 15u)) & 15u) / (int)sizeof(T));
      const int full = (p.V - h) / Chunk<T>::E;
      const int v0 = (int)((long long)part * full / parts), v1 = (int)((long long)(part + 1) * full / parts);
      const int nv = min(v1 - v0, kPrefetchVectors);
      if (nv > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<const uint4*>(x + h) + v0),
                     "r"(nv * 16)
                     : "memory");
    }
    const int row = row_of(r0, x);
    topk_part<T>(x, p.V, p.k, parts, part, sm);
    unsigned long long* out = p.keys + (long long)row * kMaxTopK;
    if (parts == 1) {
      for (int r = threadIdx.x; r < p.k; r += kThreads) out[r] = r < sm.n_top ? sm.top[r] : 0ull;
      __syncthreads();  // sm is read to the end before the next row
    } else {
      cluster_sync_all();  // every part's list is complete
      if (part == 0) {
        // thread 64 q + r has key r of part q (kMaxParts * kMaxTopK = kThreads)
        const int q = (int)threadIdx.x / kMaxTopK, r = (int)threadIdx.x % kMaxTopK;
        int before = 0, total = 0, mine = 0;
#pragma unroll
        for (int c = 0; c < kMaxParts; ++c) {
          const int n = c < parts ? ld_cluster_s32(map_rank(smem_u32(&sm.n_top), (uint32_t)c)) : 0;
          before += c < q ? n : 0;
          mine = c == q ? n : mine;
          total += n;
        }
        if (r < mine) sm.buf[before + r] = ld_cluster_u64(map_rank(smem_u32(&sm.top[r]), (uint32_t)q));
        __syncthreads();
        const int n = rank_top(sm.buf, total, p.k, out);
        for (int r2 = n + (int)threadIdx.x; r2 < p.k; r2 += kThreads) out[r2] = 0ull;
      }
      cluster_sync_all();  // CTA 0 has read the parts' lists
    }
    if constexpr (!LOOP) break;
  }
}

constexpr int kFinWarps = 16;  // warps of a finalize CTA: positions whose accept tests run together

struct FinalizeParams {
  const unsigned long long* keys;
  int B, K, V, k;
  float inv_T, top_p;
  const int32_t* draft;
  const float* uniforms;
  int32_t* accept_len;
  int32_t* committed;
  int32_t* bonus;
  // a whole round (optional): n, copies of the unconditioned rows of e~, and
  // the packed [m; u] rows of the tensor-core projections
  int32_t* n_out;
  const void* e;
  long long e_batch_stride, e_pos_stride;
  void* e_out;
  int d, elem;
  const void* hD;
  const void* hT;
  int e_dense;
  void* apack;
  void* epack;
  int32_t* rowmap;
  int32_t* R_count;
  // Windowed schedule: accept tests over rows [i0, min(i1, K)) of the listed
  // sequences (live_in NULL: 0..B-1, count_in NULL: B); a sequence that
  // accepts them all, with rows left, goes to live_out.  The last pass's last
  // CTA out zeroes the passes' counters.  With defer_copies the finaliser
  // only claims the packed rows (pack_off) and a later kernel copies.
  int i0, i1;
  const int32_t* live_in;
  const uint32_t* count_in;
  int32_t* live_out;
  uint32_t* count_out;
  uint32_t* pass_counts;
  int n_counts;
  uint32_t* exits;
  int defer_copies;
  int32_t* pack_off;
};

// The filtered distribution of one row, lane j holding entries j and 32 + j
// of the sorted list: weight (0 beyond the top-p cut) and token (-1 if none).
struct RowDist {
  float w[2];
  int tok[2];
  float total;  // sum of the kept weights
};

__device__ RowDist row_dist(const FinalizeParams& p, long long row, int lane) {
  const unsigned FULL = 0xFFFFFFFFu;
  const unsigned long long* keys = p.keys + row * kMaxTopK;
  RowDist r;
  const float v0 = key_value(keys[0]);
  float w[2];
  int tok[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = 32 * h + lane;
    const unsigned long long key = j < p.k ? keys[j] : 0ull;
    tok[h] = key ? (int)key_index(key) : -1;
    w[h] = key ? expf((key_value(key) - v0) * p.inv_T) : 0.f;
  }
  // softmax over the top k, then the shortest prefix reaching top_p
  float z = w[0] + w[1];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(FULL, z, off);
  float c0 = w[0];  // inclusive prefix over entries 0..31
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(FULL, c0, off);
    if (lane >= off) c0 += t;
  }
  const float s0 = __shfl_sync(FULL, c0, 31);
  float c1 = w[1];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(FULL, c1, off);
    if (lane >= off) c1 += t;
  }
  c1 += s0;
  // entry j is kept iff the prefix before it is below top_p
  const float before0 = c0 - w[0], before1 = c1 - w[1];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float before = h == 0 ? before0 : before1;
    const bool keep = tok[h] >= 0 && before < p.top_p * z;
    r.w[h] = keep ? w[h] : 0.f;
    r.tok[h] = keep ? tok[h] : -1;
  }
  float t = r.w[0] + r.w[1];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(FULL, t, off);
  r.total = t;
  return r;
}

// Probability of token y under the row distribution (same value on every lane).
__device__ float dist_prob(const RowDist& r, int y) {
  const unsigned FULL = 0xFFFFFFFFu;
  float w = (r.tok[0] == y ? r.w[0] : 0.f) + (r.tok[1] == y ? r.w[1] : 0.f);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(FULL, w, off);
  return w / r.total;
}

// Inverse-CDF draw over entries in list order with weights wt (this lane's
// two entries): the first entry whose inclusive cumulative weight exceeds
// u * total; the last kept entry if rounding leaves none.
__device__ int draw(const RowDist& r, const float wt[2], float u, int lane) {
  const unsigned FULL = 0xFFFFFFFFu;
  float c0 = wt[0];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(FULL, c0, off);
    if (lane >= off) c0 += t;
  }
  const float s0 = __shfl_sync(FULL, c0, 31);
  float c1 = wt[1];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float t = __shfl_up_sync(FULL, c1, off);
    if (lane >= off) c1 += t;
  }
  c1 += s0;
  const float total = __shfl_sync(FULL, c1, 31);
  const float target = u * total;
  const unsigned b0 = __ballot_sync(FULL, wt[0] > 0.f && c0 > target);
  const unsigned b1 = __ballot_sync(FULL, wt[1] > 0.f && c1 > target);
  int src, h;
  if (b0) {
    src = __ffs(b0) - 1;
    h = 0;
  } else if (b1) {
    src = __ffs(b1) - 1;
    h = 1;
  } else {  // last entry with weight
    const unsigned l0 = __ballot_sync(FULL, wt[0] > 0.f), l1 = __ballot_sync(FULL, wt[1] > 0.f);
    if (l1) {
      src = 31 - __clz(l1);
      h = 1;
    } else {
      src = 31 - __clz(l0);
      h = 0;
    }
  }
  const int t0 = __shfl_sync(FULL, r.tok[0], src), t1 = __shfl_sync(FULL, r.tok[1], src);
  return h == 0 ? t0 : t1;
}

// One CTA per sequence.  The accept tests need only p_i(x_i) and q_i(x_i):
// the warps compute them for kFinWarps positions at a time, one position each,
// and thread 0 takes the decisions in order, so the chain of dependent
// distributions is one per chunk instead of one per position.  Warp 0 then
// draws the appended token; every thread writes the outputs and, for a round,
// copies and packs rows.
__device__ void sampled_finalize_sequence(const FinalizeParams& p, int b) {
  __shared__ int s_A, s_y, s_off;
  __shared__ int s_qtok[kMaxTopK];
  __shared__ float s_qw[kMaxTopK];
  __shared__ float s_px[kFinWarps], s_qx[kFinWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int K = p.K, K1 = K + 1;
  const int32_t* dr = p.draft + (long long)b * K;
  const long long tbase = (long long)b * K1, dbase = (long long)p.B * K1 + (long long)b * K;
  const float* u = p.uniforms + (long long)b * K1;
  // rows before i0 were accepted in earlier passes
  int A = p.i1 == K1 ? K : -1;  // -1: every row of the window accepted, rows left
  const int hi = min(p.i1, K);
  for (int c0 = p.i0; c0 < hi; c0 += kFinWarps) {
    const int i = c0 + warp;
    if (i < hi) {
      const int x = dr[i];
      float px = -1.f, qx = 0.f;  // px < 0: a token outside [0, V) is rejected
      if (x >= 0 && x < p.V) {
        const RowDist pt = row_dist(p, tbase + i, lane);
        const RowDist qd = row_dist(p, dbase + i, lane);
        px = dist_prob(pt, x);
        qx = dist_prob(qd, x);
      }
      if (lane == 0) {
        s_px[warp] = px;
        s_qx[warp] = qx;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int a = -1;
      for (int j = 0; j < kFinWarps && c0 + j < hi; ++j) {
        if (!(s_px[j] >= 0.f && u[c0 + j] * s_qx[j] < s_px[j])) {
          a = c0 + j;
          break;
        }
      }
      s_A = a;
    }
    __syncthreads();
    const int a = s_A;
    if (a >= 0) {
      A = a;
      break;
    }
  }
  if (A < 0) {  // every draft of the window accepted: on to the next pass
    if (threadIdx.x == 0) p.live_out[atomicAdd(p.count_out, 1u)] = b;
    return;
  }
  if (warp == 0) {
    const RowDist pt = row_dist(p, tbase + A, lane);
    int y;
    if (A < K) {
      // residual max(0, p - q) over the target's kept tokens
      const RowDist qd = row_dist(p, dbase + A, lane);
      // (the drafter's list in shared memory: 64 entries handed round by
      // shuffles took longer than the two distributions)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        s_qtok[32 * h + lane] = qd.tok[h];
        s_qw[32 * h + lane] = qd.w[h];
      }
      __syncwarp();
      float qw[2] = {0.f, 0.f}, res[2];
      for (int t = 0; t < p.k; ++t) {
        const int tok = s_qtok[t];  // -1: cut off by top-p
        const float w = s_qw[t];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (tok >= 0 && tok == pt.tok[h]) qw[h] = w;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) res[h] = pt.tok[h] >= 0 ? fmaxf(0.f, pt.w[h] / pt.total - qw[h] / qd.total) : 0.f;
      float rs = res[0] + res[1];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) rs += __shfl_xor_sync(0xFFFFFFFFu, rs, off);
      y = rs > 0.f ? draw(pt, res, u[K], lane) : draw(pt, pt.w, u[K], lane);
    } else {
      y = draw(pt, pt.w, u[K], lane);
    }
    if (lane == 0) {
      s_y = y;
      const int nb = K - 1 - A > 0 ? K - 1 - A : 0;
      s_off = (p.R_count && nb > 0) ? atomicAdd(p.R_count, nb) : 0;
      if (p.defer_copies && p.R_count) p.pack_off[b] = s_off;
    }
  }
  __syncthreads();
  const int y = s_y;
  for (int i = threadIdx.x; i < K1; i += blockDim.x) {
    const long long o = (long long)b * K1 + i;
    p.committed[o] = i < A ? dr[i] : (i == A ? y : -1);
  }
  const int nb = K - 1 - A > 0 ? K - 1 - A : 0;
  if (threadIdx.x == 0) {
    p.accept_len[b] = A;
    p.bonus[b] = y;
    if (p.n_out) p.n_out[b] = nb;
  }
  if (!p.e_out || p.defer_copies) return;
  // rows j >= n_b keep the drafter input, bit for bit
  const long long base_row = (long long)b * K;
  const char* e_b = static_cast<const char*>(p.e) + b * p.e_batch_stride * p.elem;
  const long long rows = K - nb;
  const bool vec = (p.d * p.elem) % 16 == 0 && (uintptr_t)e_b % 16 == 0 && (uintptr_t)p.e_out % 16 == 0 &&
                   (p.e_pos_stride * p.elem) % 16 == 0;
  if (vec) {
    const int vpr = p.d * p.elem / 16;
    const long long pos_vec = p.e_pos_stride * p.elem / 16;
    const uint4* src = reinterpret_cast<const uint4*>(e_b);
    uint4* dst = reinterpret_cast<uint4*>(p.e_out) + (base_row + nb) * vpr;
    copy_vectors(rows * vpr, [&](long long i) { return __ldg(src + (nb + i / vpr) * pos_vec + i % vpr); },
                 [&](long long i, const uint4& v) { dst[i] = v; });
  } else if (p.elem == 2) {
    const uint16_t* src = reinterpret_cast<const uint16_t*>(e_b);
    uint16_t* dst = reinterpret_cast<uint16_t*>(p.e_out) + (base_row + nb) * p.d;
    for (long long i = threadIdx.x; i < rows * p.d; i += blockDim.x) {
      const long long j = nb + i / p.d, c = i % p.d;
      dst[i] = src[j * p.e_pos_stride + c];
    }
  } else {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(e_b);
    uint32_t* dst = reinterpret_cast<uint32_t*>(p.e_out) + (base_row + nb) * p.d;
    for (long long i = threadIdx.x; i < rows * p.d; i += blockDim.x) {
      const long long j = nb + i / p.d, c = i % p.d;
      dst[i] = src[j * p.e_pos_stride + c];
    }
  }
  if (!p.R_count || nb == 0) return;
  // packed rows [m_j; u_j] = [hD[b, A+1+j]; hT[b, A+j]] (Eq. 4-5), and e[b, j]
  // for a per-position e; the tensor-core path is bf16 with 16-byte rows
  const int off = s_off;
  const int vpr = p.d / 8;
  const uint4* e_v = reinterpret_cast<const uint4*>(e_b);
  const long long pos_vec = p.e_pos_stride / 8;
  for (int j = threadIdx.x; j < nb; j += blockDim.x) p.rowmap[off + j] = b * K + j;
  const uint4* hD = reinterpret_cast<const uint4*>(p.hD);
  const uint4* hT = reinterpret_cast<const uint4*>(p.hT);
  uint4* ap = reinterpret_cast<uint4*>(p.apack);
  copy_vectors(
      (long long)nb * 2 * vpr,
      [&](long long i) {
        const long long j = i / (2 * vpr), c = i % (2 * vpr);
        return c < vpr ? __ldg(hD + (base_row + A + 1 + j) * vpr + c) : __ldg(hT + (base_row + A + j) * vpr + c - vpr);
      },
      [&](long long i, const uint4& v) { ap[(long long)off * 2 * vpr + i] = v; });
  if (p.e_dense) {
    uint4* ep = reinterpret_cast<uint4*>(p.epack);
    copy_vectors((long long)nb * vpr, [&](long long i) { return __ldg(e_v + (i / vpr) * pos_vec + i % vpr); },
                 [&](long long i, const uint4& v) { ep[(long long)off * vpr + i] = v; });
  }
}

__global__ void __launch_bounds__(32 * kFinWarps) sampled_finalize_kernel(const FinalizeParams p) {
  pdl_launch_dependents();
  pdl_wait();  // the sorted lists come from the top-k kernel
  const int n_live = p.count_in ? (int)__ldcg(p.count_in) : p.B;
  if ((int)blockIdx.x < n_live) {
    sampled_finalize_sequence(p, p.live_in ? __ldg(p.live_in + blockIdx.x) : (int)blockIdx.x);
  }
  if (p.exits && threadIdx.x == 0) {  // the last pass's last CTA out resets the live counters
    __threadfence();
    if (atomicAdd(p.exits, 1u) == gridDim.x - 1u) {
      for (int k = 0; k < p.n_counts; ++k) p.pass_counts[k] = 0u;
      *p.exits = 0u;
    }
  }
}

}  // namespace

cudaError_t launch_verify_sampled(const SampledArgs& a, retrace_dtype dtype, cudaStream_t stream) {
  if (a.B <= 0) return cudaSuccess;
  TopkParams tp{};
  tp.tlogits = a.tlogits;
  tp.t_row = a.t_row;
  tp.t_batch = a.t_batch;
  tp.dlogits = a.dlogits;
  tp.d_row = a.d_row;
  tp.d_batch = a.d_batch;
  tp.B = a.B;
  tp.K = a.K;
  tp.V = a.V;
  tp.k = a.top_k;
  tp.keys = a.keys;
  FinalizeParams fp{};
  fp.keys = a.keys;
  fp.B = a.B;
  fp.K = a.K;
  fp.V = a.V;
  fp.k = a.top_k;
  fp.inv_T = 1.f / a.temperature;
  fp.top_p = a.top_p;
  fp.draft = a.draft;
  fp.uniforms = a.uniforms;
  fp.accept_len = a.accept_len;
  fp.committed = a.committed;
  fp.bonus = a.bonus;
  fp.n_out = a.n_out;
  fp.e = a.e;
  fp.e_batch_stride = a.e_batch_stride;
  fp.e_pos_stride = a.e_pos_stride;
  fp.e_out = a.e_out;
  fp.d = a.d;
  fp.elem = dtype == RETRACE_BF16 ? 2 : 4;
  fp.hD = a.hD;
  fp.hT = a.hT;
  fp.e_dense = a.e_dense;
  fp.apack = a.apack;
  fp.epack = a.epack;
  fp.rowmap = a.rowmap;
  fp.R_count = a.R_count;
  fp.pack_off = a.pack_off;
  // The outputs depend only on the target rows 0..A_b and the drafter rows
  // 0..min(A_b, K-1): the same row windows as greedy verification.  Pass k
  // scans the window's rows of the sequences that accepted every earlier
  // draft (top-k kernel), then runs their accept tests (finalize kernel).
  const int n_pass = a.windows.n;
  const int* start = a.windows.start;
  DeviceInfo info;
  cudaError_t e0 = device_info(&info);
  if (e0 != cudaSuccess) return e0;
  // Copies after the last pass, balanced over the grid: always with windows;
  // in one pass when it packs rows for fewer sequences than SMs (otherwise
  // each finalising CTA copies its own sequence's rows).
  const bool defer = a.e_out && (n_pass > 1 || (a.R_count && a.B < info.sm_count));
  const long long topk_resident = (long long)info.sm_count * 3;  // __launch_bounds__(kThreads, 3)
  fp.defer_copies = defer ? 1 : 0;
  for (int k = 0; k < n_pass; ++k) {
    const bool last = k == n_pass - 1;
    tp.i0 = fp.i0 = start[k];
    tp.i1 = fp.i1 = start[k + 1];
    tp.live_in = fp.live_in = k == 0 ? nullptr : a.live + (size_t)((k - 1) & 1) * a.B;
    tp.count_in = fp.count_in = k == 0 ? nullptr : a.pass_counts + k;
    fp.live_out = last ? nullptr : a.live + (size_t)(k & 1) * a.B;
    fp.count_out = last ? nullptr : a.pass_counts + k + 1;
    fp.pass_counts = last && n_pass > 1 ? a.pass_counts + 1 : nullptr;
    fp.n_counts = last ? n_pass - 1 : 0;
    fp.exits = last && n_pass > 1 ? a.pass_counts : nullptr;
    const int wt = tp.i1 - tp.i0, wd = (tp.i1 < a.K ? tp.i1 : a.K) - tp.i0;
    // Parts per row, where the pass may have fewer rows than resident CTAs:
    // as many as keep them in one wave, at least 16 KB of logits each.  In
    // the first pass every row is known to be there; a later pass, whose
    // rows are not known here, gets a whole resident grid in clusters of four
    // and decides on the device.
    const long long rows_max = (long long)a.B * (wt + wd);
    const long long most = std::max(1LL, (long long)a.V * fp.elem / (16 << 10));
    int parts = 1;
    while (parts < kMaxParts && 2 * parts <= most && (k > 0 ? parts < 4 : 2 * parts * rows_max <= topk_resident)) parts *= 2;
    tp.parts = parts;
    long long grid_n = k == 0 ? rows_max * parts : std::min(rows_max * parts, topk_resident);
    grid_n = std::max(1LL, grid_n / parts) * parts;
    auto topk = k == 0 ? (dtype == RETRACE_BF16 ? sampled_topk_kernel<__nv_bfloat16, false>
                                                : sampled_topk_kernel<float, false>)
                       : (dtype == RETRACE_BF16 ? sampled_topk_kernel<__nv_bfloat16, true>
                                                : sampled_topk_kernel<float, true>);
    cudaError_t err = k == 0 ? launch_cluster(topk, dim3((unsigned)grid_n), dim3(kThreads), stream, (unsigned)parts, tp)
                             : launch_dependent(topk, dim3((unsigned)grid_n), dim3(kThreads), 0, stream,
                                                (unsigned)parts, tp);
    if (err != cudaSuccess) return err;
    err = launch_dependent(sampled_finalize_kernel, dim3((unsigned)a.B), dim3(32 * kFinWarps), 0, stream, 1, fp);
    if (err != cudaSuccess) return err;
  }
  if (!defer) return cudaSuccess;
  // the row copies and packing, balanced over the grid
  VerifyArgs c{};
  c.B = a.B;
  c.K = a.K;
  c.V = a.V;
  c.accept_len = a.accept_len;
  c.e = a.e;
  c.e_batch_stride = a.e_batch_stride;
  c.e_pos_stride = a.e_pos_stride;
  c.e_out = a.e_out;
  c.d = a.d;
  c.hD = a.hD;
  c.hT = a.hT;
  c.e_dense = a.e_dense;
  c.apack = a.apack;
  c.epack = a.epack;
  c.rowmap = a.rowmap;
  c.R_count = a.R_count;
  c.pack_off = a.pack_off;
  c.cond_copy = kCondCopyKeep;
  return launch_verify_copies(c, dtype, stream);
}

}  // namespace retrace
