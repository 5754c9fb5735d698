// Conditioning projections on the CUDA cores (FFMA, fp32 accumulation).
//
// This path serves fp32 workloads (which must not use TF32) and bf16 shapes
// the tensor-core kernels do not take.  Same arithmetic as the tensor-core
// path:
//   correction  r = m + beta * W_c [m; u]                (Eq. 6-7)
//   gate        e~ = e + (W_v r) .* sigmoid(W_g [e; r])  (Eq. 8)
// with the operand rows gathered through the device-side row plan.
#include "common.cuh"
#include "internal.h"
#include "plan.cuh"
#include "tc_pair.cuh"

namespace retrace {
namespace {

// One kernel for both projections.  A unit is a tile of 64 weight rows (64
// features of W_c; for the gate 32 rows of W_v and the same 32 of W_g, so that
// v and the gate of a feature meet in one CTA) against a tile of up to 64
// conditioned rows.  The reduction is cut into 32-deep chunks, and the chunks
// of a unit are split over a cluster of S CTAs: with few rows a unit per 64
// features would leave most SMs idle and walk thousands of products one
// memory latency after another.  A chunk goes through a four-stage cp.async
// ring; thread (ty, tx) of 16 x 16 owns rows ty + 16 i and weight rows
// tx + 16 j (4 MR values) and reads both operands 16 bytes at a time along the
// reduction (rows padded to 36 floats: conflict-free).  Each CTA then leaves
// its partial tile in shared memory, and after a cluster barrier every CTA
// sums its share of the rows over the S partials in a fixed order (results
// repeat bit for bit) and applies the epilogue.  MR = rows of the tile / 16 is
// chosen on the device from R.
//
// Products are summed by eights, by chunk, by split, and the splits in pairs.
// One chain over the split took 42.4 us instead of 43.2 for a round of B = 8, K =
// 8, d = 1024, but had two to four times the rounding error (relative to 64 bits
// there 3.4e-7, now 1.4e-7; B = 1, K = 16, d = 2048: 5.6e-7, now 1.6e-7; a warp per
// feature with its lanes along the reduction 2.5e-7).  FINE (fine_sums) adds by
// fours and in pairs up to the chunk, and the splits with their rounding errors:
// by eights, short reductions over few rows had up to 8 % more error than that
// warp per feature, whose lanes held a few products each (r / e~ at B = 2, K = 16,
// d = 64: 6.50e-8 / 1.16e-7 against 6.20e-8 / 1.12e-7, now 5.78e-8 / 1.08e-7; d = 72:
// 6.68e-8 / 1.19e-7 against 6.27e-8 / 1.12e-7, now 5.69e-8 / 1.06e-7).
constexpr int kNT = 256;
constexpr int kTileRows = 64;              // most conditioned rows of a tile
constexpr int TN = 64, TK = 32;            // weight rows and reduction depth of a chunk
constexpr int kLd = TK + 4;                // floats between rows of a staged chunk
constexpr int kSimtStages = 4;
constexpr int kStageFloats = (kTileRows + TN) * kLd;
constexpr int kSimtSmem = kSimtStages * kStageFloats * 4;
static_assert(kTileRows * TN <= kSimtStages * kStageFloats, "the partial tile reuses the ring");

struct SimtParams {
  const void* a0;  // rows operand, part 0 and 1: hD, hT (correction); r, dense e (gate)
  const void* a1;
  const void* w;   // W_c (correction) or W_v (gate)
  const void* wg;  // W_g
  const void* e;
  float* ge;       // W_g[:, :d] e for a broadcast e
  float beta;
  int B, K, d;
  RowSource rows;
  void* out;
  int compact;     // the compact side of r: r_out rows (correction), r rows (gate)
  int raw;         // correction: r = m, no reduction
  int e_dense;
  int S, ftiles;   // cluster size, feature tiles
  int clusters;    // clusters with a unit; CTAs past them compute ge
  int vec;         // 16-byte fp32 copies
};

// Whether a projection of at most `rows` rows takes FINE sums.  From d = 224 on
// the sums by eights have less error than a warp per feature too, and above 32
// rows that was never the alternative.
inline bool fine_sums(long long rows, int d) { return rows <= 32 && d < 224; }

// Row numbers of the plan: the rows of this CTA's row tile nt, cut from R into
// tiles of equal size (a multiple of 16, at most kTileRows).  Fills s_b (-1
// past the last row), s_j, s_nb; returns R and the tile size and first row.
__device__ int plan_row_tile(const RowSource& rs, int B, int K, int nt, int* s_b, int* s_j, int* s_nb, int* s_scan,
                             int* tile, long long* m0) {
  constexpr int NW = kNT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int total = 0, nb = 0;
  for (int base = 0; base < B; base += kNT) {
    nb = base + tid < B ? rows_of(rs, base + tid, K) : 0;
    total += nb;
  }
  // inclusive sums over the threads (with B <= kNT: over the sequences)
  int x = total;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) s_scan[warp] = x;
  for (int q = tid; q < kTileRows; q += kNT) {
    s_b[q] = -1;
    s_j[q] = 0;
    s_nb[q] = 0;
  }
  __syncthreads();
  int before = 0, R = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    if (w < warp) before += s_scan[w];
    R += s_scan[w];
  }
  const int ntiles = (R + kTileRows - 1) / kTileRows;
  *tile = ntiles > 0 ? ((R + ntiles - 1) / ntiles + 15) / 16 * 16 : 16;
  *m0 = (long long)nt * *tile;
  if (*m0 >= R) return R;
  if (B <= kNT) {
    const long long off = before + x - nb;
    const long long lo = off > *m0 ? off : *m0, end = *m0 + *tile;
    const long long hi = off + nb < end ? off + nb : end;
    for (long long g = lo; g < hi; ++g) {
      const int q = (int)(g - *m0);
      s_b[q] = tid;
      s_j[q] = (int)(g - off);
      s_nb[q] = nb;
    }
    __syncthreads();
  } else {
    __syncthreads();  // s_scan is read to the end
    plan_tile<kNT, kTileRows>(rs, B, K, *m0, s_b, s_j, s_nb, s_scan);
  }
  return R;
}

__device__ __forceinline__ void cp_async16_zfill(uint32_t smem_dst, const void* gsrc, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gsrc), "r"(in ? 16 : 0)
               : "memory");
}

// Four consecutive elements src[k..k+3] of a row of d into staged floats; zeros
// past the row's end (k >= d) or for a row that does not exist (src NULL).
template <typename T>
__device__ __forceinline__ void stage4(float* dst, const T* src, int k, int d, const void* any, bool vec) {
  if constexpr (sizeof(T) == 4) {
    if (vec) {
      const bool in = src != nullptr && k < d;
      cp_async16_zfill(smem_u32(dst), in ? static_cast<const void*>(src + k) : any, in);
      return;
    }
  }
  float v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = (src != nullptr && k + q < d) ? to_f32(src[k + q]) : 0.f;
  *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ float warp_sum(float s) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  return s;
}

// W_g[i, :d] e by one warp: lanes stride the row, four loads in flight each.
template <typename T>
__device__ __forceinline__ float gate_bias_row(const T* Wg, const T* e, int i, int d, int lane) {
  const T* w = Wg + (long long)i * 2 * d;
  float s = 0.f;
  for (int k0 = lane; k0 < d; k0 += 4 * 32) {
    float a[4], b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + 32 * q;
      a[q] = k < d ? to_f32(w[k]) : 0.f;
      b[q] = k < d ? to_f32(e[k]) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) s = fmaf(a[q], b[q], s);
  }
  return warp_sum(s);
}

// Stages the weight rows of chunk c (of chunks [c0, c1)) of the unit at n0.
template <typename T, bool GATE>
__device__ __forceinline__ void stage_weights(const SimtParams& p, float* ring, int n0, int c, int c0) {
  const int tid = threadIdx.x, d = p.d, per = (d + TK - 1) / TK;  // chunks per part
  const int part = c >= per ? 1 : 0, kc = (c - part * per) * TK + (tid % 8) * 4;
  const T* W = reinterpret_cast<const T*>(p.w);
  const T* Wg = reinterpret_cast<const T*>(p.wg);
  float* Bs = ring + (c - c0) % kSimtStages * kStageFloats + kTileRows * kLd;
#pragma unroll
  for (int i = 0; i < TN / 32; ++i) {
    const int r = tid / 8 + 32 * i;
    const T* src;
    if constexpr (!GATE) {
      const int n = n0 + r;
      src = n < d ? W + (long long)n * 2 * d + (long long)part * d : nullptr;
    } else {
      const int n = n0 + (r & 31);  // i = 0: rows of W_v, i = 1: the same rows of W_g
      if (i == 0) {
        if (part) continue;  // the e part has a gate only
        src = n < d ? W + (long long)n * d : nullptr;
      } else {
        src = n < d ? Wg + (long long)n * 2 * d + (part ? 0 : d) : nullptr;
      }
    }
    stage4<T>(Bs + r * kLd + (tid % 8) * 4, src, kc, d, W, p.vec != 0);
  }
}
constexpr int kSimtAhead = kSimtStages - 1;  // chunks staged ahead

// v[0] = the sum of v[0..7], each addition's rounding error added at the end
// (Knuth's two-sum; the error of an infinite sum is no number and is left out).
__device__ __forceinline__ void sum_exactly(float4 (&v)[8]) {
  float4 lost = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [](float& s, float& c, float x) {
    const float t = s + x, z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
  };
#pragma unroll
  for (int s = 1; s < 8; ++s) {
    add(v[0].x, lost.x, v[s].x);
    add(v[0].y, lost.y, v[s].y);
    add(v[0].z, lost.z, v[s].z);
    add(v[0].w, lost.w, v[s].w);
  }
  auto finite = [](float c) { return fabsf(c) < INFINITY ? c : 0.f; };
  add4(v[0], make_float4(finite(lost.x), finite(lost.y), finite(lost.z), finite(lost.w)));
}

// The partial tile of this CTA: its chunks [c0, c1) of the unit with weight
// tile n0, rows at s_off0 / s_off1 (-1: no row), into ring[] as [row][TN].
// The weights of the first kSimtAhead chunks are staged already.
template <typename T, bool GATE, int MR, bool FINE>
__device__ __forceinline__ void simt_partial(const SimtParams& p, float* ring, const long long* s_off0,
                                             const long long* s_off1, int n0, int c0, int c1) {
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16, d = p.d;
  const int per = (d + TK - 1) / TK;  // chunks per part
  const T* A0 = reinterpret_cast<const T*>(p.a0);
  const T* A1 = reinterpret_cast<const T*>(p.a1);
  auto stage = [&](int c, bool weights) {
    if (c < c1) {
      const int part = c >= per ? 1 : 0, kc = (c - part * per) * TK + (tid % 8) * 4;
      float* As = ring + (c - c0) % kSimtStages * kStageFloats;
#pragma unroll
      for (int i = 0; i < (MR + 1) / 2; ++i) {
        const int r = tid / 8 + 32 * i;
        if (r < 16 * MR) {
          const long long off = part ? s_off1[r] : s_off0[r];
          stage4<T>(As + r * kLd + (tid % 8) * 4, off >= 0 ? (part ? A1 : A0) + off : nullptr, kc, d, p.w, p.vec != 0);
        }
      }
      if (weights) stage_weights<T, GATE>(p, ring, n0, c, c0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[MR][4];
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll
  for (int q = 0; q < kSimtAhead; ++q) stage(c0 + q, false);
  for (int c = c0; c < c1; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSimtAhead - 1) : "memory");
    __syncthreads();  // chunk c is staged, and chunk c - 1's slot is read
    stage(c + kSimtAhead, true);
    const float* As = ring + (c - c0) % kSimtStages * kStageFloats + ty * kLd;
    const float* Bs = ring + (c - c0) % kSimtStages * kStageFloats + (kTileRows + tx) * kLd;
    const bool gate_only = GATE && c >= per;
    float sum[MR][4], s16[MR][4];  // of this chunk, and of half of it (FINE)
#pragma unroll
    for (int k0 = 0; k0 < TK; k0 += 8) {
      float t[MR][4], t4[MR][4];
#pragma unroll
      for (int k = k0; k < k0 + 8; k += 4) {
        float4 a[MR], b[4];
#pragma unroll
        for (int i = 0; i < MR; ++i) a[i] = *reinterpret_cast<const float4*>(As + 16 * i * kLd + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(Bs + 16 * j * kLd + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j < 2 && gate_only) continue;  // weight rows tx, tx + 16: W_v
#pragma unroll
          for (int i = 0; i < MR; ++i) {
            if constexpr (FINE) {
              float& x = k == k0 ? t4[i][j] : t[i][j];
              x = a[i].x * b[j].x;
              x = fmaf(a[i].y, b[j].y, x);
              x = fmaf(a[i].z, b[j].z, x);
              x = fmaf(a[i].w, b[j].w, x);
              if (k == k0) continue;
              x += t4[i][j];
              s16[i][j] = k0 % 16 == 0 ? x : s16[i][j] + x;
              if (k0 % 16 == 8) sum[i][j] = k0 == 8 ? s16[i][j] : sum[i][j] + s16[i][j];
              continue;
            }
            t[i][j] = k == k0 ? a[i].x * b[j].x : fmaf(a[i].x, b[j].x, t[i][j]);
            t[i][j] = fmaf(a[i].y, b[j].y, t[i][j]);
            t[i][j] = fmaf(a[i].z, b[j].z, t[i][j]);
            t[i][j] = fmaf(a[i].w, b[j].w, t[i][j]);
            if (k > k0) sum[i][j] = k0 == 0 ? t[i][j] : sum[i][j] + t[i][j];
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j < 2 && gate_only) continue;
#pragma unroll
      for (int i = 0; i < MR; ++i) acc[i][j] += sum[i][j];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // the ring becomes the partial tile
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) ring[(ty + 16 * i) * TN + tx + 16 * j] = acc[i][j];
}

template <typename T, bool GATE, bool FINE>
__global__ void __launch_bounds__(kNT, 2) simt_cluster_kernel(const SimtParams p) {
  extern __shared__ float4 simt_smem[];
  __shared__ int s_b[kTileRows], s_j[kTileRows], s_nb[kTileRows], s_scan[kNT / 32 + 1];
  __shared__ long long s_off0[kTileRows], s_off1[kTileRows];
  float* ring = reinterpret_cast<float*>(simt_smem);
  const int tid = threadIdx.x, S = p.S, K = p.K, d = p.d;
  const int cid = (int)(blockIdx.x / (unsigned)S);
  pdl_launch_dependents();
  const T* e = reinterpret_cast<const T*>(p.e);
  if (cid >= p.clusters) {  // the gate's broadcast-e half (inputs only: no wait)
    const int first = ((int)blockIdx.x - p.clusters * S) * (kNT / 32) + tid / 32;
    const int stride = ((int)gridDim.x - p.clusters * S) * (kNT / 32);
    for (int i = first; i < d; i += stride) {
      const float s = gate_bias_row<T>(reinterpret_cast<const T*>(p.wg), e, i, d, tid & 31);
      if ((tid & 31) == 0) p.ge[i] = s;
    }
    return;
  }
  // The weights are inputs: those of this CTA's first chunks come while the
  // previous kernel ends and the rows are planned.
  const uint32_t rank = cluster_rank();
  constexpr int F = GATE ? 32 : 64;  // features of a unit
  const int n0 = cid % p.ftiles * F;
  const int per = (d + TK - 1) / TK;
  const int chunks = GATE ? per * (p.e_dense ? 2 : 1) : (p.raw ? 0 : 2 * per);
  const int c0 = (int)((long long)rank * chunks / S), c1 = (int)((long long)(rank + 1) * chunks / S);
#pragma unroll
  for (int q = 0; q < kSimtAhead; ++q)
    if (c0 + q < c1) stage_weights<T, GATE>(p, ring, n0, c0 + q, c0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  pdl_wait();  // the accepted lengths (and r) come from the previous kernels
  int tile;
  long long m0;
  const int R = plan_row_tile(p.rows, p.B, K, cid / p.ftiles, s_b, s_j, s_nb, s_scan, &tile, &m0);
  if (m0 >= R) {  // the whole cluster
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return;
  }
  const int rows = (int)(R - m0 < tile ? R - m0 : tile);
  if (tid < kTileRows) {
    const int b = s_b[tid];
    const long long pos = (long long)b * K + s_j[tid];
    const int A = K - 1 - s_nb[tid];
    if (b < 0) {
      s_off0[tid] = s_off1[tid] = -1;
    } else if constexpr (!GATE) {
      s_off0[tid] = (pos + A + 1) * d;  // m_j = hD[b, A+1+j]
      s_off1[tid] = (pos + A) * d;      // u_j = hT[b, A+j]
    } else {
      s_off0[tid] = (p.compact ? m0 + tid : pos) * d;
      s_off1[tid] = p.e_dense ? pos * d : 0;
    }
  }
  __syncthreads();
  if (tile == 16) {
    simt_partial<T, GATE, 1, FINE>(p, ring, s_off0, s_off1, n0, c0, c1);
  } else if (FINE || tile == 32) {
    simt_partial<T, GATE, 2, FINE>(p, ring, s_off0, s_off1, n0, c0, c1);
  } else if constexpr (!FINE) {
    if (tile == 48) simt_partial<T, GATE, 3, false>(p, ring, s_off0, s_off1, n0, c0, c1);
    else simt_partial<T, GATE, 4, false>(p, ring, s_off0, s_off1, n0, c0, c1);
  }
  cluster_sync_all();  // every partial of the cluster is in shared memory
  const int l0 = (int)rank * rows / S, l1 = ((int)rank + 1) * rows / S;  // this CTA's rows of the tile
  const uint32_t P = smem_u32(ring);
  T* out = reinterpret_cast<T*>(p.out);
  for (int x = tid; x < (l1 - l0) * (F / 4); x += kNT) {
    const int l = l0 + x / (F / 4), f = x % (F / 4) * 4;
    const uint32_t at = P + (uint32_t)((l * TN + f) * 4);
    float4 v[8], g[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {  // all loads first, then the sums, in pairs of ranks
      v[s] = g[s] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (s < S) {
        const uint32_t src = map_rank(at, (uint32_t)s);
        v[s] = ld_cluster_f4(src);
        if constexpr (GATE) g[s] = ld_cluster_f4(src + 32 * 4);
      }
    }
    if constexpr (FINE) {
      sum_exactly(v);
      if constexpr (GATE) sum_exactly(g);
    } else {
#pragma unroll
      for (int h = 1; h < 8; h *= 2)
#pragma unroll
        for (int s = 0; s + h < 8; s += 2 * h) {
          add4(v[s], v[s + h]);
          if constexpr (GATE) add4(g[s], g[s + h]);
        }
    }
    const float vv[4] = {v[0].x, v[0].y, v[0].z, v[0].w}, gg[4] = {g[0].x, g[0].y, g[0].z, g[0].w};
    const long long pos = (long long)s_b[l] * K + s_j[l];
    const long long orow = (!GATE && p.compact) ? m0 + l : pos;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = n0 + f + q;
      if (n >= d) break;
      if constexpr (!GATE) {
        const T m = reinterpret_cast<const T*>(p.a0)[s_off0[l] + n];
        out[orow * d + n] = p.raw ? m : from_f32<T>(to_f32(m) + p.beta * vv[q]);
      } else {
        const float z = gg[q] + (p.e_dense ? 0.f : p.ge[n]);
        const float ev = to_f32(e[s_off1[l] + n]);
        const float gate = 1.f / (1.f + expf(-z));
        out[orow * d + n] = from_f32<T>(ev + vv[q] * gate);
      }
    }
  }
  cluster_sync_all();  // no CTA leaves while the others read its shared memory
}

// ge = W_g[:, :d] e alone (a gate-only call), one warp per output.
template <typename T>
__global__ void __launch_bounds__(256) gate_bias_kernel(const T* __restrict__ Wg,
                                                        const T* __restrict__ e, int d,
                                                        float* __restrict__ ge) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= d) return;
  const float s = gate_bias_row<T>(Wg, e, i, d, threadIdx.x & 31);
  if ((threadIdx.x & 31) == 0) ge[i] = s;
}

// One CTA per position (b, j): n_out[b], and rows j >= n_b of the zero / copy targets.
template <typename T>
__global__ void __launch_bounds__(256) fill_rows_kernel(int B, int K, int d, RowSource rows,
                                                        int32_t* n_out, T* zero_dst, const T* e,
                                                        int e_dense, T* e_dst) {
  const int b = (int)(blockIdx.x / (unsigned)K), j = (int)(blockIdx.x % (unsigned)K);
  const int nb = rows_of(rows, b, K);
  if (j == 0 && threadIdx.x == 0 && n_out) n_out[b] = nb;
  if (j < nb) return;
  const long long row = ((long long)b * K + j) * d;
  const T* src = e + (e_dense ? row : 0);
  for (int k = threadIdx.x; k < d; k += blockDim.x) {
    if (zero_dst) zero_dst[row + k] = from_f32<T>(0.f);
    if (e_dst) e_dst[row + k] = src[k];
  }
}

// Launches a projection: one cluster of S CTAs per unit of the largest
// possible R (those past the R found on the device leave at once) and, with
// `gemv`, CTAs for W_g[:, :d] e behind them.  S: two CTAs per SM over the
// units at three quarters of the possible rows, at most 8 and one chunk each.
template <typename T, bool GATE, bool FINE>
cudaError_t launch_simt(SimtParams& p, bool gemv, cudaStream_t stream) {
  const long long rmax = (long long)p.B * (p.K - 1);
  DeviceInfo info;
  cudaError_t err = device_info(&info);
  if (err != cudaSuccess) return err;
  static std::atomic<int> attr_done[64];
  if (!attr_done[info.device & 63].load(std::memory_order_acquire)) {
    err = cudaFuncSetAttribute(simt_cluster_kernel<T, GATE, FINE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSimtSmem);
    if (err != cudaSuccess) return err;
    attr_done[info.device & 63].store(1, std::memory_order_release);
  }
  constexpr int F = GATE ? 32 : 64;
  p.ftiles = (p.d + F - 1) / F;
  const long long tiles = (3 * rmax / 4 + kTileRows) / kTileRows;
  const int chunks = (p.d + TK - 1) / TK * (GATE ? (p.e_dense ? 2 : 1) : 2);
  long long S = p.raw ? 1 : 2LL * info.sm_count / (p.ftiles * tiles);
  S = std::min<long long>(std::min<long long>(S, 8), chunks);
  p.S = S < 1 ? 1 : (int)S;
  const long long clusters = (long long)p.ftiles * ((rmax + kTileRows - 1) / kTileRows);
  const long long extra = gemv ? (p.d / 8 + p.S) / p.S : 0;  // clusters of the GEMV: about a warp per row
  if ((clusters + extra) * p.S >= (1LL << 31)) return cudaErrorInvalidConfiguration;
  p.clusters = (int)clusters;
  const size_t es = sizeof(T);
  auto al = [](const void* q) { return (uintptr_t)q % 16 == 0; };
  p.vec = es == 4 && p.d % 4 == 0 && al(p.a0) && al(p.w) && (!GATE || al(p.wg)) && (!p.a1 || al(p.a1));
  return launch_dependent(simt_cluster_kernel<T, GATE, FINE>, dim3((unsigned)((clusters + extra) * p.S)), dim3(kNT),
                          (size_t)kSimtSmem, stream, (unsigned)p.S, p);
}

template <typename T, bool GATE>
cudaError_t launch_simt(SimtParams& p, bool gemv, cudaStream_t stream) {
  const long long rmax = (long long)p.B * (p.K - 1);
  if (rmax <= 0) return cudaSuccess;
  return fine_sums(rmax, p.d) ? launch_simt<T, GATE, true>(p, gemv, stream) : launch_simt<T, GATE, false>(p, gemv, stream);
}

template <typename T>
cudaError_t correct_typed(const CorrectArgs& a, cudaStream_t stream) {
  SimtParams p{};
  p.a0 = a.hD;
  p.a1 = a.hT;
  p.w = a.Wc;
  p.wg = a.Wg;
  p.e = a.e;
  p.ge = a.ge;
  p.beta = a.beta;
  p.B = a.B;
  p.K = a.K;
  p.d = a.d;
  p.rows = a.rows;
  p.out = a.r_out;
  p.compact = a.compact_out;
  p.raw = a.raw;
  return launch_simt<T, false>(p, a.ge != nullptr, stream);
}

template <typename T>
cudaError_t gate_typed(const GateArgs& a, cudaStream_t stream) {
  SimtParams p{};
  p.a0 = a.r;
  p.a1 = a.e_dense ? a.e : nullptr;
  p.w = a.Wv;
  p.wg = a.Wg;
  p.e = a.e;
  p.ge = const_cast<float*>(a.ge);
  p.B = a.B;
  p.K = a.K;
  p.d = a.d;
  p.rows = a.rows;
  p.out = a.e_out;
  p.compact = a.r_compact;
  p.e_dense = a.e_dense;
  return launch_simt<T, true>(p, false, stream);
}

}  // namespace

cudaError_t launch_correct_simt(const CorrectArgs& a, retrace_dtype dtype, cudaStream_t stream) {
  return dtype == RETRACE_BF16 ? correct_typed<__nv_bfloat16>(a, stream) : correct_typed<float>(a, stream);
}

cudaError_t launch_gate_simt(const GateArgs& a, retrace_dtype dtype, cudaStream_t stream) {
  return dtype == RETRACE_BF16 ? gate_typed<__nv_bfloat16>(a, stream) : gate_typed<float>(a, stream);
}

cudaError_t launch_gate_bias(const void* Wg, const void* e, int d, float* ge, retrace_dtype dtype,
                             cudaStream_t stream) {
  const unsigned grid = (unsigned)((d + 7) / 8);
  if (dtype == RETRACE_BF16)
    gate_bias_kernel<__nv_bfloat16><<<grid, 256, 0, stream>>>(
        reinterpret_cast<const __nv_bfloat16*>(Wg), reinterpret_cast<const __nv_bfloat16*>(e), d, ge);
  else
    gate_bias_kernel<float><<<grid, 256, 0, stream>>>(reinterpret_cast<const float*>(Wg),
                                                      reinterpret_cast<const float*>(e), d, ge);
  return cudaGetLastError();
}

cudaError_t launch_fill_rows(int B, int K, int d, RowSource rows, int32_t* n_out, void* zero_dst,
                             const void* e, int e_dense, void* e_dst, retrace_dtype dtype,
                             cudaStream_t stream) {
  if (B <= 0 || K <= 0) return cudaSuccess;
  dim3 grid((unsigned)((long long)B * K));
  if (dtype == RETRACE_BF16)
    fill_rows_kernel<__nv_bfloat16><<<grid, 256, 0, stream>>>(
        B, K, d, rows, n_out, reinterpret_cast<__nv_bfloat16*>(zero_dst),
        reinterpret_cast<const __nv_bfloat16*>(e), e_dense, reinterpret_cast<__nv_bfloat16*>(e_dst));
  else
    fill_rows_kernel<float><<<grid, 256, 0, stream>>>(B, K, d, rows, n_out,
                                                      reinterpret_cast<float*>(zero_dst),
                                                      reinterpret_cast<const float*>(e), e_dense,
                                                      reinterpret_cast<float*>(e_dst));
  return cudaGetLastError();
}

}  // namespace retrace
