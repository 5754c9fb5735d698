// Conditioning projections on the 5th-generation tensor cores (tcgen05).
//
// Two steps per projection family:
//
// 1. pack_rows_kernel (standalone calls; in a round verification packs) lays
//    the conditioned rows out contiguously, in sequence order (R = sum_b n_b
//    rows, n_b = max(0, K-1-A_b)):
//      correction operand  Apack[g] = [ hD[b, A_b+1+j] ; hT[b, A_b+j] ]  (Eq. 4-5),
//      or the corrected signal rows r[b, j] for a standalone gate call,
//      plus, for per-position e, Epack[g] = e[b, j];
//    with rowmap[g] = b*K + j and the row count R.  Contiguous rows let the
//    GEMMs stream their A operand with tiled TMA boxes (per-row gathers were
//    measured to starve the tensor pipe).
//
// 2. one persistent launch runs both projections from a dynamic tile queue
//    (every correction tile, then every gate tile; a gate tile of a row block
//    waits until the correction epilogues of that block have written r):
//    correction (Eq. 6-7):  r = m + beta * W_c [m; u]
//        A = Apack [R, 2d]; B = W_c [d, 2d] (K-major); N = 256 tiles of c;
//        the epilogue adds m (the first d columns of Apack) and writes r bf16.
//    gated fusion (Eq. 8):  e~ = e + (W_v r) .* sigmoid(W_g [e; r])
//        A = r rows; the B tile stacks 128 rows of W_v over the matching 128
//        rows of W_g[:, d:2d], so one N = 256 MMA yields v (accumulator
//        columns 0..127) and the r half of the gate (128..255) for the same
//        output features.  The e half of the gate is a broadcast vector
//        computed once by idle warps (W_g[:, :d] e, added in the epilogue)
//        or, for per-position e, extra K blocks (Epack x W_g[:, :d])
//        accumulated into the gate columns.
//    Three kernels implement it:
//    swap_cluster_kernel  (few rows, cond_small_r; one launch per projection
//                       instead) the weights as the M side;
//    cond_pair_kernel   (more rows) clusters of two CTAs, 256-row tiles,
//                       tcgen05.mma.cta_group::2 M256 N256 K16; each CTA
//                       stages its own 128 rows and half of the weight tile
//                       (each described at the kernel);
//    cond_kernel<false> (more rows, per-position e, d a multiple of 256) one
//                       CTA per SM, 128-row tiles, tcgen05.mma.cta_group::1
//                       M128 N256 K16;
//    cond_kernel<true>  the overlapped round: the same plus verification
//                       streamed through shared memory (verify_stream.cuh).
//
// Warp roles of the persistent kernels' GEMM part (256 threads):
//   warp 0     tile scheduler + TMA producer (one elected lane);
//   warp 1     MMA issuer (one lane);
//   warp 2     TMEM allocation: 2 accumulators x 256 fp32 columns = 512 columns;
//   warps 2-3  (pair kernel) the broadcast-e GEMV W_g[:, :d] e, in static shares over
//              the grid; the overlapped round's epilogue warps claim its rows from a
//              counter before their first tile;
//   warps 4-7  epilogue: tcgen05.ld of their 32 TMEM lanes (= tile rows).
// The two accumulators alternate between tiles, so a tile's epilogue overlaps
// the next tile's main loop.  Every mbarrier wait is bounded; on expiry the CTA
// raises the workspace status flag, drains its own copies in flight, frees
// TMEM and returns.
#include "common.cuh"
#include "internal.h"
#include "plan.cuh"
#include "tc_pair.cuh"
#include "verify_stream.cuh"

namespace retrace {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;  // 64 bf16 = 128 bytes = one swizzle row
constexpr int STAGES = 4;
constexpr int THREADS = 256;
constexpr int THREADS_FUSED = 2 * THREADS + 32;  // + consumer warps 8-15 and the bookkeeper warp 16
constexpr int A_BYTES = BM * BK * 2;   // 16 KB
constexpr int B_BYTES = 256 * BK * 2;  // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;  // + slack for 1024-B alignment
// The overlapped round's kernel keeps three operand stages and gives the rest of the
// shared memory to the ring that streams the logits.
constexpr int STAGES_FUSED = 3;
constexpr int SMEM_BYTES_FUSED = STAGES_FUSED * STAGE_BYTES + kRingBufs * kChunkBytes + kStageBytes + 1024;
constexpr uint32_t ACC_COLS = 256;
constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;
constexpr uint32_t IDESC_N256 = idesc_bf16_f32(128, 256);
constexpr uint32_t IDESC_N128 = idesc_bf16_f32(128, 128);

// ---------------------------------------------------------------------------
// Row packing
// ---------------------------------------------------------------------------
// W_g[:, :d] e for the gate of a small-R call (broadcast e).
struct GateBiasParams {
  int d;
  const __nv_bfloat16* e;
  const __nv_bfloat16* Wg;
  float* ge;
};

struct PackParams {
  int B, K, d;
  RowSource rows;
  int mode;  // 0: [m; u] from hD / hT; 1: r rows from r [B, K, d]
  const __nv_bfloat16* src0;
  const __nv_bfloat16* src1;
  const __nv_bfloat16* e;
  int e_dense;
  __nv_bfloat16* apack;
  __nv_bfloat16* epack;
  int32_t* rowmap;
  int32_t* n_out;           // mode 0: n_b
  __nv_bfloat16* rest;      // [B, K, d]: rows j >= n_b are zeroed (mode 0) or set to e (mode 1)
  uint32_t* sync;           // counters of the projections: R, the others zeroed
  int sync_words;
  GateBiasParams bias;      // mode 1: W_g[:, :d] e (ge NULL: not computed)
};

// A warp copies n 16-byte vectors, eight loads in flight per lane; src NULL: zeros.
__device__ __forceinline__ void warp_copy_row(__nv_bfloat16* dst, const __nv_bfloat16* src, int n, int lane) {
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  for (int v0 = 0; v0 < n; v0 += 8 * 32) {
    uint4 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int v = v0 + k * 32 + lane;
      x[k] = src && v < n ? __ldg(s4 + v) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int v = v0 + k * 32 + lane;
      if (v < n) d4[v] = x[k];
    }
  }
}

// What precedes the projections of a standalone call, in one launch: the
// packed rows with their row map and count (in sequence order: a warp's first
// packed row is the number of rows of all earlier sequences, which it sums
// itself), n_b, the rows that carry nothing, the projections' counters and,
// before a gate, W_g[:, :d] e.  A warp takes consecutive positions (b, j), one
// each at the usual sizes.  Bound by
// latency at the sizes it runs at; as three launches (fill, memset, pack with
// one CTA per sequence) it took 2.7 + 10.4 us at B = 24, K = 12, d = 1152.
__global__ void __launch_bounds__(256) pack_rows_kernel(const PackParams p) {
  pdl_wait();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, K = p.K, d = p.d, vpr = d / 8;
  const int w = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5), nw = (int)gridDim.x * 8;
  if (blockIdx.x == 0)
    for (int k = threadIdx.x; k < p.sync_words; k += 256)
      if (k != kSyncRowCount) p.sync[k] = 0u;
  const long long all = (long long)p.B * K, per = (all + nw - 1) / nw;
  const int p0 = (int)min(w * per, all), p1 = (int)min(p0 + per, all);
  int b = p0 / K, off = 0;  // rows of the sequences before b
  for (int x0 = lane; x0 < b; x0 += 4 * 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) off += x0 + 32 * q < b ? rows_of(p.rows, x0 + 32 * q, K) : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xFFFFFFFFu, off, o);
  for (int pos = p0; pos < p1; ++pos) {
    if (pos == (b + 1) * K) off += rows_of(p.rows, b++, K);
    const int j = pos - b * K, nb = rows_of(p.rows, b, K);
    if (j == 0 && lane == 0) {
      if (p.n_out) p.n_out[b] = nb;
      if (b == p.B - 1) p.sync[kSyncRowCount] = (uint32_t)(off + nb);
    }
    const long long row = (long long)pos * d;
    if (j >= nb) {
      warp_copy_row(p.rest + row, p.mode == 0 ? nullptr : p.e + (p.e_dense ? row : 0), vpr, lane);
      continue;
    }
    const long long g = off + j;
    if (lane == 0) p.rowmap[g] = pos;
    if (p.mode == 0) {
      const int A = K - 1 - nb;
      warp_copy_row(p.apack + g * 2 * d, p.src0 + row + (long long)(A + 1) * d, vpr, lane);  // m_j (Eq. 4)
      warp_copy_row(p.apack + g * 2 * d + d, p.src1 + row + (long long)A * d, vpr, lane);    // u_j (Eq. 5)
    } else {
      warp_copy_row(p.apack + g * d, p.src0 + row, vpr, lane);
      if (p.e_dense) warp_copy_row(p.epack + g * d, p.e + row, vpr, lane);
    }
  }
  if (p.bias.ge) gate_bias_share(p.bias.e, p.bias.Wg, p.bias.ge, d, 2 * d, w, nw, lane);
}

// ---------------------------------------------------------------------------
// Persistent, dynamically scheduled projections
// ---------------------------------------------------------------------------
struct CondParams {
  int d;
  int do_correct, do_gate;
  const int32_t* R;
  const int32_t* rowmap;
  // correction
  const __nv_bfloat16* apack;  // [R, 2d]; the m half is re-read by the epilogue
  float beta;
  __nv_bfloat16* r_out;
  int compact_out;
  // gate
  const __nv_bfloat16* e;  // broadcast vector [d], or packed e rows [R, d] (e_dense)
  int e_dense;
  const __nv_bfloat16* Wg;
  float* ge;  // [d] = W_g[:, :d] e, computed here for a broadcast e
  __nv_bfloat16* e_out;
  uint32_t* sync;
  uint32_t* block_done;   // per 128-row block: correction epilogue warps finished
  uint32_t* block_ready;  // per 128-row block: packed rows published (overlapped round)
  int max_blocks;         // 128-row blocks of the largest possible R
  // CTA-pair kernel: the gate tiles of a last wave of at most split_max
  // tiles run as two K halves on two pairs.  Each half writes its fp32
  // accumulator to split_part and counts on split_ticket; the half that
  // counts second adds the other's accumulator to its own and runs the
  // epilogue.
  float* split_part;
  uint32_t* split_ticket;
  int split_max;
  uint32_t* status;
};

constexpr int TILE_SLOTS = 2;

// gate_bias_rows (tc_pair.cuh) over this kernel's broadcast e, W_g and ge.
__device__ __forceinline__ void gate_bias_rows(const CondParams& p, int d, int lane, uint32_t* next, uint32_t* done) {
  gate_bias_rows(p.e, p.Wg, p.ge, d, lane, next, done);
}

// One warp: ge for the 128 features from n0, in the order of a share's rows, so
// that the bits are the same whoever computes them.
__device__ __noinline__ void gate_bias_features(const CondParams& p, int d, int n0, int lane) {
  gate_bias_share(p.e, p.Wg, p.ge, d, 2 * d, n0, 1, lane, min(n0 + 128, d));
  __syncwarp();  // the warp reads the values back
}

// Correction epilogue of one tile row (Eq. 7): r = m + beta * c for the 256
// accumulator columns n0.., m = the first d columns of the packed row g.
// GENERAL: d may end inside the tile (at a multiple of 8 columns).
template <bool GENERAL>
__device__ __forceinline__ void epilogue_correction(const CondParams& p, uint32_t taddr, int g, bool valid, int n0,
                                                    int d) {
  const __nv_bfloat16* mrow = p.apack + (long long)g * 2 * d;
  const long long orow = valid ? (p.compact_out ? g : __ldcg(p.rowmap + g)) : 0;
  for (int cc = 0; cc < 8; ++cc) {
    float c[32];
    tmem_ld_32cols(taddr + (uint32_t)(cc * 32), c);
    if (valid) {
      const int n = n0 + cc * 32;
      const uint4* mv = reinterpret_cast<const uint4*>(mrow + n);
      uint4* ov = reinterpret_cast<uint4*>(p.r_out + orow * d + n);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        if (GENERAL && n + v * 8 >= d) break;
        const uint4 mw = __ldcg(mv + v);
        const uint32_t mwords[4] = {mw.x, mw.y, mw.z, mw.w};
        uint32_t o[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const float lo = bf16_lo(mwords[w]) + p.beta * c[v * 8 + 2 * w];
          const float hi = bf16_hi(mwords[w]) + p.beta * c[v * 8 + 2 * w + 1];
          o[w] = pack_bf16x2(lo, hi);
        }
        ov[v] = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// Gated-fusion epilogue of one tile row (Eq. 8): e~ = e + v * sigmoid(g) for
// the 128 features n0.., v in accumulator columns 0..127, the r half of the
// gate in 128..255 (plus W_g[:, :d] e from ge for a broadcast e, the same
// 32 values for every lane: one 16-byte broadcast load per four features).
// With `other` (a split tile), the other K half's accumulator of this row is
// added first: column c at other[128 c].
template <bool GENERAL>
__device__ __forceinline__ void epilogue_gate(const CondParams& p, uint32_t taddr, int g, bool valid, int n0, int d,
                                              const float* other = nullptr) {
  const long long orow = valid ? __ldcg(p.rowmap + g) : 0;
  const __nv_bfloat16* erow = p.e + (p.e_dense ? (long long)g * d : 0);
  for (int cc = 0; cc < 4; ++cc) {
    float v[32], gt[32];
    tmem_ld_32cols(taddr + (uint32_t)(cc * 32), v);
    tmem_ld_32cols(taddr + 128u + (uint32_t)(cc * 32), gt);
    if (valid) {
      const int n = n0 + cc * 32;
      if (other) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          v[i] += __ldcg(other + (cc * 32 + i) * 128);
          gt[i] += __ldcg(other + (128 + cc * 32 + i) * 128);
        }
      }
      if (!p.e_dense) {
        const float4* gb = reinterpret_cast<const float4*>(p.ge + n);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (GENERAL && n + 4 * j >= d) break;
          const float4 b = __ldcg(gb + j);
          gt[4 * j] += b.x;
          gt[4 * j + 1] += b.y;
          gt[4 * j + 2] += b.z;
          gt[4 * j + 3] += b.w;
        }
      }
      const uint4* ev = reinterpret_cast<const uint4*>(erow + n);
      uint4* ov = reinterpret_cast<uint4*>(p.e_out + orow * d + n);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        if (GENERAL && n + x * 8 >= d) break;
        const uint4 ew = __ldcg(ev + x);
        const uint32_t ewords[4] = {ew.x, ew.y, ew.z, ew.w};
        uint32_t o[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const int c0 = x * 8 + 2 * w;
          const float s0 = fast_sigmoid(gt[c0]), s1 = fast_sigmoid(gt[c0 + 1]);
          o[w] = pack_bf16x2(bf16_lo(ewords[w]) + v[c0] * s0, bf16_hi(ewords[w]) + v[c0 + 1] * s1);
        }
        ov[x] = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// Tile t < T0: correction tile (row block t / nt0, 256 output columns t % nt0);
// T0 <= t < T0 + T1: gate tile (row block (t-T0) / nt1, 128 features).  Tiles
// are handed out in this order by a global counter, so every gate tile's row
// block was handed out (to a running CTA) before it.
// FUSED: the same kernel also runs verification (verify_stream.cuh): warp 3
// streams the logits into a shared-memory ring, warps 8-15 reduce it, warp 16
// folds the keys.  Packed rows then become available while the kernel runs, so
// the tile queue is decoded in phases -- phase q holds the correction tiles of
// row block q followed by the gate tiles of row block q - kGateLag -- and the
// producer resolves each tile against the published per-block row counts
// before loading it.  R (and the last partial block) is known once every
// sequence is finalised.
// Not FUSED: a per-position e only.  Its 128-row tiles fill the last wave
// better than the pair kernel's, whose gate tiles are long with the e half
// added (a round, d = 2560, 1821 rows: 168 us here, 206 on pairs; d = 4096,
// 1821: 335 / 365; 2802: 440 / 445).
constexpr int kGateLag = 4;

template <bool FUSED>
__global__ void __launch_bounds__(FUSED ? THREADS_FUSED : THREADS, 1)
    cond_kernel(const __grid_constant__ CUtensorMap tmApack, const __grid_constant__ CUtensorMap tmWc,
                const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmE,
                const __grid_constant__ CUtensorMap tmWv, const __grid_constant__ CUtensorMap tmWg,
                const CondParams p, const VerifyStreamParams vp) {
  extern __shared__ uint8_t dsmem[];
  __shared__ __align__(8) uint64_t bar_full[STAGES];
  __shared__ __align__(8) uint64_t bar_empty[STAGES];
  __shared__ __align__(8) uint64_t bar_tfull[2];
  __shared__ __align__(8) uint64_t bar_tempty[2];
  __shared__ __align__(8) uint64_t bar_tile_full[TILE_SLOTS];
  __shared__ __align__(8) uint64_t bar_tile_empty[TILE_SLOTS];
  __shared__ int s_tile[TILE_SLOTS];
  __shared__ int s_rows[TILE_SLOTS];  // valid rows of the tile (FUSED)
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ VerifyStreamSmem vsm;

  constexpr int NST = FUSED ? STAGES_FUSED : STAGES;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = p.d;
  const int nt0 = d / 256, nt1 = d / 128;
  uint32_t* tile_queue = p.sync + kSyncTileQueue;
  uint32_t* gemv_next = p.sync + kSyncGemvNext;
  uint32_t* gemv_done = p.sync + kSyncGemvDone;
  uint32_t* block_done = p.block_done;
  const bool need_ge = FUSED && p.do_gate && !p.e_dense;

  if (tid == 0) {
    s_abort = 0;
    for (int s = 0; s < NST; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&bar_tfull[a]), 1);
      mbar_init(smem_u32(&bar_tempty[a]), 4);  // one arrival per epilogue warp
    }
    for (int a = 0; a < TILE_SLOTS; ++a) {
      mbar_init(smem_u32(&bar_tile_full[a]), 1);
      mbar_init(smem_u32(&bar_tile_empty[a]), 5);  // MMA thread + four epilogue warps
    }
    if constexpr (FUSED) vs_init(vsm);
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    if (p.do_correct) {
      tma_prefetch_desc(&tmApack);
      tma_prefetch_desc(&tmWc);
    }
    if (p.do_gate) {
      tma_prefetch_desc(&tmR);
      tma_prefetch_desc(&tmWv);
      tma_prefetch_desc(&tmWg);
      if (p.e_dense) tma_prefetch_desc(&tmE);
    }
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(&s_tmem), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t base = (smem_u32(dsmem) + 1023u) & ~1023u;
  const int kb_half = d / BK;
  // The set-up above may overlap the end of the previous kernel; R, the packed
  // rows and the row map are its outputs.
  int R = 0, T0 = 0, T = 0;
  if (!FUSED) {
    pdl_wait();
    R = *(volatile const int32_t*)p.R;
    const int tiles_m = (R + BM - 1) / BM;
    T0 = p.do_correct ? tiles_m * nt0 : 0;
    T = T0 + (p.do_gate ? tiles_m * nt1 : 0);
  }

  if (warp == 0) {
    // ---------------- tile scheduler + TMA producer ----------------
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (uint32_t lt = 0;; ++lt) {
        const uint32_t slot = lt % TILE_SLOTS, sph = (lt / TILE_SLOTS) & 1u;
        int t, rows = BM, m0, n0;
        bool corr, done = false;
        if (!FUSED) {
          t = (int)atomicAdd(tile_queue, 1u);
          done = t >= T;
          corr = t < T0;
          const int tt = corr ? t : t - T0;
          m0 = (corr ? tt / nt0 : tt / nt1) * BM;
          n0 = corr ? (tt % nt0) * 256 : (tt % nt1) * 128;
        } else {
          // next valid tile of the phased queue
          for (;;) {
            t = (int)atomicAdd(tile_queue, 1u);
            const int q = t / (nt0 + nt1), r = t % (nt0 + nt1);
            corr = r < nt0;
            const int m = corr ? q : q - kGateLag;
            n0 = corr ? r * 256 : (r - nt0) * 128;
            m0 = m * BM;
            if (m < 0) continue;  // gate slots of the first phases
            if (m >= p.max_blocks) {  // beyond any possible packed row
              if (!corr) {
                done = true;
                break;
              }
              continue;
            }
            // wait until block m is complete, or verification is over
            int state = 0;  // 1 valid, 2 past the last block
            const unsigned long long t_start = global_ns();
            for (uint32_t it2 = 0; state == 0; ++it2) {
              const uint32_t ready = ld_acquire(p.block_ready + m);
              if (ready >= (uint32_t)BM) {
                state = 1;
              } else if (ld_acquire(p.sync + kSyncSeqDone) >= (uint32_t)vp.B) {
                const int Rf = (int)ld_acquire(p.sync + kSyncRowCount);
                if (m0 >= Rf) state = 2;
                else if (ready >= (uint32_t)(Rf - m0)) { state = 1; rows = Rf - m0; }
              }
              if (state == 0) {
                __nanosleep(128);
                if ((it2 & 63u) == 63u && (s_abort || global_ns() - t_start > kWaitLimitNs)) break;
              }
            }
            if (state == 0) {
              ok = false;
              break;
            }
            if (state == 2) {
              // Block m is past the last packed row.  Gate tiles come in
              // increasing block order, so a gate tile past the end means
              // nothing valid is left; a correction tile past the end may
              // still be followed by valid gate tiles of earlier blocks.
              if (!corr) {
                done = true;
                break;
              }
              continue;
            }
            break;
          }
          if (!ok) break;
        }
        if (!mbar_wait_bounded(smem_u32(&bar_tile_empty[slot]), sph ^ 1u, &s_abort)) {
          ok = false;
          break;
        }
        s_tile[slot] = done ? -1 : t;
        s_rows[slot] = rows;
        mbar_arrive(smem_u32(&bar_tile_full[slot]));
        if (done) break;
        const int nkb = corr ? 2 * kb_half : kb_half + (p.e_dense ? kb_half : 0);
        if (!corr && p.do_correct) {
          // the r rows of this block are written by the correction epilogues
          if (!wait_counter(block_done + m0 / BM, (uint32_t)(4 * nt0), &s_abort)) {
            ok = false;
            break;
          }
          fence_proxy_async_global();
        }
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const uint32_t s = it % NST, ph = (it / NST) & 1u;
          if (!mbar_wait_bounded(smem_u32(&bar_empty[s]), ph ^ 1u, &s_abort)) {
            ok = false;
            break;
          }
          const uint32_t a_dst = base + s * STAGE_BYTES, b_dst = a_dst + A_BYTES;
          const uint32_t full = smem_u32(&bar_full[s]);
          if (corr) {
            mbar_arrive_expect_tx(full, A_BYTES + B_BYTES);
            tma_load_2d(a_dst, &tmApack, kb * BK, m0, full);  // [m; u] rows
            tma_load_2d(b_dst, &tmWc, kb * BK, n0, full);     // W_c rows n0..n0+255
          } else if (kb < kb_half) {
            mbar_arrive_expect_tx(full, A_BYTES + B_BYTES);
            tma_load_2d(a_dst, &tmR, kb * BK, m0, full);                     // r rows
            tma_load_2d(b_dst, &tmWv, kb * BK, n0, full);                    // W_v rows
            tma_load_2d(b_dst + B_BYTES / 2, &tmWg, d + kb * BK, n0, full);  // W_g[:, d:2d] rows
          } else {
            mbar_arrive_expect_tx(full, A_BYTES + B_BYTES / 2);
            tma_load_2d(a_dst, &tmE, (kb - kb_half) * BK, m0, full);                     // e rows
            tma_load_2d(b_dst + B_BYTES / 2, &tmWg, (kb - kb_half) * BK, n0, full);  // W_g[:, :d]
          }
        }
        if (!ok) break;
      }
      if (!ok) {
        raise_abort(&s_abort, p.status);
        volatile int never = 0;  // drain this CTA's own copies still in flight
        const uint32_t first = it > NST ? it - NST : 0;
        for (uint32_t k = first; k < it; ++k)
          mbar_wait_bounded(smem_u32(&bar_full[k % NST]), (k / NST) & 1u, &never);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (uint32_t lt = 0;; ++lt) {
        const uint32_t slot = lt % TILE_SLOTS, sph = (lt / TILE_SLOTS) & 1u;
        if (!mbar_wait_bounded(smem_u32(&bar_tile_full[slot]), sph, &s_abort)) {
          ok = false;
          break;
        }
        const int t = s_tile[slot];
        mbar_arrive(smem_u32(&bar_tile_empty[slot]));
        if (t < 0) break;
        const bool corr = FUSED ? (t % (nt0 + nt1)) < nt0 : t < T0;
        const int nkb = corr ? 2 * kb_half : kb_half + (p.e_dense ? kb_half : 0);
        const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
        if (!mbar_wait_bounded(smem_u32(&bar_tempty[acc]), aph ^ 1u, &s_abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem + acc * ACC_COLS;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const uint32_t s = it % NST, ph = (it / NST) & 1u;
          if (!mbar_wait_bounded(smem_u32(&bar_full[s]), ph, &s_abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_base = base + s * STAGE_BYTES, b_base = a_base + A_BYTES;
          const bool e_part = !corr && kb >= kb_half;
          // K16 steps advance the start address by 32 bytes: + 2 in the descriptor's address field
          const uint64_t adesc0 = sw128_kmajor_desc(a_base);
          const uint64_t bdesc0 = sw128_kmajor_desc(e_part ? b_base + B_BYTES / 2 : b_base);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            if (!e_part)
              tc_mma_bf16(d_tmem, adesc0 + 2u * k, bdesc0 + 2u * k, IDESC_N256, (kb > 0 || k > 0) ? 1u : 0u);
            else
              tc_mma_bf16(d_tmem + 128u, adesc0 + 2u * k, bdesc0 + 2u * k, IDESC_N128, 1u);
          }
          tc_commit(smem_u32(&bar_empty[s]));
        }
        tc_commit(smem_u32(&bar_tfull[acc]));  // accumulator ready (also after a failure)
        if (!ok) break;
      }
      if (!ok) raise_abort(&s_abort, p.status);
    }
    __syncwarp();
  } else if (FUSED && warp == 3) {
    // ---------------- logits stream into the verification ring ----------------
    if (lane == 0) vs_producer(vp, vsm, base + NST * STAGE_BYTES, &s_abort);
    __syncwarp();
  } else if (FUSED && warp == 2) {
    // ---------------- sequence finaliser (bulk copies through staging) ----------------
    vs_finalizer(vp, vsm, base + NST * STAGE_BYTES + kRingBufs * kChunkBytes, blockIdx.x, gridDim.x, lane, &s_abort);
  } else if (warp >= 16) {
    // ---------------- verification bookkeeping (FUSED only) ----------------
    if constexpr (FUSED)
      if (lane == 0) vs_bookkeeper(vp, vsm, &s_abort);
    __syncwarp();
  } else if (warp >= 8) {
    // ---------------- verification (FUSED only: warps 8-15) ----------------
    if constexpr (FUSED)
      vs_consumer(vp, vsm, reinterpret_cast<const uint4*>(dsmem + (base + NST * STAGE_BYTES - smem_u32(dsmem))),
                  warp - 8, lane, &s_abort);
  } else if (warp >= 4) {
    // ---------------- epilogue ----------------
    const int q = (warp - 4) * 32 + lane;  // tile row = TMEM lane
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    // In the overlapped round the epilogue warps have nothing to do until the
    // first rows are packed: they compute W_g[:, :d] e meanwhile.
    if (need_ge) gate_bias_rows(p, d, lane, gemv_next, gemv_done);
    bool have_ge = !need_ge;
    for (uint32_t lt = 0;; ++lt) {
      const uint32_t slot = lt % TILE_SLOTS, sph = (lt / TILE_SLOTS) & 1u;
      bool ok = warp_wait(smem_u32(&bar_tile_full[slot]), sph, &s_abort);
      if (!ok) {
        if (lane == 0) raise_abort(&s_abort, p.status);
        break;
      }
      const int t = s_tile[slot];
      const int tile_rows = s_rows[slot];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_tile_empty[slot]));
      if (t < 0) break;
      bool corr;
      int m0, n0;
      if (FUSED) {
        const int q2 = t / (nt0 + nt1), r2 = t % (nt0 + nt1);
        corr = r2 < nt0;
        m0 = (corr ? q2 : q2 - kGateLag) * BM;
        n0 = corr ? r2 * 256 : (r2 - nt0) * 128;
      } else {
        corr = t < T0;
        const int tt = corr ? t : t - T0;
        m0 = (corr ? tt / nt0 : tt / nt1) * BM;
        n0 = corr ? (tt % nt0) * 256 : (tt % nt1) * 128;
      }
      const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
      ok = warp_wait(smem_u32(&bar_tfull[acc]), aph, &s_abort);
      tc_fence_after();
      if (!ok) {
        if (lane == 0) raise_abort(&s_abort, p.status);
        break;
      }
      if (s_abort) break;
      if (!corr && !have_ge) {
        int got = 1;
        if (lane == 0) got = wait_counter(gemv_done, (uint32_t)d, &s_abort) ? 1 : 0;
        got = __shfl_sync(0xFFFFFFFFu, got, 0);
        if (!got) {
          if (lane == 0) raise_abort(&s_abort, p.status);
          break;
        }
        have_ge = true;
      }
      const int g = m0 + q;
      const bool valid = FUSED ? q < tile_rows : g < R;
      const uint32_t taddr = tmem + acc * ACC_COLS + lane_base;
      if (corr) {
        epilogue_correction<false>(p, taddr, g, valid, n0, d);
        if (p.do_gate) {
          // Publish this warp's 32 rows of the (row block, column block) of r
          // to the gate tiles: one count per epilogue warp, no wait.
          __threadfence();
          fence_proxy_async_global();
          __syncwarp();
          if (lane == 0) atomicAdd(block_done + m0 / BM, 1u);
        }
      } else {
        epilogue_gate<false>(p, taddr, g, valid, n0, d);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_tempty[acc]));
    }
  }
  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// CTA-pair projections: tcgen05.mma.cta_group::2, M = 256 over two SMs
// ---------------------------------------------------------------------------
// A cluster of two CTAs takes a 256-row pair tile, each CTA staging its own 128 rows of A and
// half of the N = 256 weight tile (correction: W_c rows n0.. and n0+128..;
// gate: the W_v rows in the leader, the matching W_g[:, d:2d] rows in the
// follower).  A stage is 128 deep in K (two 64-element swizzle boxes per
// operand, 64 KB per SM): three stages fit.  Each stage costs a fixed
// handshake (full wait, commit, empty wait, copies issued), which deeper
// stages amortise: at B = 256 the kernel took 251.9 us with seven 64-deep
// stages, 245.3 us with three 128-deep ones, 283 us with two 192-deep ones
// and 434 us with fourteen 32-deep ones.
// The leader's MMA thread issues M256 N256 K16 MMAs that read both CTAs'
// shared memory and accumulate into both CTAs' tensor memory (each CTA's
// TMEM lanes are its own 128 rows); its commits arrive on both CTAs'
// barriers (multicast).  Stage-full barriers live in the leader and count the
// bytes of both CTAs' copies.  The leader takes tiles from the global queue
// and hands each to the follower through the follower's shared memory.  A
// per-position e adds k-blocks to the gate tiles: e rows against W_g[:, :d],
// accumulated into the gate's 128 columns (M256 N128 MMAs).  Every wait is
// bounded.
constexpr int PSTAGES = 3;
constexpr int P_THREADS = 256;
constexpr int PBK = 2 * BK;                      // k-block depth of a stage: two swizzle boxes
constexpr int P_BOX_BYTES = 128 * BK * 2;        // 16 KB: one 128-row, 64-element box
constexpr int P_A_BYTES = 2 * P_BOX_BYTES;       // 32 KB: this CTA's 128 rows
constexpr int P_B_BYTES = 2 * P_BOX_BYTES;       // 32 KB: this CTA's half of the weight tile
constexpr int P_STAGE_BYTES = P_A_BYTES + P_B_BYTES;
constexpr int P_SMEM_BYTES = PSTAGES * P_STAGE_BYTES + 1024;  // + slack for 1024-B alignment
constexpr uint32_t IDESC_M256_N256 = idesc_bf16_f32(256, 256);
constexpr uint32_t IDESC_M256_N128 = idesc_bf16_f32(256, 128);
// Pair blocks (256 packed rows) per group of the tile order: inside a group
// the weight tile is the outer index, so the pairs that start together share
// weight tiles as well as row blocks (measured: 260 against 264 us for
// row-block-major order at config 5).
constexpr int kGroupBlocks = 4;
constexpr int P_TILE_SLOTS = 3;  // tile indices in flight: the leader publishes one tile ahead
// A gate tile waits this long for W_g[:, :d] e, of which every CTA of the grid
// computes a share, before its epilogue computes the 128 values of its features
// itself: a share's CTA may not be on an SM yet where kernels of another stream
// hold some, so a tile must not depend on it.  With the GPU to itself the grid is
// resident and the shares take 10 to 50 us (d = 4096 to 8192).
constexpr unsigned long long kGateBiasPatienceNs = 1000000ull;

// GENERAL = false: d a multiple of 256, where every tile is whole, and a broadcast e.  With the
// checks of the general form in its epilogue and MMA loop the kernel took
// 285 instead of 241 us at B = 256 (d = 4096).
template <bool GENERAL>
__global__ void __launch_bounds__(P_THREADS, 1)
    cond_pair_kernel(const __grid_constant__ CUtensorMap tmApack, const __grid_constant__ CUtensorMap tmWc,
                     const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmWv,
                     const __grid_constant__ CUtensorMap tmWg, const __grid_constant__ CUtensorMap tmE,
                     const __grid_constant__ CUtensorMap tmWge, const CondParams p) {
  extern __shared__ uint8_t dsmem[];
  __shared__ __align__(8) uint64_t bar_full[PSTAGES];             // leader: both CTAs' bytes of a stage
  __shared__ __align__(8) uint64_t bar_empty[PSTAGES];            // stage free (leader's commit, both CTAs)
  __shared__ __align__(8) uint64_t bar_tfull[2];                  // accumulator ready (both CTAs)
  __shared__ __align__(8) uint64_t bar_tempty[2];                 // leader: eight epilogue warps done
  __shared__ __align__(8) uint64_t bar_tile_full[P_TILE_SLOTS];   // tile index published (both CTAs)
  __shared__ __align__(8) uint64_t bar_tile_empty[P_TILE_SLOTS];  // leader: ten readers done
  __shared__ int s_tile[P_TILE_SLOTS];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;  // issues the pair's MMAs and runs the tile queue
  const int d = p.d;
  const int nt0 = GENERAL ? (d + 255) / 256 : d / 256, nt1 = GENERAL ? (d + 127) / 128 : d / 128;
  pdl_launch_dependents();
  uint32_t* tile_queue = p.sync + kSyncTileQueue;
  uint32_t* gemv_done = p.sync + kSyncGemvDone;
  uint32_t* block_done = p.block_done;
  const bool need_ge = p.do_gate && !(GENERAL && p.e_dense);

  if (tid == 0) {
    s_abort = 0;
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);  // the leader's expect_tx
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&bar_tfull[a]), 1);
      mbar_init(smem_u32(&bar_tempty[a]), 8);  // four epilogue warps in each CTA
    }
    for (int a = 0; a < P_TILE_SLOTS; ++a) {
      mbar_init(smem_u32(&bar_tile_full[a]), 1);
      mbar_init(smem_u32(&bar_tile_empty[a]), 10);  // MMA + 4 epilogue warps; producer + 4 epilogue warps
    }
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    if (p.do_correct) {
      tma_prefetch_desc(&tmApack);
      tma_prefetch_desc(&tmWc);
    }
    if (p.do_gate) {
      tma_prefetch_desc(&tmR);
      tma_prefetch_desc(&tmWv);
      tma_prefetch_desc(&tmWg);
      if (GENERAL && p.e_dense) {
        tma_prefetch_desc(&tmE);
        tma_prefetch_desc(&tmWge);
      }
    }
  }
  if (warp == 2) {
    tmem_alloc_pair(smem_u32(&s_tmem), TMEM_COLS);  // one warp of each CTA of the pair
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers initialised before any remote arrive
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t base = (smem_u32(dsmem) + 1023u) & ~1023u;
  // k-blocks of the correction (over [m; u], 2d long) and of the gate.  Past the
  // operands' ends (GENERAL) the copies fill zeros.
  const int nkb_g = GENERAL ? (d + PBK - 1) / PBK : d / PBK;
  const int nkb_c = GENERAL ? (2 * d + PBK - 1) / PBK : 2 * nkb_g;
  // The set-up above may overlap the end of the previous kernel (programmatic
  // dependent launch).  R, the packed rows and the row map are its outputs:
  // every role that reads them waits here first.  The gate-bias GEMV (warps
  // 2-3) reads only the inputs and starts at once.  With R = 0 the queue's
  // first claim already ends every role.
  int R = 0, T0 = 0, T1 = 0, X = 0, T = 0, pairs_m = 0;
  if (warp != 2 && warp != 3) {
    pdl_wait();
    R = *(volatile const int32_t*)p.R;
    pairs_m = (R + 2 * BM - 1) / (2 * BM);
    T0 = p.do_correct ? pairs_m * nt0 : 0;
    T1 = p.do_gate ? pairs_m * nt1 : 0;
    // the last wave: work units (a gate tile's worth of MMAs) beyond the
    // whole waves of the pairs
    const int last_wave = (2 * T0 + T1) % (int)(gridDim.x / 2);
    X = last_wave <= p.split_max && (!GENERAL || nkb_g > 1) ? min(last_wave, T1) : 0;
    T = T0 + T1 + X;
  }
  // Tile t: correction tiles first, then gate tiles; within each kind, groups
  // of kGroupBlocks pair blocks with the weight tile outer inside a group.
  // When the last wave of the queue would keep only a few pairs busy (at
  // most split_max tiles), its X gate tiles come as two K halves each (2X
  // queue entries, the halves of a tile next to each other), so that twice
  // as many pairs share it.  At B = 256 (12 pair blocks, 768 units on 76
  // pairs, 8 in the last wave) the kernel went from 245.8-247.9 to
  // 241.7-243.8 us.  Splitting 16 or 38 tiles whatever the last wave made
  // B = 128 slower (141.4 -> 159.8 us), where splitting 4 or 8 left it
  // unchanged.
  struct Tile {
    bool corr;
    int m0, n0;    // this CTA's first row; first output column (correction) or feature (gate)
    int kb0, nkb;  // k-blocks of PBK
    int split;     // -1, or the split tile (0..X-1) whose K half `half` this is
    int half;
  };
  auto decode = [&](int t) {
    Tile x;
    x.corr = t < T0;
    int tt = x.corr ? t : t - T0;
    x.kb0 = 0;
    x.nkb = x.corr ? nkb_c : (GENERAL && p.e_dense) ? 2 * nkb_g : nkb_g;
    x.split = -1;
    x.half = 0;
    if (!x.corr && tt >= T1 - X) {
      const int j = tt - (T1 - X);
      x.split = j >> 1;
      x.half = j & 1;
      tt = T1 - X + x.split;
      x.kb0 = x.half ? nkb_g / 2 : 0;
      x.nkb = x.half ? nkb_g - nkb_g / 2 : nkb_g / 2;
    }
    const int nt = x.corr ? nt0 : nt1;
    const int g = tt / (kGroupBlocks * nt), w = tt - g * kGroupBlocks * nt;
    const int glen = min(kGroupBlocks, pairs_m - g * kGroupBlocks);
    const int pb = g * kGroupBlocks + w % glen;  // pair block
    x.m0 = pb * 2 * BM + (int)rank * BM;         // this CTA's rows
    x.n0 = (w / glen) * (x.corr ? 256 : 128);
    return x;
  };
  // the leader's barriers as seen from either CTA
  auto leader_addr = [&](const void* local) { return map_rank(smem_u32(local), 0); };

  if (warp == 0) {
    // ---------------- tile hand-off + TMA producer (both CTAs) ----------------
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      // While more tiles remain than there are pairs, the leader publishes
      // tile lt + 1 (from the queue) before it loads tile lt, so the next
      // index is already waiting in both CTAs when their producers and the MMA
      // reach the tile switch; near the end of the queue it claims the next
      // tile at the switch, so that no pair holds a tile while others go idle.
      auto publish = [&](uint32_t l, int t) -> bool {
        const uint32_t slot = l % P_TILE_SLOTS, sph = (l / P_TILE_SLOTS) & 1u;
        if (!mbar_wait_cluster_bounded(smem_u32(&bar_tile_empty[slot]), sph ^ 1u, &s_abort)) return false;
        s_tile[slot] = t;
        st_remote_u32(map_rank(smem_u32(&s_tile[slot]), 1), (uint32_t)t);
        mbar_arrive(smem_u32(&bar_tile_full[slot]));
        mbar_arrive_remote(map_rank(smem_u32(&bar_tile_full[slot]), 1));  // release orders the store
        return true;
      };
      auto dequeue = [&]() {
        const int t = (int)atomicAdd(tile_queue, 1u);
        return t < T ? t : -1;
      };
      const int pairs = (int)(gridDim.x / 2);
      if (leader && !publish(0, dequeue())) ok = false;
      for (uint32_t lt = 0; ok; ++lt) {
        const uint32_t slot = lt % P_TILE_SLOTS, sph = (lt / P_TILE_SLOTS) & 1u;
        int t;
        bool ahead = false;  // the leader published tile lt + 1 already
        if (leader) {
          t = s_tile[slot];  // published before
          ahead = t >= 0 && t + pairs < T;
          if (ahead && !publish(lt + 1, dequeue())) {
            ok = false;
            break;
          }
        } else {
          if (!mbar_wait_cluster_bounded(smem_u32(&bar_tile_full[slot]), sph, &s_abort)) {
            ok = false;
            break;
          }
          t = s_tile[slot];
          mbar_arrive_remote(leader_addr(&bar_tile_empty[slot]));
        }
        if (t < 0) break;
        const Tile x = decode(t);
        const bool corr = x.corr;
        const int m0 = x.m0, n0 = x.n0;
        if (!corr && p.do_correct) {
          // the r rows of this CTA's block are written by the correction epilogues
          if (!wait_counter(block_done + m0 / BM, (uint32_t)(4 * nt0), &s_abort)) {
            ok = false;
            break;
          }
          fence_proxy_async_global();
        }
        for (int kb = x.kb0; kb < x.kb0 + x.nkb; ++kb, ++it) {
          const uint32_t s = it % PSTAGES, ph = (it / PSTAGES) & 1u;
          if (!mbar_wait_bounded(smem_u32(&bar_empty[s]), ph ^ 1u, &s_abort)) {
            ok = false;
            break;
          }
          const uint32_t a_dst = base + s * P_STAGE_BYTES, b_dst = a_dst + P_A_BYTES;
          const uint32_t full = leader_addr(&bar_full[s]);
          if (GENERAL && !corr && kb >= nkb_g) {
            // per-position e: the gate's e half, e rows against 128 rows of
            // W_g[:, :d], 64 in each CTA
            if (leader) mbar_arrive_expect_tx(smem_u32(&bar_full[s]), 2 * (P_A_BYTES + P_B_BYTES / 2));
            const int xe = (kb - nkb_g) * PBK;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              tma_load_2d_pair(a_dst + (uint32_t)h * P_BOX_BYTES, &tmE, xe + h * BK, m0, full);
              tma_load_2d_pair(b_dst + (uint32_t)h * P_BOX_BYTES, &tmWge, xe + h * BK, n0 + (int)rank * 64, full);
            }
            continue;
          }
          if (leader) mbar_arrive_expect_tx(smem_u32(&bar_full[s]), 2 * P_STAGE_BYTES);  // both CTAs' bytes
          // [m; u] or r rows; this CTA's half of the weight tile: W_c rows n0..
          // (leader) or n0 + 128.. (follower), or the W_v rows (leader) and the
          // matching W_g[:, d:2d] rows (follower); each as two 64-element boxes
          const CUtensorMap* mb = corr ? &tmWc : (leader ? &tmWv : &tmWg);
          const int xb = (corr || leader) ? kb * PBK : d + kb * PBK;
          const int yb = corr ? n0 + (int)rank * 128 : n0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            tma_load_2d_pair(a_dst + (uint32_t)h * P_BOX_BYTES, corr ? &tmApack : &tmR, kb * PBK + h * BK, m0, full);
            tma_load_2d_pair(b_dst + (uint32_t)h * P_BOX_BYTES, mb, xb + h * BK, yb, full);
          }
        }
        if (!ok) break;
        if (leader && !ahead && !publish(lt + 1, dequeue())) ok = false;  // near the end: claim at the switch
      }
      if (!ok) {
        raise_abort(&s_abort, p.status);
        if (leader) {
          volatile int never = 0;  // wait for the copies in flight into the pair's stages
          const uint32_t first = it > PSTAGES ? it - PSTAGES : 0;
          for (uint32_t k = first; k < it; ++k)
            mbar_wait_bounded(smem_u32(&bar_full[k % PSTAGES]), (k / PSTAGES) & 1u, &never);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader) ----------------
    if (leader && lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (uint32_t lt = 0;; ++lt) {
        const uint32_t slot = lt % P_TILE_SLOTS, sph = (lt / P_TILE_SLOTS) & 1u;
        if (!mbar_wait_bounded(smem_u32(&bar_tile_full[slot]), sph, &s_abort)) {
          ok = false;
          break;
        }
        const int t = s_tile[slot];
        mbar_arrive(smem_u32(&bar_tile_empty[slot]));
        if (t < 0) break;
        const Tile x = decode(t);
        const int nkb = x.nkb;
        const int nkb_full = GENERAL && !x.corr ? min(nkb, nkb_g) : nkb;  // the others: the gate's e half
        const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
        if (!mbar_wait_cluster_bounded(smem_u32(&bar_tempty[acc]), aph ^ 1u, &s_abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem + acc * ACC_COLS;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const uint32_t s = it % PSTAGES, ph = (it / PSTAGES) & 1u;
          if (!mbar_wait_bounded(smem_u32(&bar_full[s]), ph, &s_abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a_base = base + s * P_STAGE_BYTES, b_base = a_base + P_A_BYTES;
          // K16 steps advance the start address by 32 bytes (+ 2 in the
          // descriptor's address field) inside a box, by the box's 16 KB (+ 1024)
          // from the first box to the second
          const uint64_t adesc0 = sw128_kmajor_desc(a_base), bdesc0 = sw128_kmajor_desc(b_base);
#pragma unroll
          for (int k = 0; k < PBK / 16; ++k) {
            const uint64_t step = (uint64_t)((k / (BK / 16)) * (P_BOX_BYTES >> 4) + 2 * (k % (BK / 16)));
            if (!GENERAL || kb < nkb_full)
              tc_mma_pair(d_tmem, adesc0 + step, bdesc0 + step, IDESC_M256_N256, (kb > 0 || k > 0) ? 1u : 0u);
            else  // into the gate's columns only
              tc_mma_pair(d_tmem + 128u, adesc0 + step, bdesc0 + step, IDESC_M256_N128, 1u);
          }
          tc_commit_pair(smem_u32(&bar_empty[s]));  // stage free in both CTAs
        }
        tc_commit_pair(smem_u32(&bar_tfull[acc]));  // accumulator ready (also after a failure)
        if (!ok) break;
      }
      if (!ok) raise_abort(&s_abort, p.status);
    }
    __syncwarp();
  } else if (warp == 2 || warp == 3) {
    // ---------------- W_g[:, :d] e for the broadcast e (idle warps) ----------------
    if (need_ge) {
      const int w = 2 * (int)blockIdx.x + warp - 2, nw = 2 * (int)gridDim.x;
      gate_bias_share(p.e, p.Wg, p.ge, d, 2 * d, w, nw, lane);
      pdl_wait();  // the counters are zero from here on
      __threadfence();
      __syncwarp();
      if (lane == 0 && w < d) atomicAdd(gemv_done, (uint32_t)((d - w + nw - 1) / nw));
    }
  } else {
    // ---------------- epilogue (warps 4-7 of both CTAs) ----------------
    const int q = (warp - 4) * 32 + lane;  // tile row = TMEM lane
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    bool have_ge = !need_ge;
    unsigned long long patience = kGateBiasPatienceNs;
    for (uint32_t lt = 0;; ++lt) {
      const uint32_t slot = lt % P_TILE_SLOTS, sph = (lt / P_TILE_SLOTS) & 1u;
      bool ok = warp_wait_cluster(smem_u32(&bar_tile_full[slot]), sph, &s_abort);
      if (!ok) {
        if (lane == 0) raise_abort(&s_abort, p.status);
        break;
      }
      const int t = s_tile[slot];
      __syncwarp();
      if (lane == 0) {
        if (leader) mbar_arrive(smem_u32(&bar_tile_empty[slot]));
        else mbar_arrive_remote(leader_addr(&bar_tile_empty[slot]));
      }
      if (t < 0) break;
      const Tile x = decode(t);
      const bool corr = x.corr;
      const int m0 = x.m0, n0 = x.n0;
      const uint32_t acc = lt & 1u, aph = (lt >> 1) & 1u;
      ok = warp_wait(smem_u32(&bar_tfull[acc]), aph, &s_abort);
      tc_fence_after();
      if (!ok) {
        if (lane == 0) raise_abort(&s_abort, p.status);
        break;
      }
      if (s_abort) break;
      if (!corr && !have_ge) {
        int got = 1;
        if (lane == 0) got = wait_counter(gemv_done, (uint32_t)d, &s_abort, patience) ? 1 : 0;
        have_ge = __shfl_sync(0xFFFFFFFFu, got, 0) != 0;
        if (!have_ge) {
          if (__shfl_sync(0xFFFFFFFFu, s_abort, 0)) break;
          patience = 0ull;  // of this warp's later tiles
          // (every warp of the tile, and the share's owner, write the same bits)
          gate_bias_features(p, d, n0, lane);
        }
      }
      const int g = m0 + q;
      const bool valid = g < R;
      const uint32_t taddr = tmem + acc * ACC_COLS + lane_base;
      if (corr) {
        epilogue_correction<GENERAL>(p, taddr, g, valid, n0, d);
        if (p.do_gate) {
          __threadfence();
          fence_proxy_async_global();
          __syncwarp();
          if (lane == 0) atomicAdd(block_done + m0 / BM, 1u);
        }
      } else if (x.split < 0) {
        epilogue_gate<GENERAL>(p, taddr, g, valid, n0, d);
      } else {
        // A K half: this row's accumulator goes to the half's slot ([column][row]
        // per CTA, so that a warp's stores are contiguous); the warp that counts
        // second on the ticket of its 32 rows adds the other half's slot and
        // runs the epilogue.  Fence before the count, fence after it (the
        // last-arriver pattern): no wait on the other pair.
        const size_t slot_floats = (size_t)2 * BM * 128;
        float* own = p.split_part + ((size_t)(x.split * 2 + x.half) * 2 + rank) * slot_floats + q;
        const float* other = p.split_part + ((size_t)(x.split * 2 + (x.half ^ 1)) * 2 + rank) * slot_floats + q;
        for (int cc = 0; cc < 8; ++cc) {
          float c[32];
          tmem_ld_32cols(taddr + (uint32_t)(cc * 32), c);
#pragma unroll
          for (int i = 0; i < 32; ++i) __stcg(own + (cc * 32 + i) * 128, c[i]);
        }
        __threadfence();
        __syncwarp();
        uint32_t before = 0;
        if (lane == 0) {
          before = atomicAdd(p.split_ticket + x.split * 8 + (int)rank * 4 + (warp - 4), 1u);
          __threadfence();
        }
        before = __shfl_sync(0xFFFFFFFFu, before, 0);
        __syncwarp();
        if (before == 1u) epilogue_gate<GENERAL>(p, taddr, g, valid, n0, d, other);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) mbar_arrive(smem_u32(&bar_tempty[acc]));
        else mbar_arrive_remote(leader_addr(&bar_tempty[acc]));
      }
    }
  }
  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer is done with this CTA's shared and tensor memory
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

// One thread runs the pipelined kernels' bounded waits on a condition the
// caller controls (retrace_wait_selftest): kind 0 waits until *flag >= target
// (the counter wait), kind 1 for an mbarrier phase that completes only if
// target == 0 (the phase wait).  An expired wait sets the status flag, as in
// the kernels, and the kernel returns.
__global__ void wait_selftest_kernel(int kind, const uint32_t* flag, uint32_t target, uint32_t* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ volatile int s_abort;
  if (threadIdx.x != 0) return;
  s_abort = 0;
  bool ok;
  if (kind == 0) {
    ok = wait_counter(flag, target, &s_abort);
  } else {
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
    if (target == 0) mbar_arrive(smem_u32(&bar));  // phase 0 completes: the wait returns at once
    ok = mbar_wait_bounded(smem_u32(&bar), 0, &s_abort);
  }
  if (!ok) atomicOr(status, kFlagWaitTimeout);
}

// ---------------------------------------------------------------------------
// Small R (cond_small_r): the weights on the M side
// ---------------------------------------------------------------------------
// With few rows the 256-row pair tiles are mostly padding and only d/256
// correction tiles exist, so a handful of SMs stream the weights.  Here the
// GEMMs run transposed: c^T = W_c [m; u]^T and [v; g_r]^T = [W_v; W_g,r] r^T,
// the weights as the A operand in 128-row tiles (M = 128, no padding), the
// rows as B in tiles of up to 256, and the K range split so that about one
// resident wave of CTAs streams the weights.
//
// The S K-splits of one (weight tile, row tile) unit run as one cluster of S
// CTAs.  Each CTA accumulates its k-range in TMEM, moves the fp32 partial into
// its own shared memory (the drained pipeline stages), and after a cluster
// barrier sums its slice of the rows over the S partials through distributed
// shared memory, in rank order (results repeat bit for bit), and applies the
// epilogue: r = m + beta c (Eq. 7) for the correction tiles of W_c, or the
// gated fusion e~ = e + v sigmoid(g_r + W_g[:, :d] e) (Eq. 8) for the gate
// tiles, whose 128 weight rows stack 64 rows of W_v over the same 64 rows of
// W_g[:, d:2d] (v and g_r of a feature in TMEM lanes f and 64 + f).  With a
// per-position e the gate has three products of d-long rows, W_v r, W_g,r r and
// W_g,e e: a cluster then holds 128 features of all three, each product in
// its own CTAs (S = 3 splits), and the sum adds the last two.  (As further
// k-blocks of the stacked tiles, W_v's half zeros, a gate tile had twice the
// k-blocks on as many CTAs: 36 us at B = 32, d = 2560.)  Nothing goes through
// global partials and no reduction kernel follows.  The partial is stored row-major ([row][feature]) so that both the TMEM drain and the
// cluster's reads move whole 128- and 256-byte rows.
//
// The row tiles are cut on the device from R (swap_cut): as many as the
// resident clusters can take side by side, so that every SM has work and a
// k-block costs an SM little more than its 16 KB of weights (a stage goes
// through shared memory twice, about 2 (128 + N) cycles at 128 B per clock).
constexpr int SW_STAGES = 8;      // most pipeline stages
constexpr int SW_MIN_BLOCKS = 4;  // least k-blocks of a split
constexpr int SW_THREADS = 256;
constexpr int SW_A_BYTES = BM * BK * 2;  // 16 KB: 128 weight rows of a k-block
constexpr int SW_ROW_STEP = 32;          // row boxes come in multiples of this many rows
constexpr int SW_ROW_MAPS = 256 / SW_ROW_STEP;
// Dynamic shared memory of a CTA at most (its barriers beside it): four stages
// with a box of 256 rows.  With more, CTAs that sit beside verification's leave
// it too little L1 and room (rounds of B = 64, d = 2560: 102 us, 110 at 208 KB and
// above), though their own loop gains from a fifth stage at 192 rows.
constexpr int SW_SMEM_RING = 198 * 1024;
// The gate's where no verification kernel is launched ahead beside it.
constexpr int SW_SMEM_MAX = 222 * 1024;
// Largest d at which the correction's idle warps compute W_g[:, :d] e.  They keep 24
// KB per SM in flight, so above it they outlast the correction (d = 8192: 103 us of
// a correction that takes 56 without them) and a launch of its own runs beside
// it.  Rounds, V = 32000, B = 1 / 8 / 16, us, in idle warps and alone: d = 4096: 52
// / 61 / 70 and 49 / 61 / 71; 4608: 62 / 72 / 80 and 56 / 71 / 78; 6144: 106 / 111 /
// 119 and 91 / 104 / 113; 8192: 161 / 164 / 175 and 133 / 153 / 162.
constexpr int kGateBiasAlone = 4096;

// Row tiles of R rows for `clusters` resident clusters over `mtiles` weight
// tiles: `ntiles` tiles of `tile_n` rows (a multiple of 16, at most 256).
// The units u < mtiles * ntiles (weight tile u % mtiles) are taken by cluster
// u mod clusters.
struct SwapCut {
  int ntiles, tile_n;
};
__host__ __device__ __forceinline__ SwapCut swap_cut(int R, int mtiles, int clusters) {
  const int nrows = (R + 15) / 16 * 16;
  if (clusters < 2 * mtiles && nrows <= 256) return {nrows > 0 ? 1 : 0, nrows};  // one tile
  const int need = (nrows + 255) / 256;
  const int fit = clusters / mtiles, most = (nrows + SW_ROW_STEP - 1) / SW_ROW_STEP;
  int n = fit < most ? fit : most;
  if (n < need) n = need;
  if (n < 1) n = 1;
  SwapCut c;
  c.tile_n = ((nrows + n - 1) / n + 15) / 16 * 16;
  c.ntiles = c.tile_n > 0 ? (nrows + c.tile_n - 1) / c.tile_n : 0;
  return c;
}
__host__ __device__ __forceinline__ int swap_box_rows(int tile_n) {
  return (tile_n + SW_ROW_STEP - 1) / SW_ROW_STEP * SW_ROW_STEP;
}
// Pipeline stages (a weight tile and a row box each) that `bytes` of shared memory hold.
__host__ __device__ __forceinline__ int swap_stages(int bytes, int box_rows) {
  const int n = bytes / (SW_A_BYTES + box_rows * BK * 2);
  return n < SW_STAGES ? n : SW_STAGES;
}

// The rows operand once per box height: map i has boxes of SW_ROW_STEP (i + 1) rows.
struct RowMaps {
  CUtensorMap m[SW_ROW_MAPS];
};

// A round of few sequences without packed rows (DIRECT).  Sequence b has the KP
// tile rows from b KP on (KP = K - 1 rounded up to 8; those past n_b compute
// nothing that is stored), so the row tile's size is known on the host, and
// the correction reads the carried rows where they lie: m_j and u_j of a
// sequence are consecutive rows of hD and hT, one box per sequence and k-block.
// Every warp finds the accepted lengths for itself from the argmax keys, so
// no kernel stands between verification and the correction.  Warps 2-7 of the
// correction write the outputs of verification and the rows j >= n_b of e~, the
// gate's first CTA zeroes the keys.
struct DirectRows {
  int B, K, KP;
  unsigned long long* keys;  // argmax keys of the verification (NULL: accept_len is given)
  const int32_t* draft;
  int32_t* accept_len;
  int32_t* committed;
  int32_t* bonus;
  int32_t* n_out;            // optional
  const __nv_bfloat16* hD;   // m, for the correction's epilogue
  const __nv_bfloat16* e;
  __nv_bfloat16* e_out;
};
constexpr int kDirectChunks = 3;  // (sequence, row) pairs per lane: B K <= 32 * kDirectChunks

// Accepted length of sequence `lane` (lanes below B; the others return K): the
// whole warp.  Read from accept_len once decided, else from the keys: the
// first of the K drafts that is not its row's argmax, from ballots over 32
// (sequence, row) pairs at a time.  The draft tokens are inputs, read before
// the wait on verification.
struct DirectDrafts {
  int tok[kDirectChunks];  // of (sequence, row) pair 32 c + lane
};
__device__ __forceinline__ DirectDrafts direct_drafts(const DirectRows& q, int lane) {
  DirectDrafts t;
#pragma unroll
  for (int c = 0; c < kDirectChunks; ++c) t.tok[c] = c * 32 + lane < q.B * q.K ? __ldg(q.draft + c * 32 + lane) : -1;
  return t;
}
__device__ __forceinline__ int direct_accepted(const DirectRows& q, const DirectDrafts& t, bool decided, int lane) {
  const int B = q.B, K = q.K;
  if (decided) {
    const int A = lane < B ? __ldcg(q.accept_len + lane) : K;
    return min(max(A, 0), K);
  }
  bool miss[kDirectChunks];
#pragma unroll
  for (int c = 0; c < kDirectChunks; ++c) {
    const int x = c * 32 + lane, b = x / K;
    miss[c] = x < B * K && (int)key_index(__ldcg(q.keys + (long long)b * (K + 1) + (x - b * K))) != t.tok[c];
  }
  int A = K;
#pragma unroll
  for (int c = 0; c < kDirectChunks; ++c) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, miss[c]);
    const int lo = lane * K - c * 32, hi = lo + K;  // this sequence's rows in the chunk
    if (lane < B && A == K && lo < 32 && hi > 0) {
      const unsigned above = lo > 0 ? ~0u << lo : ~0u, below = hi < 32 ? (1u << hi) - 1u : ~0u;
      const unsigned own = m & above & below;
      if (own) A = __ffs(own) - 1 - lo;
    }
  }
  return A;
}

enum { kCorrect = 0, kGateStacked = 1, kGateParts = 2 };
struct SwapClusterParams {
  const int32_t* R;
  int d;
  int mtiles;  // weight tiles
  int nkb;     // 64-deep k-blocks of the GEMM
  int nkb_m;   // DIRECT correction: those of the m half
  int S;       // cluster size: K splits, or 3 times them (kGateParts)
  int gate;    // kCorrect: tiles of W_c (128 features); kGateStacked: [W_v; W_g,r] tiles (64 features);
               // kGateParts: per-position e, W_v, W_g,r and W_g,e tiles (128 features each)
  int stage_bytes;  // shared memory of the pipeline stages
  int pre;          // stages whose weight tiles are loaded before the wait on the previous kernel
  int row_maps;     // maps of the rows operand
  uint32_t tmem_cols;
  // correction epilogue
  const __nv_bfloat16* apack;  // m = the first d columns of each packed row
  float beta;
  __nv_bfloat16* r_out;
  int compact_out;
  GateBiasParams bias;  // correction: W_g[:, :d] e of the gate to come (ge NULL: not computed)
  // gate epilogue.  kGateStacked: e [d], and ge = W_g[:, :d] e, complete before
  // this launch; kGateParts: e packed rows [R, d].
  const __nv_bfloat16* e;
  const float* ge;
  __nv_bfloat16* e_out;
  const int32_t* rowmap;
  uint32_t* status;
  DirectRows direct;  // DIRECT only
};

// The sum over the cluster's S partials and the epilogue of `total` positions
// (row l0 + x / 32, features 4 (x % 32).. for the correction; 16 per row for
// the gate) of the unit at weight tile mt and packed row row0.  A thread has NB
// positions and, for each, the loads of NS partials in flight: with one
// position and one partial at a time a CTA with 80 rows took a chain of
// twenty round trips.  The partials are added in rank order.
template <bool DIRECT, int NB, int NS>
__device__ __forceinline__ void swap_correction_rows(const SwapClusterParams& p, uint32_t P, int mt, int row0, int l0,
                                                     int total, const int* s_A) {
  const int d = p.d, S = p.S, n0 = mt * 128;
  for (int x0 = threadIdx.x; x0 < total; x0 += NB * SW_THREADS) {
    float4 c[NB];
    uint2 mw[NB];
    long long orow[NB];
    uint32_t at[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      // (features past d, in the last tile: d + 127 < 2 d keeps their loads inside the packed rows)
      const int x = min(x0 + q * SW_THREADS, total - 1), l = l0 + x / 32, f = (x % 32) * 4, g = row0 + l;
      if constexpr (DIRECT) {
        const int b = l / p.direct.KP, j = l - b * p.direct.KP, A = s_A[b];
        orow[q] = j < p.direct.K - 1 - A && n0 + f < d ? l : -1;
        if (orow[q] >= 0)
          mw[q] = __ldg(reinterpret_cast<const uint2*>(p.direct.hD + ((long long)b * p.direct.K + A + 1 + j) * d + n0 + f));
      } else {
        mw[q] = __ldcg(reinterpret_cast<const uint2*>(p.apack + (long long)g * 2 * d + n0 + f));
        orow[q] = n0 + f >= d ? -1 : p.compact_out ? g : __ldcg(p.rowmap + g);
      }
      at[q] = P + (uint32_t)(l * 512 + f * 4);
      c[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int s0 = 0; s0 < S; s0 += NS) {
      float4 v[NS][NB];
#pragma unroll
      for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int q = 0; q < NB; ++q)
          v[s][q] = s0 + s < S ? ld_cluster_f4(map_rank(at[q], (uint32_t)(s0 + s))) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int q = 0; q < NB; ++q) add4(c[q], v[s][q]);
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int x = x0 + q * SW_THREADS;
      if (x < total && orow[q] >= 0)
        *reinterpret_cast<uint2*>(p.r_out + orow[q] * d + n0 + (x % 32) * 4) =
            make_uint2(pack_bf16x2(bf16_lo(mw[q].x) + p.beta * c[q].x, bf16_hi(mw[q].x) + p.beta * c[q].y),
                       pack_bf16x2(bf16_lo(mw[q].y) + p.beta * c[q].z, bf16_hi(mw[q].y) + p.beta * c[q].w));
    }
  }
}
template <bool DIRECT, int NB, int NS>
__device__ __forceinline__ void swap_gate_rows(const SwapClusterParams& p, uint32_t P, int mt, int row0, int l0,
                                               int total, const int* s_A) {
  const int d = p.d, S = p.S;
  const int f = ((int)threadIdx.x % 16) * 4, n = mt * 64 + f;  // the same features at every step
  if (n >= d) return;  // past the last feature (no barrier below)
  const float4 gb = __ldcg(reinterpret_cast<const float4*>(p.ge + n));
  const uint2 ew = __ldg(reinterpret_cast<const uint2*>(p.e + n));
  for (int x0 = threadIdx.x; x0 < total; x0 += NB * SW_THREADS) {
    float4 v[NB], a[NB];
    long long orow[NB];
    uint32_t at[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int l = l0 + min(x0 + q * SW_THREADS, total - 1) / 16;
      if constexpr (DIRECT) {
        const int b = l / p.direct.KP, j = l - b * p.direct.KP;
        orow[q] = j < p.direct.K - 1 - s_A[b] ? (long long)b * p.direct.K + j : -1;
      } else {
        orow[q] = __ldcg(p.rowmap + row0 + l);
      }
      at[q] = P + (uint32_t)(l * 512 + f * 4);
      v[q] = a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int s0 = 0; s0 < S; s0 += NS) {
      float4 xv[NS][NB], xa[NS][NB];
#pragma unroll
      for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          const bool in = s0 + s < S;
          const uint32_t src = map_rank(at[q], (uint32_t)(in ? s0 + s : 0));
          xv[s][q] = in ? ld_cluster_f4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
          xa[s][q] = in ? ld_cluster_f4(src + 256u) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
      for (int s = 0; s < NS; ++s)
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          add4(v[q], xv[s][q]);
          add4(a[q], xa[s][q]);
        }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if (x0 + q * SW_THREADS >= total || (DIRECT && orow[q] < 0)) continue;
      const float s0 = fast_sigmoid(a[q].x + gb.x), s1 = fast_sigmoid(a[q].y + gb.y);
      const float s2 = fast_sigmoid(a[q].z + gb.z), s3 = fast_sigmoid(a[q].w + gb.w);
      *reinterpret_cast<uint2*>(p.e_out + orow[q] * d + n) =
          make_uint2(pack_bf16x2(bf16_lo(ew.x) + v[q].x * s0, bf16_hi(ew.x) + v[q].y * s1),
                     pack_bf16x2(bf16_lo(ew.y) + v[q].z * s2, bf16_hi(ew.y) + v[q].w * s3));
    }
  }
}

// kGateParts: v is the sum of the first third of the cluster's partials, the
// gate that of the others.
__device__ __forceinline__ void swap_parts_rows(const SwapClusterParams& p, uint32_t P, int mt, int row0, int l0,
                                                int total) {
  constexpr int NB = 4;
  const int d = p.d, S = p.S;
  for (int x0 = threadIdx.x; x0 < total; x0 += NB * SW_THREADS) {
    float4 v[NB], a[NB];
    uint2 ew[NB];
    long long orow[NB];
    uint32_t at[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int x = min(x0 + q * SW_THREADS, total - 1), l = l0 + x / 32, f = (x % 32) * 4, n = mt * 128 + f;
      orow[q] = n < d ? __ldcg(p.rowmap + row0 + l) : -1;
      ew[q] = n < d ? __ldcg(reinterpret_cast<const uint2*>(p.e + (long long)(row0 + l) * d + n)) : make_uint2(0u, 0u);
      at[q] = P + (uint32_t)(l * 512 + f * 4);
      v[q] = a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int s = 0; s < S / 3; ++s) {
      float4 x[3][NB];
#pragma unroll
      for (int part = 0; part < 3; ++part)
#pragma unroll
        for (int q = 0; q < NB; ++q) x[part][q] = ld_cluster_f4(map_rank(at[q], (uint32_t)(part * (S / 3) + s)));
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        add4(v[q], x[0][q]);
        add4(a[q], x[1][q]);
        add4(a[q], x[2][q]);
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int x = x0 + q * SW_THREADS;
      if (x >= total || orow[q] < 0) continue;
      const float s0 = fast_sigmoid(a[q].x), s1 = fast_sigmoid(a[q].y);
      const float s2 = fast_sigmoid(a[q].z), s3 = fast_sigmoid(a[q].w);
      *reinterpret_cast<uint2*>(p.e_out + orow[q] * d + mt * 128 + (x % 32) * 4) =
          make_uint2(pack_bf16x2(bf16_lo(ew[q].x) + v[q].x * s0, bf16_hi(ew[q].x) + v[q].y * s1),
                     pack_bf16x2(bf16_lo(ew[q].y) + v[q].z * s2, bf16_hi(ew[q].y) + v[q].w * s3));
    }
  }
}

template <bool DIRECT>
__global__ void __launch_bounds__(SW_THREADS, 1)
    swap_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmA2,
                        const __grid_constant__ CUtensorMap tmA3, const __grid_constant__ RowMaps tmB,
                        const __grid_constant__ RowMaps tmE, const SwapClusterParams p) {
  extern __shared__ uint8_t dsmem[];
  __shared__ __align__(8) uint64_t bar_full[SW_STAGES];
  __shared__ __align__(8) uint64_t bar_empty[SW_STAGES];
  __shared__ __align__(8) uint64_t bar_acc;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ int s_A[32];  // DIRECT: the sequences' accepted lengths
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.S, d = p.d;
  const uint32_t rank = cluster_rank();
  const int cid = (int)(blockIdx.x / (unsigned)S), clusters = (int)(gridDim.x / (unsigned)S);
  pdl_launch_dependents();
  if (threadIdx.x < SW_STAGES) {
    mbar_init(smem_u32(&bar_full[threadIdx.x]), 2);  // the weight tile's and the row box's expect_tx
    mbar_init(smem_u32(&bar_empty[threadIdx.x]), 1);
    if (threadIdx.x == 0) {
      s_abort = 0;
      mbar_init(smem_u32(&bar_acc), 1);
    }
    fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmA2);
  }
  if (warp == 1 && lane < p.row_maps) {
    tma_prefetch_desc(&tmB.m[lane]);
    if (p.gate == kGateParts) tma_prefetch_desc(&tmE.m[lane]);
  }
  if (warp == 2) {
    tmem_alloc(smem_u32(&s_tmem), p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t base = (smem_u32(dsmem) + 1023u) & ~1023u;
  // the partial [row][128 features], in the drained pipeline stages (the same offset in every CTA)
  float* P = reinterpret_cast<float*>(dsmem + (base - smem_u32(dsmem)));
  // this CTA's product (kGateParts) and k-blocks
  const int splits = p.gate == kGateParts ? S / 3 : S;
  const int part = (int)rank / splits, split = (int)rank - part * splits;
  const int kb0 = (int)((long long)split * p.nkb / splits), kb1 = (int)((long long)(split + 1) * p.nkb / splits);
  // Weight tiles lie at 16 KB steps from `base`, whatever the row boxes' size.
  auto load_a = [&](int mt, int kb, uint32_t s) {
    const uint32_t a_dst = base + s * (uint32_t)SW_A_BYTES, bar = smem_u32(&bar_full[s]);
    mbar_arrive_expect_tx(bar, (uint32_t)SW_A_BYTES);
    if (DIRECT && !p.gate) {  // W_c's m columns, then its u columns
      const bool u = kb >= p.nkb_m;
      tma_load_2d(a_dst, u ? &tmA2 : &tmA, (u ? kb - p.nkb_m : kb) * BK, mt * 128, bar);
    } else if (p.gate == kGateStacked) {  // rows 0-63: W_v rows f0..; rows 64-127: the same rows of W_g[:, d:2d]
      tma_load_2d(a_dst, &tmA, kb * BK, mt * 64, bar);
      tma_load_2d(a_dst + (uint32_t)(SW_A_BYTES / 2), &tmA2, d + kb * BK, mt * 64, bar);
    } else if (p.gate == kGateParts) {
      tma_load_2d(a_dst, part == 0 ? &tmA : part == 1 ? &tmA2 : &tmA3, (part == 1 ? d : 0) + kb * BK, mt * 128, bar);
    } else {
      tma_load_2d(a_dst, &tmA, kb * BK, mt * 128, bar);
    }
  };
  // The weights are inputs: the producer loads the first stages' tiles of the
  // cluster's first unit before the wait on the previous kernel, and their
  // row boxes after it.
  const int npre = min(p.pre, kb1 - kb0);
  if (warp == 0 && lane == 0)
    for (int i = 0; i < npre; ++i) load_a(cid % p.mtiles, kb0 + i, (uint32_t)i);  // every stage is free at the start
  // The gate's W_g[:, :d] e needs inputs only: warps 2-7, which have no work
  // before the accumulator is complete, compute it while the previous kernels
  // end (the memory is idle then) and the first k-blocks run.
  if (p.bias.ge && warp >= 2)
    gate_bias_share(p.bias.e, p.bias.Wg, p.bias.ge, d, 2 * d, (int)blockIdx.x * 6 + warp - 2, (int)gridDim.x * 6, lane);
  DirectDrafts drafts;
  if (DIRECT && !p.gate && p.direct.keys) drafts = direct_drafts(p.direct, lane);
  pdl_wait();  // R and the activation rows come from the previous kernels
  int R;
  SwapCut cut;
  int my_A = 0, boxes = 0;  // DIRECT: accepted length of sequence `lane`; sequences with carried rows
  if constexpr (DIRECT) {
    const DirectRows& q = p.direct;
    my_A = direct_accepted(q, drafts, p.gate || !q.keys, lane);
    boxes = __popc(__ballot_sync(0xFFFFFFFFu, my_A < q.K - 1));
    R = q.B * q.KP;
    cut = {boxes > 0 ? 1 : 0, (R + 15) / 16 * 16};
    if (warp == 0) s_A[lane] = my_A;  // for the epilogue, a block barrier later
    if (warp >= 2) {
      const int w = (int)blockIdx.x * 6 + warp - 2, nw = (int)gridDim.x * 6;
      if (!p.gate) {
        // the outputs of verification, and the rows of e~ that carry nothing
        if (q.keys) {
          for (int b = w; b < q.B; b += nw) {
            const int A = __shfl_sync(0xFFFFFFFFu, my_A, b);
            const unsigned long long* key = q.keys + (long long)b * (q.K + 1);
            for (int i = lane; i <= q.K; i += 32) q.committed[(long long)b * (q.K + 1) + i] = i <= A ? (int)key_index(__ldcg(key + i)) : -1;
            if (lane == 0) {
              q.accept_len[b] = A;
              q.bonus[b] = (int)key_index(__ldcg(key + A));
              if (q.n_out) q.n_out[b] = max(0, q.K - 1 - A);
            }
          }
        }
        for (int x = w; x < q.B * q.K; x += nw) {
          const int b = x / q.K, j = x - b * q.K;
          if (j < q.K - 1 - __shfl_sync(0xFFFFFFFFu, my_A, b)) continue;  // the gate writes it
          const uint4* src = reinterpret_cast<const uint4*>(q.e);
          uint4* dst = reinterpret_cast<uint4*>(q.e_out + (long long)x * d);
          for (int v = lane; v < d / 8; v += 32) dst[v] = __ldg(src + v);
        }
      } else if (blockIdx.x == 0 && q.keys) {
        for (int x = threadIdx.x - 64; x < q.B * (q.K + 1); x += SW_THREADS - 64) q.keys[x] = 0ull;
      }
    }
  } else {
    R = *(volatile const int32_t*)p.R;
    cut = swap_cut(R, p.mtiles, clusters);
  }
  const int units = p.mtiles * cut.ntiles;
  const int box = swap_box_rows(cut.tile_n);
  const int nst = swap_stages(p.stage_bytes, box > 0 ? box : SW_ROW_STEP);  // >= p.pre
  const uint32_t b_bytes = (uint32_t)(box * BK * 2);
  const uint32_t b_base = base + (uint32_t)nst * (uint32_t)SW_A_BYTES;
  const CUtensorMap* mb = &(part == 2 ? tmE : tmB).m[box > 0 ? box / SW_ROW_STEP - 1 : 0];

  if (cid >= units && warp == 0 && lane == 0) {  // (always so with R = 0)
    // no unit: let the copies issued above land before the CTA leaves
    volatile int never = 0;
    for (int i = 0; i < npre; ++i) {
      mbar_arrive(smem_u32(&bar_full[i]));
      mbar_wait_bounded(smem_u32(&bar_full[i]), 0u, &never);
    }
  }
  uint32_t s = 0, ph = 0;  // ring position and phase of the next k-block (producer and MMA thread)
  auto advance = [&]() {
    if (++s == (uint32_t)nst) {
      s = 0;
      ph ^= 1u;
    }
  };
  uint32_t acc_ph = 0u;  // phase of bar_acc
  int pre = npre;        // weight tiles of this unit already loaded
  for (int u = cid; u < units; u += clusters, acc_ph ^= 1u, pre = 0) {
    const int mt = u % p.mtiles, nt = u / p.mtiles;
    const int row0 = nt * cut.tile_n;
    const int rows = min(R - row0, cut.tile_n);  // of this unit, > 0
    const int mma_n = (rows + 15) / 16 * 16;
    if (warp == 0) {
      // ---------------- TMA producer ----------------
      if (lane == 0 || (DIRECT && !p.gate)) {
        int i = 0;
        for (; i < kb1 - kb0; ++i, advance()) {
          if constexpr (DIRECT) {
            if (!p.gate) {  // the whole warp: lane 0 the weights, lane b the rows of sequence b
              int ok = 1;
              if (lane == 0) {
                if (i >= pre) {
                  ok = mbar_wait_bounded(smem_u32(&bar_empty[s]), ph ^ 1u, &s_abort) ? 1 : 0;
                  if (ok) load_a(mt, kb0 + i, s);
                }
                if (ok) mbar_arrive_expect_tx(smem_u32(&bar_full[s]), (uint32_t)(boxes * p.direct.KP * BK * 2));
              }
              if (!__shfl_sync(0xFFFFFFFFu, ok, 0)) break;
              if (my_A < p.direct.K - 1) {  // (lanes past B have my_A = K)
                const int kb = kb0 + i;
                const bool u = kb >= p.nkb_m;
                tma_load_2d(b_base + s * b_bytes + (uint32_t)(lane * p.direct.KP * BK * 2), &tmB.m[u ? 1 : 0],
                            (u ? kb - p.nkb_m : kb) * BK, lane * p.direct.K + my_A + (u ? 0 : 1), smem_u32(&bar_full[s]));
              }
              continue;
            }
          }
          if (i >= pre) {
            if (!mbar_wait_bounded(smem_u32(&bar_empty[s]), ph ^ 1u, &s_abort)) break;
            load_a(mt, kb0 + i, s);
          }
          mbar_arrive_expect_tx(smem_u32(&bar_full[s]), b_bytes);
          tma_load_2d(b_base + s * b_bytes, mb, (kb0 + i) * BK, row0, smem_u32(&bar_full[s]));
        }
        if (i < kb1 - kb0 && lane == 0) {
          // a wait expired: flag it, let the copies in flight land
          raise_abort(&s_abort, p.status);
          volatile int never = 0;
          for (int k = 0; k < min(i, nst); ++k) {  // the last min(i, nst) k-blocks, backwards
            ph ^= s == 0 ? 1u : 0u;
            s = s == 0 ? (uint32_t)nst - 1u : s - 1u;
            mbar_wait_bounded(smem_u32(&bar_full[s]), ph, &never);
          }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------- MMA issuer ----------------
      // (the whole warp waits, one lane issues: 1.5 % of a round against a loop in lane 0)
      const uint32_t idesc = idesc_bf16_f32(128, mma_n);
      bool ok = true;
      for (int i = 0; i < kb1 - kb0; ++i, advance()) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(smem_u32(&bar_full[s]), ph, &s_abort));
        if (!ok) break;
        tc_fence_after();
        const uint64_t adesc0 = sw128_kmajor_desc(base + s * (uint32_t)SW_A_BYTES);
        const uint64_t bdesc0 = sw128_kmajor_desc(b_base + s * b_bytes);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            tc_mma_bf16(tmem, adesc0 + 2u * k, bdesc0 + 2u * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
          tc_commit(smem_u32(&bar_empty[s]));
        }
        __syncwarp();
      }
      if (!ok && lane == 0) raise_abort(&s_abort, p.status);
      if (elect_one()) tc_commit(smem_u32(&bar_acc));  // accumulator ready (also after a failure)
      __syncwarp();
    }
    // ---------------- the partial into shared memory (every warp) ----------------
    {
      // weight row of the tile = TMEM lane = feature; a warp reaches the lanes
      // 32 (warp % 4) .. + 31: warps 4-7 take the first half of the columns
      const int q = (warp & 3) * 32 + lane;
      const bool ok = warp_wait(smem_u32(&bar_acc), acc_ph, &s_abort);
      tc_fence_after();
      if (!ok && lane == 0) raise_abort(&s_abort, p.status);
      if (ok && !s_abort) {
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int chunks = (mma_n + 31) / 32, half = (chunks + 1) / 2;
        const int ch0 = warp >= 4 ? 0 : half, ch1 = warp >= 4 ? half : chunks;
        for (int c0 = ch0 * 32; c0 < ch1 * 32; c0 += 32) {
          float v[32];
          tmem_ld_32cols(taddr + (uint32_t)c0, v);
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (c0 + j < mma_n) P[(c0 + j) * 128 + q] = v[j];  // a warp stores 128 contiguous bytes
        }
      }
    }
    // ---------------- the cluster's sum and the epilogue ----------------
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool go = !s_abort;  // every role is done with the unit: the same in every thread of the CTA
    cluster_sync_all();        // every partial of the cluster is in shared memory
    if (go) {
      // this CTA's rows of the tile
      const int l0 = (int)rank * rows / S, l1 = ((int)rank + 1) * rows / S;
      const int total = (l1 - l0) * (p.gate == kGateStacked ? 16 : 32);  // four features each
      if (p.gate == kGateParts) {
        if constexpr (!DIRECT) swap_parts_rows(p, smem_u32(P), mt, row0, l0, total);
      } else if (p.gate) {
        if (total <= SW_THREADS) swap_gate_rows<DIRECT, 1, 8>(p, smem_u32(P), mt, row0, l0, total, s_A);
        else swap_gate_rows<DIRECT, 4, 2>(p, smem_u32(P), mt, row0, l0, total, s_A);
      } else {
        if (total <= SW_THREADS) swap_correction_rows<DIRECT, 1, 8>(p, smem_u32(P), mt, row0, l0, total, s_A);
        else swap_correction_rows<DIRECT, 4, 2>(p, smem_u32(P), mt, row0, l0, total, s_A);
      }
    }
    fence_proxy_async_shared();  // the partial's space goes back to the copies of the next unit
    cluster_sync_all();          // no CTA moves on while the others read its shared memory
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

// W_g[:, :d] e alone: a round whose gate follows verification (the raw variant),
// and beside the correction above kGateBiasAlone.  Few registers, so that its CTAs
// fit on the SMs beside the correction's.
__global__ void __launch_bounds__(256) swap_gemv_kernel(const GateBiasParams p) {
  pdl_launch_dependents();
  gate_bias_share_small(p.e, p.Wg, p.ge, p.d, 2 * p.d, (int)blockIdx.x * 8 + (threadIdx.x >> 5), (int)gridDim.x * 8,
                        threadIdx.x & 31);
  // Complete only after the previous kernel: the next kernel's programmatic
  // wait, which covers this kernel alone, then covers that one too.  One CTA
  // waiting is enough (the grid completes with its last CTA); the others
  // leave and free their SM for the next kernel.
  if (blockIdx.x == 0) pdl_wait();
}

}  // namespace

cudaError_t launch_wait_selftest(int kind, const uint32_t* flag, uint32_t target, uint32_t* status,
                                 cudaStream_t stream) {
  wait_selftest_kernel<<<1, 32, 0, stream>>>(kind, flag, target, status);
  return cudaGetLastError();
}

bool tc_supported(retrace_dtype dtype, int d) {
  return dtype == RETRACE_BF16 && d >= 128 && d % 8 == 0;
}

bool direct_rows_supported(int B, int K, int d) {
  // K >= 5: the tile rows are at most twice the carried ones.  The corrected
  // signal's tile rows lie in the swp region.
  const long long rows = (long long)B * direct_tile_rows(K);
  return K >= 5 && rows <= kDirectMaxRows && B <= 32 && (long long)B * K <= 32 * kDirectChunks &&
         (size_t)(rows * d) * 2 <= swap_part_bytes(B, K, d);
}

cudaError_t launch_pack(const PackArgs& a, cudaStream_t stream) {
  if (a.B <= 0) return cudaSuccess;
  DeviceInfo info;
  cudaError_t err = device_info(&info);
  if (err != cudaSuccess) return err;
  PackParams p{};
  p.B = a.B;
  p.K = a.K;
  p.d = a.d;
  p.rows = a.rows;
  p.mode = a.mode;
  p.src0 = reinterpret_cast<const __nv_bfloat16*>(a.src0);
  p.src1 = reinterpret_cast<const __nv_bfloat16*>(a.src1);
  p.e = reinterpret_cast<const __nv_bfloat16*>(a.e);
  p.e_dense = a.e_dense;
  p.apack = reinterpret_cast<__nv_bfloat16*>(a.apack);
  p.epack = reinterpret_cast<__nv_bfloat16*>(a.epack);
  p.rowmap = a.rowmap;
  p.n_out = a.n_out;
  p.rest = reinterpret_cast<__nv_bfloat16*>(a.rest);
  p.sync = a.sync;
  p.sync_words = (int)(a.sync_bytes / 4);
  // the CTA-pair kernel computes W_g[:, :d] e itself
  if (a.mode == 1 && !a.e_dense && cond_small_r(a.B, a.K, a.d))
    p.bias = {a.d, p.e, reinterpret_cast<const __nv_bfloat16*>(a.Wg), a.ge};
  // a warp per position, four CTAs per SM at most; all of them for the GEMV
  const long long most = 4LL * info.sm_count, ctas = ((long long)a.B * a.K + 7) / 8;
  const unsigned grid = (unsigned)(p.bias.ge || ctas > most ? most : ctas);
  return launch_dependent(pack_rows_kernel, dim3(grid), dim3(256), 0, stream, 1u, p);
}

static cudaError_t launch_cond_pair(const TcCondArgs& a, int clusters, cudaStream_t stream) {
  const long long rmax = (long long)a.B * (a.K - 1);
  const uint64_t d = (uint64_t)a.d;
  CUtensorMap mApack, mWc, mR, mWv, mWg, mE, mWge;
  // Maps of operands a call does not use point at a used buffer (never read).
  const void* apack = a.do_correct ? a.apack : a.rpack;
  const void* wc = a.do_correct ? a.Wc : a.Wv;
  const void* rp = a.do_gate ? a.rpack : a.apack;
  const void* wv = a.do_gate ? a.Wv : a.Wc;
  const void* wg = a.do_gate ? a.Wg : a.Wc;
  const void* erows = a.do_gate && a.e_dense ? a.epack : rp;
  if (encode_tensor_map_2d(&mApack, apack, a.do_correct ? 2 * d : d, (uint64_t)rmax, (a.do_correct ? 4 : 2) * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWc, wc, a.do_correct ? 2 * d : d, d, (a.do_correct ? 4 : 2) * d, BK, 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mR, rp, d, (uint64_t)rmax, 2 * (a.r_row_stride ? (uint64_t)a.r_row_stride : d), BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWv, wv, a.do_gate ? d : 2 * d, d, (a.do_gate ? 2 : 4) * d, BK, 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWg, wg, 2 * d, d, 4 * d, BK, 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mE, erows, d, (uint64_t)rmax, 2 * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWge, wg, d, d, 4 * d, BK, 64) != CUDA_SUCCESS)  // the e half: zeros past column d
    return cudaErrorInvalidValue;
  CondParams p{};
  p.d = a.d;
  p.do_correct = a.do_correct;
  p.do_gate = a.do_gate;
  p.R = a.R;
  p.rowmap = a.rowmap;
  p.apack = reinterpret_cast<const __nv_bfloat16*>(a.apack);
  p.beta = a.beta;
  p.r_out = reinterpret_cast<__nv_bfloat16*>(a.r_out);
  p.compact_out = a.compact_out;
  p.e = reinterpret_cast<const __nv_bfloat16*>(a.e_dense ? a.epack : a.e);
  p.e_dense = a.e_dense;
  p.Wg = reinterpret_cast<const __nv_bfloat16*>(a.Wg);
  p.ge = a.ge;
  p.e_out = reinterpret_cast<__nv_bfloat16*>(a.e_out);
  p.sync = a.sync;
  p.block_done = a.sync + kSyncBlocks;
  p.block_ready = a.sync + kSyncBlocks + blocks_max(a.B, a.K);
  p.split_part = a.split_part;
  p.split_ticket = a.sync + kSyncBlocks + 2 * blocks_max(a.B, a.K);
  // (a K half over a per-position e would hold the gate's columns only)
  p.split_max = (a.split_part && a.do_gate && !a.e_dense) ? kPairSplitTiles : 0;
  p.status = a.status;
  // clusters of two CTAs; set-up may overlap the previous kernel's end
  auto kern = d % 256 == 0 && !p.e_dense ? cond_pair_kernel<false> : cond_pair_kernel<true>;
  return launch_dependent(kern, dim3(2 * (unsigned)clusters), dim3(P_THREADS), P_SMEM_BYTES, stream, 2, mApack, mWc, mR,
                          mWv, mWg, mE, mWge, p);
}

// Pairs of CTAs of cond_pair_kernel to launch: those the device keeps resident
// (cached per device; 0: none fits), or fewer when the call has fewer tiles.
static int pair_clusters(const TcCondArgs& a, long long tiles_max, cudaError_t* err) {
  static std::atomic<int> max_clusters[64];  // 0: not yet known, -1: none
  int dev = 0;
  if ((*err = cudaGetDevice(&dev)) != cudaSuccess) return 0;
  int n = max_clusters[dev & 63].load(std::memory_order_acquire);
  if (n == 0) {
    // (the two forms of the kernel have the same threads and shared memory, one CTA per SM)
    for (auto kern : {cond_pair_kernel<false>, cond_pair_kernel<true>})
      if ((*err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, P_SMEM_BYTES)) != cudaSuccess)
        return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(P_THREADS, 1, 1);
    cfg.dynamicSmemBytes = P_SMEM_BYTES;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((*err = cudaOccupancyMaxActiveClusters(&n, cond_pair_kernel<true>, &cfg)) != cudaSuccess) return 0;
    if (n < 1) n = -1;
    max_clusters[dev & 63].store(n, std::memory_order_release);
  }
  if (n < 0) return 0;
  // every pair when the gate-bias GEMV is needed: pairs without tiles compute it
  if (a.do_gate && !a.e_dense) return n;
  return (int)(tiles_max < n ? tiles_max : n);
}

// Clusters of S CTAs of swap_cluster_kernel that the device holds at once
// with `smem` bytes each (0: none), cached per device, S and shared memory.
static int swap_cluster_capacity(int dev, int S, int smem, cudaError_t* err) {
  static std::atomic<int> cache[64][9][17];  // [device][S][smem in 16 KB steps]; 0: not yet known, -1: none
  std::atomic<int>& slot = cache[dev & 63][S][smem >> 14];
  int n = slot.load(std::memory_order_acquire);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S, 1, 1);
    cfg.blockDim = dim3(SW_THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int m = 0;
    if ((*err = cudaOccupancyMaxActiveClusters(&m, swap_cluster_kernel<false>, &cfg)) != cudaSuccess) return 0;
    n = m > 0 ? m : -1;
    slot.store(n, std::memory_order_release);
  }
  return n > 0 ? n : 0;
}

// Cluster size of a small-R GEMM, `parts` products of S / parts K splits each:
// the one with the least estimated time.  R itself is known on the device only,
// so the estimate is the sum of two, at a half and at three quarters of the
// possible rows (direct rows: one tile of all the tile rows).  A wave of units
// costs its k-blocks (measured: 750 cycles each at N = 160, 830 at 177, 1070 at
// 250; the issue of the MMAs and the stage's handshake make most of a small
// one), 60 cycles per row of the tile (the drain and the sum over the splits),
// `wave` to start and end (4000), and with packed rows 700 per CTA of the cluster (they
// wait for each other).  Packed rows take four K splits at most: larger
// clusters are not all placed at once beside the last CTAs of the kernel before
// (a round, V = 2048, d = 3584, B = 32, 384 rows: 108 us with S = 5 for the
// correction, which one wave should hold, 72 with S = 2; direct rows, B = 8, K = 5,
// whose larger clusters are counted as seven eighths: 61 us with S = 5, 48 with
// S = 4).  Over 160 rounds of
// d = 1024 to 4096 and 64 to 733 rows, and 33 pairs of standalone calls, each
// timed with every S, the choice takes 1.5 % more than the best S of each (11 %
// at most); one estimate at three quarters, 2 (128 + N) cycles per k-block, 24
// per row, any S: 6 % (32 % at most).  Above d = 4096 a further wave costs far more,
// 20000: over 164 rounds of d = 4352 to 12288 the choice takes 1.9 % more than the
// best S of each (15 % at most), with 4000 5.5 % (78 %).  Below, 20000 changes 5 of 80
// choices, for 10 % more at one of two acceptance rates and 7 % less at the other.
static cudaError_t swap_pick_splits(int dev, int smem, int rmax, bool direct, int parts, int mtiles, int nkb, int wave,
                                    int* S_out, int* clusters) {
  long long best = -1;
  cudaError_t err = cudaSuccess;
  for (int splits = std::min(direct ? 8 : 4, 8 / parts); splits >= 1; --splits) {
    const int S = splits * parts;
    if (splits > 1 && nkb / splits < SW_MIN_BLOCKS) continue;
    const int cap = swap_cluster_capacity(dev, S, smem, &err);
    if (err != cudaSuccess) return err;
    if (cap == 0) continue;
    const int held = splits > 4 ? cap - cap / 8 : cap;  // at once, beside the kernel before
    long long cost = 0;
    for (const int rows : {(rmax + 1) / 2, (3 * rmax + 3) / 4}) {
      const SwapCut cut = direct ? SwapCut{1, (rmax + 15) / 16 * 16} : swap_cut(rows, mtiles, cap);
      const long long waves = ((long long)mtiles * cut.ntiles + held - 1) / held;
      const int block = std::max(750, 17 * cut.tile_n / 4);
      cost += waves * ((long long)((nkb + splits - 1) / splits) * block + 60 * cut.tile_n + wave + (direct ? 0 : 700 * S));
    }
    if (best < 0 || cost < best) {
      best = cost;
      *S_out = S;
      *clusters = cap;
    }
  }
  return best < 0 ? cudaErrorInvalidConfiguration : cudaSuccess;
}

// The rows operand of a small-R GEMM: `rows` rows of `inner` elements, one
// map per box height up to the largest tile of `rows` rows.
static bool encode_row_maps(RowMaps* maps, const void* base, uint64_t inner, int rows, uint64_t row_stride_bytes) {
  const int most = swap_box_rows(std::min(256, (rows + 15) / 16 * 16)) / SW_ROW_STEP;
  for (int i = 0; i < most; ++i)
    if (encode_tensor_map_2d(&maps->m[i], base, inner, (uint64_t)rows, row_stride_bytes, BK,
                             (uint32_t)(SW_ROW_STEP * (i + 1))) != CUDA_SUCCESS)
      return false;
  return true;
}

// The small-R path (cond_small_r): the correction GEMM with the gate-bias GEMV,
// then the gate GEMM; each launch waits on the one before inside the kernel,
// and cuts its work from the R it reads.  Past the operands' ends (d no multiple
// of the tiles) the copies fill zeros and the epilogues store nothing.
static cudaError_t launch_cond_swap(const TcCondArgs& a, cudaStream_t stream) {
  const bool direct = a.direct;
  // rows of the operands: tile rows (direct), or the most there can be
  const int rmax = direct ? a.B * direct_tile_rows(a.K) : (int)((long long)a.B * (a.K - 1));
  const int d = a.d;
  DeviceInfo info;
  cudaError_t err = device_info(&info);
  if (err != cudaSuccess) return err;
  const int dev = info.device;
  static std::atomic<int> attr_done[64];
  if (!attr_done[dev & 63].load(std::memory_order_acquire)) {
    // (the two forms have the same threads and, but for 128 bytes, shared memory)
    for (auto kern : {swap_cluster_kernel<false>, swap_cluster_kernel<true>}) {
      err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SW_SMEM_MAX);
      if (err != cudaSuccess) return err;
    }
    attr_done[dev & 63].store(1, std::memory_order_release);
  }
  const int box_max = swap_box_rows(std::min(256, (rmax + 15) / 16 * 16));
  // Stages with the largest row box, their weight tiles loaded before the wait.
  // (The kernel runs as many as fit with the box it needs.)  With a gate-bias
  // GEMV before that wait, four: it has the memory busy (rounds at d = 4096, B =
  // 8: 61.7 us with four, 64.1 with six).  Else all that fit (per-position e, V =
  // 2048, d = 4096, B = 8: 64.0 -> 58.5 us; d = 2560: 43.0 -> 40.9).
  int pre = swap_stages(SW_SMEM_RING - 1024, box_max);
  if (!(a.do_gate && a.e_dense)) pre = std::min(pre, 4);
  // at least half of an SM's shared memory: one CTA per SM, so the K splits
  // of one wave stream over distinct SMs
  const int smem = std::max(pre * (SW_A_BYTES + box_max * BK * 2) + 1024, 117 * 1024);
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < std::min(256, rmax)) tmem_cols <<= 1;
  const uint64_t du = (uint64_t)d;
  SwapClusterParams sp{};
  sp.R = a.R;
  sp.d = d;
  sp.stage_bytes = smem - 1024;
  sp.pre = pre;
  sp.row_maps = box_max / SW_ROW_STEP;
  sp.tmem_cols = tmem_cols;
  sp.rowmap = a.rowmap;
  sp.status = a.status;
  if (direct)
    sp.direct = {a.B, a.K, direct_tile_rows(a.K), a.keys, a.draft, a.accept_len, a.committed, a.bonus, a.n_out,
                 reinterpret_cast<const __nv_bfloat16*>(a.hD), reinterpret_cast<const __nv_bfloat16*>(a.e),
                 reinterpret_cast<__nv_bfloat16*>(a.e_out)};
  // whole row tiles side by side where the resident clusters can take every
  // row so, else all of them in turn over the units
  auto grid_of = [&](const SwapClusterParams& c, int clusters) {
    const int fit = clusters / c.mtiles, most = (rmax + SW_ROW_STEP - 1) / SW_ROW_STEP;
    if (direct) clusters = std::min(clusters, c.mtiles);
    else if (fit * 256 >= rmax) clusters = c.mtiles * std::min(fit, most);
    return dim3((unsigned)(clusters * c.S));
  };
  GateBiasParams gp{};
  gp.d = d;
  gp.e = reinterpret_cast<const __nv_bfloat16*>(a.e);
  gp.Wg = reinterpret_cast<const __nv_bfloat16*>(a.Wg);
  gp.ge = a.ge;
  const bool bias_alone = d > kGateBiasAlone;
  const int wave = d > 4096 && !a.e_dense ? 20000 : 4000;
  if (a.do_correct) {
    CUtensorMap mA, mA2;
    RowMaps mB;
    SwapClusterParams c = sp;
    c.mtiles = (d + 127) / 128;
    if (direct) {
      // the m and u halves apart: zeros past column d of either
      const uint64_t all = (uint64_t)a.B * a.K;
      const uint32_t box = (uint32_t)direct_tile_rows(a.K);
      if (encode_tensor_map_2d(&mA, a.Wc, du, du, 4 * du, BK, 128) != CUDA_SUCCESS ||
          encode_tensor_map_2d(&mA2, static_cast<const __nv_bfloat16*>(a.Wc) + d, du, du, 4 * du, BK, 128) != CUDA_SUCCESS ||
          encode_tensor_map_2d(&mB.m[0], a.hD, du, all, 2 * du, BK, box) != CUDA_SUCCESS ||
          encode_tensor_map_2d(&mB.m[1], a.hT, du, all, 2 * du, BK, box) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
      c.row_maps = 2;
      c.nkb_m = (d + BK - 1) / BK;
      c.nkb = 2 * c.nkb_m;
    } else {
      if (encode_tensor_map_2d(&mA, a.Wc, 2 * du, du, 4 * du, BK, 128) != CUDA_SUCCESS ||
          !encode_row_maps(&mB, a.apack, 2 * du, rmax, 4 * du))
        return cudaErrorInvalidValue;
      mA2 = mA;
      c.nkb = (2 * d + BK - 1) / BK;
    }
    c.apack = reinterpret_cast<const __nv_bfloat16*>(a.apack);
    c.beta = a.beta;
    c.r_out = reinterpret_cast<__nv_bfloat16*>(a.r_out);
    c.compact_out = a.compact_out;
    if (a.do_gate && !a.e_dense && !bias_alone) c.bias = gp;
    int clusters = 0;
    if ((err = swap_pick_splits(dev, smem, rmax, direct, 1, c.mtiles, c.nkb, wave, &c.S, &clusters)) != cudaSuccess) return err;
    err = launch_dependent(direct ? swap_cluster_kernel<true> : swap_cluster_kernel<false>, grid_of(c, clusters),
                           dim3(SW_THREADS), (size_t)smem, stream, (unsigned)c.S, mA, mA2, mA, mB, mB, c);
    if (err != cudaSuccess) return err;
  }
  if (a.do_gate) {
    const uint64_t rstride = 2 * (a.r_row_stride ? (uint64_t)a.r_row_stride : du);
    CUtensorMap mA, mA2, mA3;
    RowMaps mB, mE;
    const uint32_t box = a.e_dense ? 128 : 64;
    if (encode_tensor_map_2d(&mA, a.Wv, du, du, 2 * du, BK, box) != CUDA_SUCCESS ||
        encode_tensor_map_2d(&mA2, a.Wg, 2 * du, du, 4 * du, BK, box) != CUDA_SUCCESS ||
        encode_tensor_map_2d(&mA3, a.Wg, du, du, 4 * du, BK, box) != CUDA_SUCCESS ||  // the e half: zeros past column d
        !encode_row_maps(&mB, a.rpack, du, rmax, rstride) ||
        (a.e_dense && !encode_row_maps(&mE, a.epack, du, rmax, 2 * du)))
      return cudaErrorInvalidValue;
    if ((!a.do_correct || bias_alone) && !a.e_dense && !a.ge_ready) {  // W_g[:, :d] e in its own launch
      err = launch_dependent(swap_gemv_kernel, dim3((unsigned)(info.sm_count * 4)), dim3(256), 0, stream, 1u, gp);
      if (err != cudaSuccess) return err;
    }
    SwapClusterParams g = sp;
    g.mtiles = a.e_dense ? (d + 127) / 128 : (d + 63) / 64;
    g.nkb = (d + BK - 1) / BK;
    g.gate = a.e_dense ? kGateParts : kGateStacked;
    g.e = reinterpret_cast<const __nv_bfloat16*>(a.e_dense ? a.epack : a.e);
    g.ge = a.ge;
    g.e_out = reinterpret_cast<__nv_bfloat16*>(a.e_out);
    // all the shared memory where it buys stages and no verification follows
    // ahead: temperature-1 rounds, d = 4096, B = 32: 152.8 -> 150.2 us; per-position
    // e, V = 32000, B = 48: 205 -> 196
    const int gsmem = a.last && rmax > 256 ? SW_SMEM_MAX : smem;
    g.stage_bytes = gsmem - 1024;
    int clusters = 0;
    if ((err = swap_pick_splits(dev, gsmem, rmax, direct, a.e_dense ? 3 : 1, g.mtiles, g.nkb, wave, &g.S, &clusters)) != cudaSuccess)
      return err;
    err = launch_dependent(direct ? swap_cluster_kernel<true> : swap_cluster_kernel<false>, grid_of(g, clusters),
                           dim3(SW_THREADS), (size_t)gsmem, stream, (unsigned)g.S, mA, mA2, mA3, mB,
                           a.e_dense ? mE : mB, g);
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

// A per-position e with many rows (d a multiple of 256).
static cudaError_t launch_cond_one_sm(const TcCondArgs& a, cudaStream_t stream) {
  DeviceInfo info;
  cudaError_t err = device_info(&info);
  if (err != cudaSuccess) return err;
  static std::atomic<int> attr_done[64];
  if (!attr_done[info.device & 63].load(std::memory_order_acquire)) {
    err = cudaFuncSetAttribute(cond_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (err != cudaSuccess) return err;
    attr_done[info.device & 63].store(1, std::memory_order_release);
  }
  const long long rmax = (long long)a.B * (a.K - 1);
  const uint64_t d = (uint64_t)a.d;
  CUtensorMap mApack, mWc, mR, mE, mWv, mWg;
  // Maps of operands a call does not use point at a used buffer (never read).
  const void* apack = a.do_correct ? a.apack : a.rpack;
  const void* wc = a.do_correct ? a.Wc : a.Wv;
  if (encode_tensor_map_2d(&mApack, apack, a.do_correct ? 2 * d : d, (uint64_t)rmax, (a.do_correct ? 4 : 2) * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWc, wc, a.do_correct ? 2 * d : d, d, (a.do_correct ? 4 : 2) * d, BK, a.do_correct ? 256 : 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mR, a.rpack, d, (uint64_t)rmax, 2 * (a.r_row_stride ? (uint64_t)a.r_row_stride : d), BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mE, a.epack, d, (uint64_t)rmax, 2 * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWv, a.Wv, d, d, 2 * d, BK, 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWg, a.Wg, 2 * d, d, 4 * d, BK, 128) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  CondParams p{};
  p.d = a.d;
  p.do_correct = a.do_correct;
  p.do_gate = 1;
  p.R = a.R;
  p.rowmap = a.rowmap;
  p.apack = reinterpret_cast<const __nv_bfloat16*>(a.apack);
  p.beta = a.beta;
  p.r_out = reinterpret_cast<__nv_bfloat16*>(a.r_out);
  p.compact_out = a.compact_out;
  p.e = reinterpret_cast<const __nv_bfloat16*>(a.epack);
  p.e_dense = 1;
  p.e_out = reinterpret_cast<__nv_bfloat16*>(a.e_out);
  p.sync = a.sync;
  p.block_done = a.sync + kSyncBlocks;
  p.status = a.status;
  const long long tiles_max = (rmax + BM - 1) / BM * ((a.do_correct ? a.d / 256 : 0) + a.d / 128);
  const unsigned grid = (unsigned)std::min<long long>(tiles_max, info.sm_count);
  const VerifyStreamParams vp{};
  return launch_dependent(cond_kernel<false>, dim3(grid), dim3(THREADS), (size_t)SMEM_BYTES, stream, 1u, mApack, mWc,
                          mR, mE, mWv, mWg, p, vp);
}

cudaError_t launch_cond_tc(const TcCondArgs& a, cudaStream_t stream) {
  const long long rmax = (long long)a.B * (a.K - 1);
  if (rmax <= 0 || (!a.do_correct && !a.do_gate)) return cudaSuccess;
  auto path = [&](int pairs) {
    return cond_path(a.B, a.K, a.d, a.direct != 0, a.do_gate && a.e_dense, pairs);
  };
  if (path(1) == kCondSwap) return launch_cond_swap(a, stream);
  if (path(1) == kCondOneSm) return launch_cond_one_sm(a, stream);
  const long long tiles_max = (rmax + 2 * BM - 1) / (2 * BM) *
                              ((a.do_correct ? (a.d + 255) / 256 : 0) + (a.do_gate ? (a.d + 127) / 128 : 0));
  cudaError_t err;
  const int clusters = pair_clusters(a, tiles_max, &err);
  if (err != cudaSuccess) return err;
  if (path(clusters) == kCondPair) return launch_cond_pair(a, clusters, stream);
  TcCondArgs b = a;
  b.ge_ready = 0;  // launch_pack leaves it to the CTA-pair kernel above the small-R line
  return launch_cond_swap(b, stream);
}

}  // namespace retrace

namespace retrace {

bool round_fused_supported(const TcRoundArgs& a) {
  // contiguous logits with rows of at least one stream chunk, so that a chunk
  // is one contiguous copy and spans at most two rows
  return a.d >= 256 && a.d % 256 == 0 && 4 * a.d <= kStageBytes && ((uintptr_t)a.logits % 16 == 0) && a.V % 8 == 0 &&
         a.V >= 8 * kChunkSlots && a.row_stride == a.V && a.batch_stride == (long long)(a.K + 1) * a.V &&
         a.K >= 2 && (long long)a.B * (a.K + 1) * (a.V / 8) < (1ll << 32) - kChunkSlots;
}

cudaError_t launch_round_tc(const TcRoundArgs& a, cudaStream_t stream) {
  DeviceInfo info;
  cudaError_t err = device_info(&info);
  if (err != cudaSuccess) return err;
  static std::atomic<int> attr_done[64];
  if (!attr_done[info.device & 63].load(std::memory_order_acquire)) {
    err = cudaFuncSetAttribute(cond_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES_FUSED);
    if (err != cudaSuccess) return err;
    attr_done[info.device & 63].store(1, std::memory_order_release);
  }
  const uint64_t d = (uint64_t)a.d;
  const long long rmax = (long long)a.B * (a.K - 1);
  CUtensorMap mApack, mWc, mR, mE, mWv, mWg;
  if (encode_tensor_map_2d(&mApack, a.apack, 2 * d, (uint64_t)rmax, 4 * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWc, a.Wc, 2 * d, d, 4 * d, BK, 256) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mR, a.rpack, d, (uint64_t)rmax, 2 * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mE, a.e_dense ? a.epack : a.rpack, d, (uint64_t)rmax, 2 * d, BK, BM) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWv, a.Wv, d, d, 2 * d, BK, 128) != CUDA_SUCCESS ||
      encode_tensor_map_2d(&mWg, a.Wg, 2 * d, d, 4 * d, BK, 128) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const long long blocks = blocks_max(a.B, a.K);
  CondParams p{};
  p.d = a.d;
  p.do_correct = 1;
  p.do_gate = 1;
  p.R = reinterpret_cast<const int32_t*>(a.sync + kSyncRowCount);
  p.rowmap = a.rowmap;
  p.apack = reinterpret_cast<const __nv_bfloat16*>(a.apack);
  p.beta = a.beta;
  p.r_out = reinterpret_cast<__nv_bfloat16*>(a.rpack);
  p.compact_out = 1;
  p.e = reinterpret_cast<const __nv_bfloat16*>(a.e_dense ? a.epack : a.e);
  p.e_dense = a.e_dense;
  p.Wg = reinterpret_cast<const __nv_bfloat16*>(a.Wg);
  p.ge = a.ge;
  p.e_out = reinterpret_cast<__nv_bfloat16*>(a.e_out);
  p.sync = a.sync;
  p.block_done = a.sync + kSyncBlocks;
  p.block_ready = a.sync + kSyncBlocks + blocks;
  p.max_blocks = (int)blocks;
  p.status = a.status;

  VerifyStreamParams vp{};
  vp.logits = reinterpret_cast<const __nv_bfloat16*>(a.logits);
  vp.B = a.B;
  vp.K = a.K;
  vp.V = a.V;
  vp.draft = a.draft;
  vp.accept_len = a.accept_len;
  vp.committed = a.committed;
  vp.bonus = a.bonus;
  vp.target_argmax = a.target_argmax;
  vp.n_out = a.n_out;
  vp.keys = a.keys;
  vp.tickets = a.tickets;
  vp.e = reinterpret_cast<const __nv_bfloat16*>(a.e);
  vp.e_batch_stride = a.e_batch_stride;
  vp.e_pos_stride = a.e_pos_stride;
  vp.e_out = reinterpret_cast<__nv_bfloat16*>(a.e_out);
  vp.d = a.d;
  vp.hD = reinterpret_cast<const __nv_bfloat16*>(a.hD);
  vp.hT = reinterpret_cast<const __nv_bfloat16*>(a.hT);
  vp.e_dense = a.e_dense;
  vp.apack = reinterpret_cast<__nv_bfloat16*>(a.apack);
  vp.epack = reinterpret_cast<__nv_bfloat16*>(a.epack);
  vp.rowmap = a.rowmap;
  vp.R_count = a.sync + kSyncRowCount;
  vp.rows_ready = a.sync + kSyncBlocks + blocks;
  vp.seq_done = a.sync + kSyncSeqDone;
  vp.slots_per_row = a.V / 8;
  vp.total_slots = (long long)a.B * (a.K + 1) * vp.slots_per_row;
  vp.total_chunks = (uint32_t)((vp.total_slots + kChunkSlots - 1) / kChunkSlots);
  vp.chunk_next = a.sync + kSyncChunkNext;
  vp.status = a.status;

  const long long grid = info.sm_count;
  // Cooperative: every CTA's share of the logits feeds other CTAs' tiles, so
  // all CTAs must be resident together (one per SM); the launch fails
  // instead of starting if they cannot be.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(THREADS_FUSED);
  cfg.dynamicSmemBytes = SMEM_BYTES_FUSED;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, cond_kernel<true>, mApack, mWc, mR, mE, mWv, mWg, p, vp);
}

}  // namespace retrace
