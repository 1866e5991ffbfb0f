// TF32-family tensor-core kernels (sm_103a): the TF32 and 3xTF32 forms of the pairwise
// GEMM C[b] = A[b] (m x k) . B[b] (n x k)^T, complex (4M) and real, with or without
// exponent scaling:
//   contract_tc_kernel<REAL, SCALED>   TF32: A_re, A_im, B_re, B_im fp32 tiles, 32-deep
//                                      k-blocks, 3 stages, D_rr / D_ii / D_x accumulators
//                                      (Re C = D_rr - D_ii, Im C = D_x); 192 threads (real
//                                      tiles: 2 stages, 320 threads, two CTAs per SM);
//   contract_tc3t_kernel<REAL, SCALED, BT>  3xTF32: sixteen warps split each staged tile into
//                                      hi = RN_tf32(v) and lo = v - hi, A's into tensor memory;
//                                      hi.hi in 32-term chunks folded into round-to-nearest
//                                      registers, cross terms in their own accumulator; 576
//                                      threads, tiles of 64-192 (real) or 32-64 (complex) columns.
// Real TF32 steps take 128 x 256 output tiles (two B tiles read as one 256-row operand).
// Every mbarrier wait is bounded by wall time; on expiry the CTA records an error code,
// drains its copies, frees its tensor memory and returns.
#include <cstdint>

#include <cuda.h>
#include <cuda_runtime.h>

#include "kernels.h"
#include "mbarrier.cuh"
#include "scale.cuh"
#include "split_bf16.cuh"
#include "tc_common.cuh"
#include "pdl.cuh"

namespace tn {
namespace {

// TF32 form (contract_tc_kernel). A complex stage holds A_re A_im B_re B_im (3 stages, one
// CTA per SM; tensor memory D_rr @0, D_ii @128, D_x @256; warps 0 TMA, 1 MMA, 2-9 epilogue).
// A real one holds A B_0 B_1, the two B tiles of a 256-column tile, in 2 stages, and its
// accumulator takes 256 columns: two CTAs fit on an SM, so one's epilogue overlaps the
// other's MMAs. Eight epilogue warps store a tile's results: warp w drains TMEM lane quarter
// w % 4, the first or second half of the columns.
template <bool REAL>
struct Cfg {
  static constexpr int BK = 32;                             // fp32 elements per k-block
  static constexpr int ROWB = BK * 4;                       // bytes per tile row (= swizzle span)
  static constexpr int TILE_A = BM * ROWB;
  static constexpr int TILE_B = BN * ROWB;
  static constexpr int OFF_B = REAL ? TILE_A : 2 * TILE_A;  // first B tile
  static constexpr int STAGE = REAL ? TILE_A + 2 * TILE_B : 2 * TILE_A + 2 * TILE_B;
  static constexpr int STAGES = REAL ? 2 : 3;
  static constexpr int THREADS = 320;
  static constexpr uint32_t TMEM_COLS = REAL ? 256 : 512;
  static constexpr int OFFSETS = 8 * (BM + (REAL ? 2 : 1) * BN);  // output offsets of the rows and columns
  static constexpr int SMEM = STAGES * STAGE + 512 /*barriers*/ + OFFSETS + 1024 /*align*/;
  static_assert(SMEM <= 232448 && STAGE % 1024 == 0 && OFF_B % 1024 == 0, "stages fit, swizzle-aligned tiles");
  static_assert(8 * 2 * 32 * 33 * 4 <= STAGES * STAGE, "epilogue transposes fit the stages");
};

// v rounded to the nearest value with 10 fraction bits (ties away from zero): half a unit in
// the 10th fraction bit is added to the magnitude and the low 13 bits cleared (finite v
// below the largest TF32-representable value; an overflow would carry into the exponent).
__device__ __forceinline__ float tf32_rn(float v) {
  return __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
}

// REAL: a real step. Its tile is 128 x 256: the stage holds A and the B tiles of columns
// n0 .. n0 + 127 and n0 + 128 .. n0 + 255 side by side, one 128 x 256 MMA per k-atom reads
// the two as one operand, and the accumulator's 256 columns are the tile's output columns
// in order. SCALED: exponent scaling (a.recs).
// Measured (GB300; before: MMAs issued from a divergent lane, the block order sorted per block, four
// epilogue warps for a complex tile): complex 4096^3 822 -> 952 TFLOP/s, 8192 x 8192 x 512
// 439 -> 593, 1024 x 65536 x 256 304 -> 432; real 16384 x 32768 x 1024 539 -> 667, 8192 x 16384 x 256
// 229 -> 343 (bound by its stores, 2.7 TB/s). cuBLAS sustains 914-930.
template <bool REAL, bool SCALED>
__global__ void __launch_bounds__(Cfg<REAL>::THREADS, REAL ? 2 : 1)
    contract_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       StepArgs a, int64_t t_first, int* err) {
  using G = Cfg<REAL>;
  constexpr int STAGES = G::STAGES, BK = G::BK, ROWB = G::ROWB;
  constexpr int TILE_A = G::TILE_A, TILE_B = G::TILE_B, STAGE = G::STAGE, OFF_B = G::OFF_B;
  constexpr int TN = REAL ? 2 * BN : BN;            // output columns per tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE);
  uint64_t* full = bars;                     // [STAGES]
  uint64_t* empty = bars + STAGES;           // [STAGES]
  uint64_t* acc_full = bars + 2 * STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  int64_t* row_off = reinterpret_cast<int64_t*>(bars + 64);  // [BM] output offsets of the tile's rows
  int64_t* col_off = row_off + BM;                           // [TN] and columns

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  // grouped raster over output tiles for L2 reuse of A and B tiles
  const int64_t tiles_m = (a.m + BM - 1) / BM, tiles_n = (a.n + TN - 1) / TN;
  const int64_t t = t_first + blockIdx.x;  // this launch's tiles start at t_first
  const int64_t per_group = GROUP_M * tiles_n;
  const int64_t first_m = (t / per_group) * GROUP_M;
  const int64_t gm = tiles_m - first_m < GROUP_M ? tiles_m - first_m : GROUP_M;
  const int64_t tm = first_m + (t % per_group) % gm, tn = (t % per_group) / gm;
  const int m0 = static_cast<int>(tm * BM), n0 = static_cast<int>(tn * TN);
  const int b = blockIdx.y;
  const int num_kb = static_cast<int>((a.k + BK - 1) / BK);
  // plane of this batch entry's copy in the TMA maps: 2b + {re, im} complex, b real
  const int pa = a.a_bstride ? (REAL ? b : 2 * b) : 0, pb = a.b_bstride ? (REAL ? b : 2 * b) : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "r"(G::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = uniform_u32(*tmem_slot);
  pdl_wait();
  pdl_next();

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < num_kb; ++kb) {
        const int s = kb % STAGES;
        const uint32_t ph = (kb / STAGES) & 1;
        if (!mbar_wait(&empty[s], ph ^ 1)) {
          atomicExch(err, 1);
          break;
        }
        mbar_expect_tx(&full[s], STAGE);
        uint8_t* st = smem + s * STAGE;
        const int k0 = kb * BK;
        tma_load_3d(st, &tmA, &full[s], k0, m0, pa);
        if constexpr (REAL) {
          // the second B tile may lie wholly past n: the box is then zero-filled
          tma_load_3d(st + OFF_B, &tmB, &full[s], k0, n0, pb);
          tma_load_3d(st + OFF_B + TILE_B, &tmB, &full[s], k0, n0 + BN, pb);
        } else {
          tma_load_3d(st + TILE_A, &tmA, &full[s], k0, m0, pa + 1);
          tma_load_3d(st + 2 * TILE_A, &tmB, &full[s], k0, n0, pb);
          tma_load_3d(st + 2 * TILE_A + TILE_B, &tmB, &full[s], k0, n0, pb + 1);
        }
        issued = kb + 1;
      }
      // drain: every stage's last issued load has landed before the CTA can exit
      for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
        if (!mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1)) atomicExch(err, 2);
    }
  } else if (warp == 1) {
    const bool leader = elect_one();
    constexpr uint32_t idesc = idesc_tf32(BM, TN);
    const uint32_t d_rr = tmem, d_ii = tmem + 128, d_x = tmem + 256;
    const uint64_t desc0 = smem_desc<ROWB>(su32(smem));
    for (int kb = 0; kb < num_kb; ++kb) {
      const int s = kb % STAGES;
      const uint32_t ph = (kb / STAGES) & 1;
      if (!mbar_wait_warp(&full[s], ph)) {
        if (leader) atomicExch(err, 3);
        break;
      }
      fence_after();
      const uint64_t st = desc0 + static_cast<uint32_t>(s * (STAGE >> 4));
      if (leader) {
#pragma unroll
        for (int j = 0; j < BK / 8; ++j) {
          const uint32_t acc = (kb > 0 || j > 0) ? 1u : 0u;
          const uint64_t ar = st + 2 * j, ai = st + (TILE_A >> 4) + 2 * j;
          const uint64_t br = st + (OFF_B >> 4) + 2 * j, bi = st + ((OFF_B + TILE_B) >> 4) + 2 * j;
          if constexpr (REAL) {
            mma_tf32(tmem, ar, br, idesc, acc);  // br: the 256 B rows of both tiles
          } else {
            mma_tf32(d_rr, ar, br, idesc, acc);
            mma_tf32(d_ii, ai, bi, idesc, acc);
            mma_tf32(d_x, ar, bi, idesc, acc);
            mma_tf32(d_x, ai, br, idesc, 1u);
          }
        }
        mma_commit(&empty[s]);
      }
      __syncwarp();
    }
    if (leader) mma_commit(acc_full);  // also on error: lets the epilogue see in-flight MMAs retire
    __syncwarp();
  } else {
    // epilogue: TMEM lane quarter of this warp = warp % 4
    // output offsets, while the first loads and MMAs run
    for (int x = threadIdx.x - 64; x < BM + TN; x += 256) {
      if (x < BM) row_off[x] = m0 + x < a.m ? map_offset(a.rows, m0 + x) : 0;
      else col_off[x - BM] = n0 + x - BM < a.n ? map_offset(a.cols, n0 + x - BM) : 0;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const bool ok = mbar_wait_warp(acc_full, 0);
    if (!ok && lane == 0) atomicExch(err, 6);
    fence_after();
    const int q = warp & 3, half = (warp - 2) >> 2;
    const bool row_ok = ok && m0 + q * 32 + lane < a.m;
    const int64_t rows_left = ok ? a.m - m0 - 32 * q : 0;
    float* C = a.C + static_cast<int64_t>(b) * a.c_bstride;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    // Each 32 x 32 block goes through shared memory (the drained stage buffers) and is
    // stored in address order: 32 consecutive elements per warp store for the usual layouts.
    float* tr = reinterpret_cast<float*>(smem) + (warp - 2) * 2 * 32 * 33;  // [2][32][33]
    const TcScale sc = tc_scale(a, b);
    int lmax = -127;
    constexpr int NCB = TN / 64;  // this warp's 32-column blocks
#pragma unroll 1
    for (int c = half * NCB; c < (half + 1) * NCB; ++c) {
      const int64_t cols_left = a.n - n0 - 32 * c;
      if constexpr (REAL) {
        float v[32];
        tmem_ld32(tmem + lane_base + c * 32, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          if constexpr (SCALED) {
            v[j] = v[j] * sc.sa * sc.sb;
            if (row_ok && j < cols_left) lmax = max(lmax, exp_of(fabsf(v[j])));
          }
          tr[lane * 33 + j] = v[j];
        }
      } else {
        float rr[32], ii[32], xx[32];
        tmem_ld32(tmem + lane_base + c * 32, rr);
        tmem_ld32(tmem + lane_base + 128 + c * 32, ii);
        tmem_ld32(tmem + lane_base + 256 + c * 32, xx);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          float re = rr[j] - ii[j], im = xx[j];
          if constexpr (SCALED) {
            re = re * sc.sa * sc.sb;
            im = im * sc.sa * sc.sb;
            if (row_ok && j < cols_left) lmax = max(lmax, exp_of(fmaxf(fabsf(re), fabsf(im))));
          }
          tr[lane * 33 + j] = re;
          tr[32 * 33 + lane * 33 + j] = im;
        }
      }
      __syncwarp();
      store_block_planned<REAL>(C, a.c_plane, kFmtPlanar, tr, 33, 32 * 33, row_off + 32 * q, col_off + 32 * c,
                                static_cast<int>(rows_left < 32 ? rows_left : 32),
                                static_cast<int>(cols_left < 32 ? cols_left : 32), a.blk, lane, 0, 1);
      __syncwarp();
    }
    if constexpr (SCALED) tc_scale_finish(a, b, lmax, t == 0 && threadIdx.x == 64);
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G::TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------------
// 3xTF32 with round-to-nearest accumulation across k.
//
// The tensor core's FP32 accumulator truncates each addition, so a long TMEM accumulation
// drifts toward zero by ~k * 2^-25 relative (measured). Here the hi.hi MMAs of 32 terms go into a
// chunk accumulator, which warps add into running totals in their registers with ordinary
// round-to-nearest FP32 additions (longer chunks lose more: 64 terms were 5 % faster but left the
// FP32-accurate form at twice plain FP32's error on long paths); the cross terms (2^-11 of the
// result) keep one accumulator over all of k. A complex tile's B planes are [-B_im | B_re | B_im],
// so A_re.[B_re | B_im] and A_im.[-B_im | B_re] add into (Re | Im) with one MMA each.
//
// What bounds it: shared-memory bandwidth. Per k-block TMA writes the raw tiles, the split reads
// them and writes hi and lo, and every MMA reads its operands (A and B three times). The split
// therefore writes A's hi and lo into tensor memory (tcgen05.st, thread = row), where the MMAs
// read them: no A stores to shared memory, no A reads from it. Per 32 terms of a real 128 x 192
// tile that is 200 KB of shared-memory traffic for 1152 clocks of MMAs (a 128 x 256 tile with A in
// shared memory: 336 KB for 1536). Tensor memory sets the tile: chunk and cross accumulators of N
// columns and two buffers of A (hi and lo, 32 columns each, re and im) in 512 columns.
//
// Measured (GB300; before: 128 x 256 real, 128 x 128 complex tiles, A in shared memory, MMAs
// issued from a divergent lane): real 16384 x 32768 x 1024 7.87 -> 5.21 ms (140 -> 211 TFLOP/s),
// 2048 x 16384 x 8192 166 -> 234; complex 4096^3 231 -> 305, few tiles: 512 x 128 x 2048 178 -> 53 us,
// 256 x 256 x 256 36 -> 14 us. cuBLAS's sustained TF32 rate over three products is 305.
// BT rows of B per plane; the narrow tiles (64 real, 32 complex) put a small step's outputs on
// more SMs.
// Warps: 0 TMA, 1 MMA + TMEM, 2-17 split / fold / epilogue. Sixteen of them, because a block's
// split and fold are a chain of latencies (shared memory, tensor memory, fences, barriers) that
// eight warps could not finish within the block's MMAs (1920 against 1330 clocks): warp w owns
// TMEM lanes 32 (w % 4) .. + 31, and of a row the part (w - 2) / 4 splits a quarter of A's terms
// (real) or half of a plane's (complex) and folds every fourth 16-column unit.
template <bool REAL, int BT>
struct C3T {
  static constexpr int BK = 32, ROWB = 128;
  static constexpr int NP = REAL ? 1 : 2;
  static constexpr int N = NP * BT;                         // MMA columns
  static constexpr int TILE_A = BM * ROWB, TILE_B = BT * ROWB;
  static constexpr int OFF_B = NP * TILE_A;                 // the B area: [B], or [-B_im | B_re | B_im]
  static constexpr int AREA_B = (REAL ? 1 : 3) * TILE_B;
  static constexpr int STAGE = OFF_B + AREA_B;
  static constexpr int LOADED = NP * (TILE_A + TILE_B);     // TMA bytes per stage
  static constexpr int LO = 2, FIT = (232448 - 1536 - 8 * (BM + BT) - LO * AREA_B) / STAGE;
  static constexpr int STAGES = FIT < 5 ? FIT : 5;
  static constexpr int THREADS = 576, WORKERS = 512;
  static constexpr int OFFSETS = 8 * (BM + BT);             // output offsets of the rows and columns
  static constexpr int SMEM = STAGES * STAGE + LO * AREA_B + 512 + OFFSETS + 1024;  // + barriers, alignment
  static constexpr int ACOLS = NP * 2 * BK;                 // one buffer of A: plane p hi @32 p, lo @32 (NP + p)
  static constexpr uint32_t COLS = 512;
  // chunk accumulators: two where they fit, so that a chunk's hi.hi need not wait for the fold of
  // the one before
  static constexpr int HI = 3 * N + 2 * ACOLS <= 512 ? 2 : 1;
  static constexpr int D_LO = HI * N, A_COL = D_LO + N;     // columns of the cross-term accumulator and of A
  static constexpr int UNITS = BT / 16;                     // 16-column units of a plane
  static constexpr int MINE = (UNITS + 3) / 4;              // units a warp folds at most
  static constexpr int FOLDERS = UNITS >= 4 ? 16 : 4 * UNITS;
  static constexpr int NB = BT / 32;                        // 32-column blocks of the tile
  static_assert(A_COL + 2 * ACOLS <= 512 && N % 16 == 0 && TILE_B % 1024 == 0, "tensor memory and swizzle");
  static_assert(SMEM <= 232448 && 4 * NB * NP * 32 * 33 * 4 <= STAGES * STAGE, "stages; epilogue transposes");
};

template <bool REAL, bool SCALED, int BT>
__global__ void __launch_bounds__(576, 1)
    contract_tc3t_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                         StepArgs a, int64_t t_first, int* err) {
  using G = C3T<REAL, BT>;
  constexpr int STAGES = G::STAGES, BK = G::BK, ROWB = G::ROWB, NP = G::NP;
  constexpr int TILE_A = G::TILE_A, TILE_B = G::TILE_B, STAGE = G::STAGE;
  // B planes in the B area (hi in the stage, lo in the lo buffer)
  constexpr int B_RE = REAL ? 0 : TILE_B, B_IM = 2 * TILE_B;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* lo_base = smem + STAGES * STAGE;
  uint64_t* bars = reinterpret_cast<uint64_t*>(lo_base + G::LO * G::AREA_B);
  uint64_t* full = bars;                     // [STAGES]
  uint64_t* empty = bars + STAGES;           // [STAGES]
  uint64_t* conv_full = bars + 2 * STAGES;   // [2] block split
  uint64_t* lo_empty = conv_full + 2;        // [2] lo buffer and A buffer read
  uint64_t* acc_full = lo_empty + 2;         // [HI] chunk accumulated
  uint64_t* acc_empty = acc_full + G::HI;    // [HI] chunk folded
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + G::HI);
  int64_t* row_off = reinterpret_cast<int64_t*>(bars + 64);  // [BM] output offsets of the tile's rows
  int64_t* col_off = row_off + BM;                           // [BT] and columns

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int64_t tiles_m = (a.m + BM - 1) / BM, tiles_n = (a.n + BT - 1) / BT;
  const int64_t t = t_first + blockIdx.x;  // this launch's tiles start at t_first
  const int64_t per_group = GROUP_M * tiles_n;
  const int64_t first_m = (t / per_group) * GROUP_M;
  const int64_t gm = tiles_m - first_m < GROUP_M ? tiles_m - first_m : GROUP_M;
  const int64_t tm = first_m + (t % per_group) % gm, tn = (t % per_group) / gm;
  const int m0 = static_cast<int>(tm * BM), n0 = static_cast<int>(tn * BT);
  const int b = blockIdx.y;
  const int num_kb = static_cast<int>((a.k + BK - 1) / BK);
  const int pa = a.a_bstride ? NP * b : 0, pb = a.b_bstride ? NP * b : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&conv_full[i], G::WORKERS);
      mbar_init(&lo_empty[i], 1);
    }
    for (int i = 0; i < G::HI; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], G::FOLDERS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "r"(G::COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = uniform_u32(*tmem_slot);
  pdl_wait();
  pdl_next();

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int kb = 0; kb < num_kb; ++kb) {
        const int s = kb % STAGES;
        if (!mbar_wait(&empty[s], ((kb / STAGES) & 1) ^ 1)) {
          atomicExch(err, 71);
          break;
        }
        mbar_expect_tx(&full[s], G::LOADED);
        uint8_t* st = smem + s * STAGE;
        const int k0 = kb * BK;
        tma_load_3d(st, &tmA, &full[s], k0, m0, pa);
        tma_load_3d(st + G::OFF_B + B_RE, &tmB, &full[s], k0, n0, pb);
        if constexpr (!REAL) {
          tma_load_3d(st + TILE_A, &tmA, &full[s], k0, m0, pa + 1);
          tma_load_3d(st + G::OFF_B + B_IM, &tmB, &full[s], k0, n0, pb + 1);
        }
        issued = kb + 1;
      }
      for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
        if (!mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1)) atomicExch(err, 72);
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = idesc_tf32(BM, G::N);  // complex: (Re | Im) at once
    const bool leader = elect_one();
    const uint32_t d_lo = tmem + G::D_LO;
    // descriptors of the first stage's and lo buffer's B areas; 16-byte units are added to them
    const uint64_t hi0 = smem_desc<ROWB>(su32(smem + G::OFF_B)), lo0 = smem_desc<ROWB>(su32(lo_base));
    bool mma_ok = true;
    int s = 0;
    for (int kb = 0; kb < num_kb; ++kb, s = s + 1 == STAGES ? 0 : s + 1) {
      if (!mbar_wait_warp(&conv_full[kb & 1], (kb >> 1) & 1)) {
        if (leader) atomicExch(err, 74);
        mma_ok = false;
        break;
      }
      fence_after();
      const uint64_t hi = hi0 + static_cast<uint32_t>(s * (STAGE >> 4));
      const uint64_t lo = lo0 + static_cast<uint32_t>((kb & 1) * (G::AREA_B >> 4));
      const uint32_t at = tmem + G::A_COL + (kb & 1) * G::ACOLS;
      const uint32_t ar = at, ai = at + BK, arl = at + NP * BK, ail = arl + BK;
      // the cross terms first (their accumulator runs over all of k), so that they overlap the
      // fold of the previous chunk; then, once that is folded, the chunk's hi.hi
      if (leader) {
#pragma unroll
        for (int j = 0; j < BK / 8; ++j) {
          const uint64_t b_ri = hi + (B_RE >> 4) + 2 * j, bl_ri = lo + (B_RE >> 4) + 2 * j;
          const uint64_t b_nr = hi + 2 * j, bl_nr = lo + 2 * j;
          mma_tf32_ts(d_lo, arl + 8 * j, b_ri, idesc, (kb > 0 || j > 0) ? 1u : 0u);
          if constexpr (!REAL) mma_tf32_ts(d_lo, ail + 8 * j, b_nr, idesc, 1u);
          mma_tf32_ts(d_lo, ar + 8 * j, bl_ri, idesc, 1u);
          if constexpr (!REAL) mma_tf32_ts(d_lo, ai + 8 * j, bl_nr, idesc, 1u);
        }
      }
      const int h = kb % G::HI;
      const uint32_t d_hi = tmem + h * G::N;
      if (!mbar_wait_warp(&acc_empty[h], ((kb / G::HI) & 1) ^ 1)) {
        if (leader) atomicExch(err, 73);
        mma_ok = false;
        break;
      }
      fence_after();
      if (leader) {
#pragma unroll
        for (int j = 0; j < BK / 8; ++j) {
          mma_tf32_ts(d_hi, ar + 8 * j, hi + (B_RE >> 4) + 2 * j, idesc, j > 0 ? 1u : 0u);
          if constexpr (!REAL) mma_tf32_ts(d_hi, ai + 8 * j, hi + 2 * j, idesc, 1u);
        }
        mma_commit(&empty[s]);
        mma_commit(&lo_empty[kb & 1]);
        mma_commit(&acc_full[h]);
      }
      __syncwarp();
    }
    if (!mma_ok && leader) mma_commit(&acc_full[0]);  // tracks the issued MMAs
    __syncwarp();
  } else {
    const int et = threadIdx.x - 64;  // 0..511
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int row = q * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    const bool folds = part < G::UNITS;  // (warp-uniform)
    float run[NP][G::MINE][16];
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int i = 0; i < G::MINE; ++i)
#pragma unroll
        for (int j = 0; j < 16; ++j) run[p][i][j] = 0.f;
    bool ok = true;
    // output offsets, while the first loads are on their way
    if (et < BM) row_off[et] = m0 + et < a.m ? map_offset(a.rows, m0 + et) : 0;
    else if (et < BM + BT) col_off[et - BM] = n0 + et - BM < a.n ? map_offset(a.cols, n0 + et - BM) : 0;
    for (int kb = 0; kb <= num_kb; ++kb) {
      if (kb < num_kb) {
        const int s = kb % STAGES;
        if (!mbar_wait_warp(&full[s], (kb / STAGES) & 1) || !mbar_wait_warp(&lo_empty[kb & 1], ((kb >> 1) & 1) ^ 1)) {
          if (lane == 0) atomicExch(err, 75);
          ok = false;
          break;
        }
        fence_after();
        // every shared-memory read of the block first: B's pieces, then A's
        constexpr int PB = NP * TILE_B / 16 / G::WORKERS;
        static_assert(PB * G::WORKERS * 16 == NP * TILE_B, "whole pieces per thread");
        float4* src = reinterpret_cast<float4*>(smem + s * STAGE + G::OFF_B);
        float4* dst = reinterpret_cast<float4*>(lo_base + (kb & 1) * G::AREA_B);
        float4 bv[PB];
#pragma unroll
        for (int i = 0; i < PB; ++i) bv[i] = src[et + G::WORKERS * i + B_RE / 16];
        // A: W terms of this thread's row (of plane part / 2 in a complex step), from the
        // 128-byte swizzled tile (16-byte piece c at c ^ (row % 8)): hi rounded to the nearest
        // TF32, lo the exact rest, into the buffer's columns
        constexpr int W = REAL ? 8 : 16;
        const int k_first = REAL ? 8 * part : 16 * (part & 1), plane = REAL ? 0 : part >> 1;
        const uint8_t* arow = smem + s * STAGE + plane * TILE_A + row * ROWB;
        const uint32_t at = tmem + lane_base + G::A_COL + (kb & 1) * G::ACOLS + plane * BK + k_first;
        float h[W], l[W];
#pragma unroll
        for (int c = 0; c < W / 4; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(arow + (((k_first / 4 + c) ^ (row & 7)) << 4));
          const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            h[4 * c + e] = tf32_rn(x[e]);
            l[4 * c + e] = x[e] - h[4 * c + e];
          }
        }
        tmem_st(at, h);
        tmem_st(at + NP * BK, l);
        // B: hi in place, lo into the lo buffer; of B_im also their negatives
#pragma unroll
        for (int i = 0; i < PB; ++i) {
          const int f = et + G::WORKERS * i + B_RE / 16;
          const float4 v = bv[i];
          float4 x, y;
          x.x = tf32_rn(v.x);
          x.y = tf32_rn(v.y);
          x.z = tf32_rn(v.z);
          x.w = tf32_rn(v.w);
          y.x = v.x - x.x;
          y.y = v.y - x.y;
          y.z = v.z - x.z;
          y.w = v.w - x.w;
          src[f] = x;
          dst[f] = y;
          if (!REAL && f >= B_IM / 16) {
            const int g = f - B_IM / 16;
            src[g] = make_float4(-x.x, -x.y, -x.z, -x.w);
            dst[g] = make_float4(-y.x, -y.y, -y.z, -y.w);
          }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        fence_before();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&conv_full[kb & 1]);
      }
      // fold chunk kb - 1 (its MMAs ran while this block was split) into the register totals with
      // round-to-nearest additions and release the accumulator
      if (kb > 0 && folds) {
        const int d = (kb - 1) % G::HI;
        if (!mbar_wait_warp(&acc_full[d], ((kb - 1) / G::HI) & 1)) {
          if (lane == 0) atomicExch(err, 76);
          ok = false;
          break;
        }
        fence_after();
        auto add = [&](uint32_t first) {  // the accumulator at column `first`
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            float v[G::MINE][16];
#pragma unroll
            for (int i = 0; i < G::MINE; ++i)
              tmem_ld16_async(tmem + lane_base + first + p * BT + 16 * (part + 4 * i), v[i]);
            tmem_ld_wait(v);
#pragma unroll
            for (int i = 0; i < G::MINE; ++i)
#pragma unroll
              for (int j = 0; j < 16; ++j) run[p][i][j] += v[i][j];
          }
        };
        add(d * G::N);
        if (kb == num_kb) add(G::D_LO);  // last chunk: the cross terms too
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[d]);
      }
    }
    // Epilogue: the four warps of a lane quarter put their columns into 32 x 32 blocks in shared
    // memory and store them in address order. The stage buffers are free: the last fold waited
    // for the final MMA, which waited for every warp's last split; no TMA load is outstanding.
    // (A warp that gave up a wait stores nothing; its barrier below still completes.)
    float* C = a.C + static_cast<int64_t>(b) * a.c_bstride;
    constexpr int BLK = NP * 32 * 33;
    float* tr = reinterpret_cast<float*>(smem) + q * G::NB * BLK;
    if (folds) {
      const TcScale sc = tc_scale(a, b);
      int lmax = -127;
#pragma unroll
      for (int i = 0; i < G::MINE; ++i) {
        const int u = part + 4 * i;
        float* t = tr + (u >> 1) * BLK + lane * 33 + 16 * (u & 1);
        // (rows past m and columns past n hold zeros: their operands were zero-filled by TMA)
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float re = run[0][i][j], im = REAL ? 0.f : run[NP - 1][i][j];
          if constexpr (SCALED) {
            re = re * sc.sa * sc.sb;
            im = im * sc.sa * sc.sb;
            lmax = max(lmax, exp_of(REAL ? fabsf(re) : fmaxf(fabsf(re), fabsf(im))));
          }
          t[j] = re;
          if constexpr (!REAL) t[32 * 33 + j] = im;
        }
      }
      if constexpr (SCALED) tc_scale_finish(a, b, lmax, t == 0 && threadIdx.x == 64);
    }
    // (the row offsets come from warps of other quarters: a barrier of all workers)
    asm volatile("bar.sync 1, 512;" ::: "memory");
    // blocks dealt out four at a time; a last round of fewer is shared by the warps
    static_assert(G::NB % 4 != 3, "parts of the last round");
    const int64_t rows_left = ok ? a.m - m0 - 32 * q : 0, cols_left = a.n - n0;
#pragma unroll 1
    for (int c0 = 0; c0 < G::NB; c0 += 4) {
      const int left = G::NB - c0 < 4 ? G::NB - c0 : 4, parts = 4 / left;
      const int c = c0 + part / parts;
      store_block_planned<REAL>(C, a.c_plane, kFmtPlanar, tr + c * BLK, 33, 32 * 33, row_off + 32 * q, col_off + 32 * c,
                                static_cast<int>(rows_left < 32 ? rows_left : 32),
                                static_cast<int>(cols_left - 32 * c < 32 ? cols_left - 32 * c : 32), a.blk, lane,
                                part % parts, parts);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G::COLS));
  }
}

// Planes of an operand's TMA map: 2 per stored copy (re, im) for a complex step, 1 for a
// real one (plane p of a real batched operand starts at p * its batch stride, which equals
// its plane size); one copy unless the operand is batched.
int64_t map_planes(bool batched, int32_t nb, bool real) {
  return (batched ? static_cast<int64_t>(nb) : 1) * (real ? 1 : 2);
}
// Tiles of a TF32 step: 128 x 256 real, 128 x 128 complex.
int64_t tf32_tiles(int64_t m, int64_t n, bool real) {
  const int64_t tn = real ? 2 * BN : BN;
  return ((m + BM - 1) / BM) * ((n + tn - 1) / tn);
}
int64_t tc3t_tiles(int64_t m, int64_t n, int bt) { return ((m + BM - 1) / BM) * ((n + bt - 1) / bt); }

// Columns of a 3xTF32 step's tile: the least waves x (k-blocks x time of one + time of a tile's
// prologue and epilogue), in microseconds as measured with full waves (the bits do not depend on
// it). Wide tiles have the cheaper k-blocks per output, narrow ones fill the SMs when there are
// few outputs: real 1024 x 4096 x 256 33 / 25 / 35 us with 192 / 128 / 64 columns.
int tc3t_bt(int64_t m, int64_t n, int64_t k, int32_t nb, bool real) {
  struct Form {
    int bt;
    double block, tile;
  };
  static const Form kReal[] = {{192, 0.92, 6.7}, {128, 0.66, 4.9}, {64, 0.48, 3.8}};
  static const Form kCplx[] = {{64, 1.0, 5.8}, {32, 0.70, 4.4}};
  const int64_t sms = device_sms() > 0 ? device_sms() : 148;
  const double kb = double((k + 31) / 32);
  int best = 0;
  double best_t = 0.0;
  for (int i = 0; i < (real ? 3 : 2); ++i) {
    const Form& f = real ? kReal[i] : kCplx[i];
    const double waves = double((tc3t_tiles(m, n, f.bt) * nb + sms - 1) / sms), t = waves * (kb * f.block + f.tile);
    if (best == 0 || t < best_t) {
      best = f.bt;
      best_t = t;
    }
  }
  return best;
}

template <bool REAL, bool SCALED>
cudaError_t launch_tf32(const StepArgs& a, int32_t nb, int* err, cudaStream_t st) {
  using G = Cfg<REAL>;
  static const cudaError_t configured = cudaFuncSetAttribute(
      contract_tc_kernel<REAL, SCALED>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (configured != cudaSuccess) return configured;
  CUtensorMap ta, tb;
  if (!make_map(&ta, a.A, a.m, a.k, map_planes(a.a_bstride != 0, nb, REAL), a.a_plane, BM, G::BK) ||
      !make_map(&tb, a.B, a.n, a.k, map_planes(a.b_bstride != 0, nb, REAL), a.b_plane, BN, G::BK))
    return cudaErrorInvalidValue;
  return launch_bands(contract_tc_kernel<REAL, SCALED>, tf32_tiles(a.m, a.n, REAL), nb, G::THREADS, G::SMEM, st, ta,
                      tb, a, err);
}

template <bool REAL, bool SCALED, int BT>
cudaError_t launch_tc3t(const StepArgs& a, int32_t nb, int* err, cudaStream_t st) {
  using G = C3T<REAL, BT>;
  static const cudaError_t configured = cudaFuncSetAttribute(
      contract_tc3t_kernel<REAL, SCALED, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
  if (configured != cudaSuccess) return configured;
  CUtensorMap ta, tb;
  if (!make_map(&ta, a.A, a.m, a.k, map_planes(a.a_bstride != 0, nb, REAL), a.a_plane, BM, G::BK) ||
      !make_map(&tb, a.B, a.n, a.k, map_planes(a.b_bstride != 0, nb, REAL), a.b_plane, BT, G::BK))
    return cudaErrorInvalidValue;
  return launch_bands(contract_tc3t_kernel<REAL, SCALED, BT>, tc3t_tiles(a.m, a.n, BT), nb, G::THREADS, G::SMEM, st,
                      ta, tb, a, err);
}

template <bool SCALED>
cudaError_t launch_3xtf32(const StepArgs& a, int32_t nb, bool cplx, int* err, cudaStream_t st) {
  const int bt = tc3t_bt(a.m, a.n, a.k, nb, !cplx);
  if (cplx)
    return bt == 32 ? launch_tc3t<false, SCALED, 32>(a, nb, err, st) : launch_tc3t<false, SCALED, 64>(a, nb, err, st);
  if (bt == 64) return launch_tc3t<true, SCALED, 64>(a, nb, err, st);
  if (bt == 128) return launch_tc3t<true, SCALED, 128>(a, nb, err, st);
  return launch_tc3t<true, SCALED, 192>(a, nb, err, st);
}

}  // namespace

cudaError_t launch_contract_tf32(const StepArgs& a, int32_t nb, int32_t prec, bool cplx, int* err,
                                 cudaStream_t st) {
  const bool sc = a.recs != nullptr;
  if (!cplx) {
    if (prec == TN_R32_TF32) return sc ? launch_tf32<true, true>(a, nb, err, st) : launch_tf32<true, false>(a, nb, err, st);
    if (prec == TN_R32_3XTF32) return sc ? launch_3xtf32<true>(a, nb, false, err, st) : launch_3xtf32<false>(a, nb, false, err, st);
    return cudaErrorNotSupported;
  }
  if (prec == TN_C64_TF32) return sc ? launch_tf32<false, true>(a, nb, err, st) : launch_tf32<false, false>(a, nb, err, st);
  if (prec == TN_C64_3XTF32) return sc ? launch_3xtf32<true>(a, nb, true, err, st) : launch_3xtf32<false>(a, nb, true, err, st);
  return cudaErrorNotSupported;
}

int64_t tf32_launches(int64_t m, int64_t n, int64_t k, int32_t nb, int32_t prec) {
  const bool real = prec == TN_R32_TF32 || prec == TN_R32_3XTF32;
  const int64_t tiles = prec == TN_C64_3XTF32 || prec == TN_R32_3XTF32
                            ? tc3t_tiles(m, n, tc3t_bt(m, n, k, nb, real))
                            : tf32_tiles(m, n, real);
  const int64_t per = sm_band_tiles(tiles, nb);
  return (tiles + per - 1) / per;
}

}  // namespace tn
