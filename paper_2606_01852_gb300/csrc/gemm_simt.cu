// CUDA-core pairwise steps (sm_103a): C[b] = A[b] (m x k) . B[b] (n x k)^T in FP32 FMAs (or
// max-plus), any shape, written through the separable row/column offset maps.
//
// What bounds it: the FP32 pipe (128 FMAs per clock and SM) once k is a few tens, the output's
// stores below that. One kernel template, three tile shapes: every output is one thread's
// accumulator with k in order, so all shapes give the same bits and the choice is free
// (launch_form). A warp owns an (8 TM) x (4 TN) block of the tile, thread (lane / 4, lane % 4) the
// TM x TN outputs of it; both operands sit in shared memory k-major, so a complex 4 x 8 thread
// tile issues 128 FMAs per six 16-byte shared-memory loads. Global loads are 16 bytes along k
// (scalar when k or the planes are not 4-aligned), one k-block ahead of the arithmetic in
// registers, into the buffer the previous block is not read from: one barrier per 16 terms.
// The stored column is XORed with 8 x (k / 4 % 4), which spreads a warp's transposing stores
// over all banks and keeps 4-column runs whole.
//
// Max-plus: two terms of k side by side in shared memory, one packed add (add.rn.f32x2) and one
// three-input maximum per pair: 1 + 1 instructions for two terms instead of 2 + 2, and the
// maximum's half-rate pipe works once per pair. Maxima are exact, so the pairing changes nothing.
//
// The FMAs are packed, two columns at a time (fma.rn.f32x2): with three different registers read
// per instruction a scalar FMA issues at 82 lanes per clock and SM, a packed one at 2 x 53
// (measured), and each half rounds as the scalar one does.
//
// Measured (GB300, 77 TFLOP/s of FP32 FMA; one scalar FMA per term, 64 x 64 tiles and loads
// waited for in place before): complex 2048 x 8192 x 1024 3.88 -> 2.30 ms (35.4 -> 59.7 TFLOP/s),
// 1024 x 4096 x 16384 16.1 -> 9.5 ms; real 2048 x 8192 x 1024 1.30 -> 0.68 ms (26.5 -> 50.2);
// max-plus the same 1.60 -> 1.16 ms (21.5 -> 29.6); few outputs, complex 32 x 2048 x 2048
// 180 -> 54 us; shallow, complex 2048 x 16384 x 4 311 -> 108 us (0.87 -> 2.5 TB/s). What is left
// is the shared-memory read bandwidth: a 16-byte load returns 512 bytes to a warp in 4 clocks,
// 75 % (complex) or all (real, max-plus) of the packed instructions' time. Larger thread tiles
// (8 x 16) cut that but leave 8 warps on an SM: slower (42.8 TFLOP/s real).
//
// The epilogue puts each warp's 32 x 32 blocks through shared memory and stores them in address
// order (store_block): with interleaved consumer orders a row of outputs is scattered in runs of
// a few elements, and the shallow steps (k <= 16) are bound by these stores.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "kernels.h"
#include "scale.cuh"
#include "split_bf16.cuh"
#include "tc_common.cuh"
#include "pdl.cuh"

namespace tn {
namespace {

enum class Arith { Complex, Real, MaxPlus };

constexpr int kSBK = 16;  // terms of k per shared-memory buffer

template <Arith AR, int TM_, int TN_, int WM_, int WN_>
struct SimtCfg {
  static constexpr Arith ar = AR;
  static constexpr int TM = TM_, TN = TN_, WM = WM_, WN = WN_;  // thread tile, warps per tile side
  static constexpr int M = 8 * TM * WM, N = 4 * TN * WN;        // output tile
  static constexpr int THREADS = 32 * WM * WN;
  static constexpr int NP = AR == Arith::Complex ? 2 : 1;
  static constexpr int BUF = NP * kSBK * (M + N);               // floats of one buffer
  static constexpr int BLK = NP * 32 * 33;                      // floats of one staged 32 x 32 block
  static constexpr int BLOCKS = (M / 32) * (N / 32);
  // blocks staged at a time: one per warp (a warp of several blocks stages them in turn)
  static constexpr int STAGED = BLOCKS < WM * WN ? BLOCKS : WM * WN;
  // resident CTAs per SM the registers are cut for
  static constexpr int MIN_CTAS = THREADS == 256 ? 2 : (TM * TN * NP >= 32 ? 3 : 4);
  static constexpr int SMEM = 4 * (2 * BUF > STAGED * BLK ? 2 * BUF : STAGED * BLK);
};

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Two FP32 values side by side in a 64-bit register (the packed instructions' operand).
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(f2 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ void fma2(f2& c, f2 a, f2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// The values of R consecutive rows (R = 2, 4 or a multiple of 8) from row x0 of one stored k, W
// floats each (max-plus: a pair of terms), undoing the XOR by sw, which moves whole runs of 8.
template <int R, int W>
__device__ __forceinline__ void lds(float (&v)[R * W], const float* p, int x0, int sw) {
  if constexpr (R * W == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p + (x0 ^ sw));
    v[0] = x.x;
    v[1] = x.y;
  } else {
    constexpr int RUN = R < 8 ? R : 8;
#pragma unroll
    for (int r = 0; r < R; r += RUN)
#pragma unroll
      for (int h = 0; h < RUN * W; h += 4) {
        const float4 x = *reinterpret_cast<const float4*>(p + W * ((x0 + r) ^ sw) + h);
        v[r * W + h] = x.x;
        v[r * W + h + 1] = x.y;
        v[r * W + h + 2] = x.z;
        v[r * W + h + 3] = x.w;
      }
  }
}

// One operand tile of ROWS rows, k0 .. k0 + 15: global to registers, registers to shared
// memory. Element (row, k) sits at [k][row ^ sw(k)] (max-plus: the pair (k, k + 1) at
// [k / 2][row ^ sw(k)]), sw(k) = 8 (k / 4 % 4).
template <int ROWS, int THREADS, bool PAIRS>
struct Tile {
  static constexpr int Q = ROWS * (kSBK / 4);            // 4-term pieces
  static constexpr int PER = (Q + THREADS - 1) / THREADS;
  const float* p[PER];  // this thread's pieces of the rows, at k = 0 (null: row out of range)

  __device__ __forceinline__ void init(const float* X, int64_t r0, int64_t rows, int64_t k) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int idx = threadIdx.x + i * THREADS;
      const int64_t r = r0 + (idx >> 2);
      p[i] = idx < Q && r < rows ? X + r * k + 4 * (idx & 3) : nullptr;
    }
  }
  // the pieces at k0 of the plane at +plane floats; left: terms of k from this thread's first
  __device__ __forceinline__ void load(float4 (&v)[PER], int64_t plane, int64_t k0, int64_t left, bool vec,
                                       float fill) const {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      v[i] = make_float4(fill, fill, fill, fill);
      if (p[i] == nullptr || left <= 0) continue;
      const float* x = p[i] + plane + k0;
      if (vec) {
        v[i] = *reinterpret_cast<const float4*>(x);
      } else {
        v[i].x = x[0];
        if (left > 1) v[i].y = x[1];
        if (left > 2) v[i].z = x[2];
        if (left > 3) v[i].w = x[3];
      }
    }
  }
  // s: the operand's exact power of two (exponent scaling; 1 without), applied here and not at
  // the load, where it would wait for the value before the block's arithmetic
  __device__ __forceinline__ void store(const float4 (&w)[PER], float* S, float s) const {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int idx = threadIdx.x + i * THREADS;
      if (idx >= Q) break;
      const float4 v = make_float4(w[i].x * s, w[i].y * s, w[i].z * s, w[i].w * s);
      const int r = idx >> 2, q = idx & 3, c = r ^ (8 * q);
      if constexpr (PAIRS) {
        float2* P = reinterpret_cast<float2*>(S);
        P[(2 * q) * ROWS + c] = make_float2(v.x, v.y);
        P[(2 * q + 1) * ROWS + c] = make_float2(v.z, v.w);
      } else {
        S[(4 * q) * ROWS + c] = v.x;
        S[(4 * q + 1) * ROWS + c] = v.y;
        S[(4 * q + 2) * ROWS + c] = v.z;
        S[(4 * q + 3) * ROWS + c] = v.w;
      }
    }
  }
};

// A thread's accumulators: pairs of columns (the packed FMAs' two halves), or single values in
// the max-plus form.
template <typename G>
struct Acc {
  static constexpr bool kPairs = G::ar != Arith::MaxPlus;
  static constexpr int W = kPairs ? G::TN / 2 : G::TN;
  using T = std::conditional_t<kPairs, f2, float>;
  T re[G::TM][W];
  T im[G::NP == 2 ? G::TM : 1][G::NP == 2 ? W : 1];

  __device__ __forceinline__ void init(float zero) {
#pragma unroll
    for (int i = 0; i < G::TM; ++i)
#pragma unroll
      for (int j = 0; j < W; ++j) {
        if constexpr (kPairs) re[i][j] = pack2(zero, zero);
        else re[i][j] = zero;
        if constexpr (G::NP == 2) im[i][j] = pack2(0.f, 0.f);
      }
  }
  // output (i, 2 j) and (i, 2 j + 1)
  __device__ __forceinline__ void get(int i, int j, float& r0, float& r1, float& i0, float& i1) const {
    if constexpr (kPairs) {
      unpack2(re[i][j], r0, r1);
    } else {
      r0 = re[i][2 * j];
      r1 = re[i][2 * j + 1];
    }
    if constexpr (G::NP == 2) unpack2(im[i][j], i0, i1);
    else i0 = i1 = 0.f;
  }
};

// the terms kk (and kk + 1, max-plus) of one shared-memory buffer
template <typename G>
__device__ __forceinline__ void mac(Acc<G>& acc, const float* buf, int kk, int row, int col) {
  constexpr int TM = G::TM, TN = G::TN;
  const float* As = buf;
  const float* Bs = buf + G::NP * kSBK * G::M;
  const int sw = 8 * ((kk >> 2) & 3);
  if constexpr (G::ar == Arith::MaxPlus) {
    float a[2 * TM], b[2 * TN];
    lds<TM, 2>(a, As + (kk >> 1) * 2 * G::M, row, sw);
    lds<TN, 2>(b, Bs + (kk >> 1) * 2 * G::N, col, sw);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        float t0, t1;
        unpack2(add2(pack2(a[2 * i], a[2 * i + 1]), pack2(b[2 * j], b[2 * j + 1])), t0, t1);
        acc.re[i][j] = max3(acc.re[i][j], t0, t1);
      }
  } else {
    float ar[TM], br[TN];
    lds<TM, 1>(ar, As + kk * G::M, row, sw);
    lds<TN, 1>(br, Bs + kk * G::N, col, sw);
    if constexpr (G::ar == Arith::Complex) {
      float ai[TM], bi[TN];
      lds<TM, 1>(ai, As + kSBK * G::M + kk * G::M, row, sw);
      lds<TN, 1>(bi, Bs + kSBK * G::N + kk * G::N, col, sw);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f2 xr = pack2(ar[i], ar[i]), xi = pack2(ai[i], ai[i]), nxi = pack2(-ai[i], -ai[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
          const f2 yr = pack2(br[2 * j], br[2 * j + 1]), yi = pack2(bi[2 * j], bi[2 * j + 1]);
          fma2(acc.re[i][j], xr, yr);
          fma2(acc.re[i][j], nxi, yi);
          fma2(acc.im[i][j], xr, yi);
          fma2(acc.im[i][j], xi, yr);
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f2 x = pack2(ar[i], ar[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) fma2(acc.re[i][j], x, pack2(br[2 * j], br[2 * j + 1]));
      }
    }
  }
}

template <typename G>
__global__ void __launch_bounds__(G::THREADS, G::MIN_CTAS) contract_simt_kernel(StepArgs a) {
  constexpr bool CPLX = G::ar == Arith::Complex, MP = G::ar == Arith::MaxPlus;
  constexpr int TM = G::TM, TN = G::TN;
  extern __shared__ __align__(16) float sm[];
  const float fill = MP ? __int_as_float(0xff800000) : 0.f;  // the semiring's zero
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  pdl_next();
  const int64_t tiles_n = (a.n + G::N - 1) / G::N;
  const int64_t tile = blockIdx.x;
  const int64_t m0 = (tile / tiles_n) * G::M, n0 = (tile % tiles_n) * G::N;
  const int b = blockIdx.y;
  const float* A = a.A + b * a.a_bstride;
  const float* B = a.B + b * a.b_bstride;
  float* C = a.C + b * a.c_bstride;
  // this CTA's part of k (all of it unless the step is split, blockIdx.z = part)
  const int64_t kc = a.ksplit > 1 ? ((a.k + a.ksplit - 1) / a.ksplit + kSBK - 1) / kSBK * kSBK : a.k;
  const int64_t kbeg = blockIdx.z * kc, kend = kbeg + kc < a.k ? kbeg + kc : a.k;
  const bool vec = (a.k & 3) == 0 && ((a.a_plane | a.b_plane) & 3) == 0 &&
                   ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
  float sa = 1.f, sb = 1.f;
  if (a.recs) {
    sa = pow2_neg(scale_exp(a.recs + a.rec_a + (a.a_bstride ? b : 0)));
    sb = pow2_neg(scale_exp(a.recs + a.rec_b + (a.b_bstride ? b : 0)));
  }
  const int wrow = (warp / G::WN) * 8 * TM, wcol = (warp % G::WN) * 4 * TN;  // the warp's block in the tile
  const int row = wrow + (lane >> 2) * TM, col = wcol + (lane & 3) * TN;     // this thread's outputs
  Acc<G> acc;
  acc.init(fill);

  using TA = Tile<G::M, G::THREADS, MP>;
  using TB = Tile<G::N, G::THREADS, MP>;
  TA ta;
  TB tb;
  ta.init(A, m0, a.m, a.k);
  tb.init(B, n0, a.n, a.k);
  float4 va[G::NP][TA::PER], vb[G::NP][TB::PER];
  auto load = [&](int64_t k0) {
    const int64_t left = kend - k0 - 4 * (tid & 3);
#pragma unroll
    for (int p = 0; p < G::NP; ++p) {
      ta.load(va[p], p ? a.a_plane : 0, k0, left, vec, fill);
      tb.load(vb[p], p ? a.b_plane : 0, k0, left, vec, fill);
    }
  };
  auto store = [&](int s) {
    float* buf = sm + s * G::BUF;
#pragma unroll
    for (int p = 0; p < G::NP; ++p) {
      ta.store(va[p], buf + p * kSBK * G::M, sa);
      tb.store(vb[p], buf + G::NP * kSBK * G::M + p * kSBK * G::N, sb);
    }
  };
  load(kbeg);
  store(0);
  __syncthreads();
  int s = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += kSBK, s ^= 1) {
    const bool more = k0 + kSBK < kend;
    if (more) load(k0 + kSBK);  // in flight during this block's arithmetic
    const float* buf = sm + s * G::BUF;
    if (k0 + kSBK <= kend) {
#pragma unroll
      for (int kk = 0; kk < kSBK; kk += MP ? 2 : 1) mac<G>(acc, buf, kk, row, col);
    } else {  // the last, partial block: only its terms
      const int left = static_cast<int>(kend - k0);
      for (int kk = 0; kk < left; kk += MP ? 2 : 1) mac<G>(acc, buf, kk, row, col);
    }
    if (more) store(s ^ 1);  // the buffer read before the last barrier
    __syncthreads();
  }

  if (a.ksplit > 1) {
    // partial tile of this part of k, dense [part][b][plane][m][n]; combined and written
    // through the offset maps by simt_combine_kernel
    float* P0 = a.part + ((int64_t(blockIdx.z) * gridDim.y + b) * G::NP) * a.m * a.n;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int64_t m = m0 + row + i;
      if (m >= a.m) continue;
#pragma unroll
      for (int j = 0; j < TN / 2; ++j) {
        const int64_t n = n0 + col + 2 * j;
        float r[2], x[2];
        acc.get(i, j, r[0], r[1], x[0], x[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (n + e >= a.n) continue;
          P0[m * a.n + n + e] = r[e];
          if constexpr (CPLX) P0[a.m * a.n + m * a.n + n + e] = x[e];
        }
      }
    }
    return;
  }
  int lmax = -127;
  if (a.recs) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN / 2; ++j) {
        float r[2], x[2];
        acc.get(i, j, r[0], r[1], x[0], x[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (m0 + row + i >= a.m || n0 + col + 2 * j + e >= a.n) continue;
          lmax = max(lmax, exp_of(CPLX ? fmaxf(fabsf(r[e]), fabsf(x[e])) : fabsf(r[e])));
        }
      }
  }
  // epilogue: 32 x 32 blocks through shared memory (the buffers are free: the loop's last
  // barrier), stored in address order
  constexpr int CS = 32 * 33;
  auto block_out = [&](const float* t, int64_t br0, int64_t bc0, int part, int parts) {
    const int64_t r = br0 + lane, c = bc0 + lane;
    const bool rok = r < a.m, cok = c < a.n;
    store_block<!CPLX>(C, a.c_plane, a.c_split, t, 33, CS, rok ? map_offset(a.rows, r) : 0,
                       cok ? map_offset(a.cols, c) : 0, rok, cok, a.blk, lane, part, parts);
  };
  if constexpr (8 * TM >= 32) {
    // the warp's block is (8 TM) x (4 TN): its 32 x 32 blocks one after the other
    static_assert(4 * TN % 32 == 0, "whole 32 x 32 blocks");
    float* t = sm + warp * G::BLK;
#pragma unroll
    for (int h = 0; h < TM / 4; ++h)
#pragma unroll
      for (int w = 0; w < TN / 8; ++w) {
        // the lanes whose outputs are in this block
        if ((lane >> 2) / (32 / TM) == h && (lane & 3) / (32 / TN) == w) {
#pragma unroll
          for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) {
              const int o = ((lane >> 2) * TM + i - 32 * h) * 33 + (lane & 3) * TN + 2 * j - 32 * w;
              float r0, r1, x0, x1;
              acc.get(i, j, r0, r1, x0, x1);
              t[o] = r0;
              t[o + 1] = r1;
              if constexpr (CPLX) {
                t[CS + o] = x0;
                t[CS + o + 1] = x1;
              }
            }
        }
        __syncwarp();
        block_out(t, m0 + wrow + 32 * h, n0 + wcol + 32 * w, 0, 1);
        __syncwarp();
      }
  } else {
    // a 32 x 32 tile of four warps: one block, each warp storing a part of it
    static_assert(G::M == 32 && G::N == 32, "one staged block");
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN / 2; ++j) {
        const int o = (row + i) * 33 + col + 2 * j;
        float r0, r1, x0, x1;
        acc.get(i, j, r0, r1, x0, x1);
        sm[o] = r0;
        sm[o + 1] = r1;
        if constexpr (CPLX) {
          sm[CS + o] = x0;
          sm[CS + o + 1] = x1;
        }
      }
    __syncthreads();
    block_out(sm, m0, n0, warp, G::WM * G::WN);
  }
  if (a.recs) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lmax = max(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    ScaleRec* rc = a.recs + a.rec_c + (a.c_bstride ? b : 0);
    if (lane == 0) atomicMax(&rc->emax, lmax);
    if (tile == 0 && tid == 0) {
      const ScaleRec* ra = a.recs + a.rec_a + (a.a_bstride ? b : 0);
      const ScaleRec* rb = a.recs + a.rec_b + (a.b_bstride ? b : 0);
      rc->log2 = ra->log2 + rb->log2 + scale_exp(ra) + scale_exp(rb);
    }
  }
}

// Combine the k parts of a split SIMT step in part order (sum, or max for max-plus) and
// write C through the offset maps. One thread per output element of every batch entry.
__global__ void simt_combine_kernel(StepArgs a, int32_t nb, int32_t cplx) {
  pdl_wait();
  pdl_next();
  const int64_t mn = a.m * a.n, np = cplx ? 2 : 1;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nb * mn;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / mn, o = e - b * mn;
    const float* P0 = a.part + b * np * mn + o;
    const int64_t pstride = (int64_t)nb * np * mn;  // one part to the next
    float vr = P0[0], vi = cplx ? P0[mn] : 0.f;
    for (int s = 1; s < a.ksplit; ++s) {
      const float xr = P0[s * pstride];
      if (a.maxplus) {
        vr = fmaxf(vr, xr);
      } else {
        vr += xr;
        if (cplx) vi += P0[s * pstride + mn];
      }
    }
    const int64_t i = o / a.n, j = o - i * a.n;
    const int64_t off = map_offset(a.rows, i) + map_offset(a.cols, j);
    float* C = a.C + b * a.c_bstride;
    if (cplx) store_cplx(C, a.c_plane, off, vr, vi, a.c_split);
    else C[off] = vr;
  }
}

template <typename G>
void launch(const StepArgs& a, int32_t nb, cudaStream_t st) {
  static_assert(G::SMEM <= kDefaultSmem, "no allowance to set");
  const int64_t tiles = ((a.m + G::M - 1) / G::M) * ((a.n + G::N - 1) / G::N);
  dim3 grid((unsigned)tiles, (unsigned)nb, (unsigned)(a.ksplit > 1 ? a.ksplit : 1));
  launch_pdl(contract_simt_kernel<G>, grid, G::THREADS, G::SMEM, st, a);
}

// A tile shape's time per k term, in units of a full-rate 128 x 128 real (64 x 64 complex) tile:
// `share` of an SM whose `resident` CTAs run together, `alone` for a CTA without company (latency
// instead of throughput). From the shapes' rates: max-plus 29.6 / 26.9 / 19.3 TFLOP/s (128 x 128,
// 64 x 128, 64 x 64), real 50.2 / 41.5 (64 x 128, 64 x 64), complex 60 (64 x 64); and steps of few
// tiles: max-plus 256 128-square tiles 5.1 ms, the same as 512 64 x 128 ones 7.2 ms.
struct TileCost {
  double share, alone;
  int resident;
  double time(int64_t ctas, int num_sms) const {
    const int64_t n = (ctas + num_sms - 1) / num_sms, rest = n % resident;
    return double(n - rest) * share + (rest ? std::max(double(rest) * share, alone) : 0.0);
  }
};

// The tile of a step: the least time by TileCost (the bits do not depend on it). Large tiles have
// the better rate; with few outputs a step is bound by its serial k loop, and small tiles spread
// it over more SMs.
template <Arith AR>
void launch_form(const StepArgs& a, int32_t nb, int num_sms, cudaStream_t st) {
  auto ctas = [&](int64_t tm, int64_t tn) {
    return ((a.m + tm - 1) / tm) * ((a.n + tn - 1) / tn) * nb * (a.ksplit > 1 ? a.ksplit : 1);
  };
  using Widest = SimtCfg<AR, 8, 8, 2, 4>;
  using Wide = SimtCfg<AR, 8, 8, 1, 4>;
  using Square = SimtCfg<AR, 4, 8, 2, 2>;
  using Small = SimtCfg<AR, 2, 4, 2, 2>;
  constexpr bool kCplx = AR == Arith::Complex, kMax = AR == Arith::MaxPlus;
  constexpr TileCost square = kCplx ? TileCost{1.0, 1.8, 3} : (kMax ? TileCost{0.39, 0.6, 3} : TileCost{0.30, 0.5, 3});
  constexpr TileCost small = kCplx ? TileCost{0.43, 0.75, 4} : (kMax ? TileCost{0.14, 0.25, 4} : TileCost{0.11, 0.22, 4});
  const double t_square = square.time(ctas(Square::M, Square::N), num_sms);
  const double t_small = small.time(ctas(Small::M, Small::N), num_sms);
  const double t_rest = std::min(t_square, t_small);
  if constexpr (!kCplx) {  // real outputs take half the registers: an 8 x 8 thread tile
    constexpr TileCost wide = kMax ? TileCost{0.55, 1.0, 3} : TileCost{0.5, 0.9, 3};
    const double t_wide = wide.time(ctas(Wide::M, Wide::N), num_sms);
    if constexpr (kMax) {
      constexpr TileCost widest{1.0, 1.2, 2};
      const double t_widest = widest.time(ctas(Widest::M, Widest::N), num_sms);
      if (t_widest <= t_wide && t_widest <= t_rest) return launch<Widest>(a, nb, st);
    }
    if (t_wide <= t_rest) return launch<Wide>(a, nb, st);
  }
  if (t_square <= t_small) launch<Square>(a, nb, st);
  else launch<Small>(a, nb, st);
}

}  // namespace

int32_t simt_ksplit(int64_t m, int64_t n, int64_t k, int64_t copies, int num_sms, bool scaled) {
  if (scaled || k < 2048) return 1;
  // aim at four 64 x 64 tiles per SM
  const int64_t tiles = ((m + 63) / 64) * ((n + 63) / 64) * copies;
  if (tiles >= 2 * int64_t(num_sms)) return 1;
  int64_t s = (4 * int64_t(num_sms) + tiles - 1) / tiles;
  s = std::min<int64_t>(s, k / 1024);
  s = std::min<int64_t>(s, 32);
  return s > 1 ? int32_t(s) : 1;
}

void launch_contract_simt(const StepArgs& a, int32_t nb, bool cplx, int num_sms, cudaStream_t st) {
  if (cplx) launch_form<Arith::Complex>(a, nb, num_sms, st);
  else if (a.maxplus) launch_form<Arith::MaxPlus>(a, nb, num_sms, st);
  else launch_form<Arith::Real>(a, nb, num_sms, st);
  if (a.ksplit > 1) {
    const int64_t total = int64_t(nb) * a.m * a.n;
    const unsigned blocks = (unsigned)std::min<int64_t>((total + 255) / 256, 4096);
    launch_pdl(simt_combine_kernel, blocks, 256, 0, st, a, nb, cplx ? 1 : 0);
  }
}

}  // namespace tn
