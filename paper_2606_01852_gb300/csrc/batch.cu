// Batched independent small networks in one persistent launch.
//
// Each network has its own path and its own plan (the same planner as tn_plan: step
// analysis, GEMM-oriented reordering of Sec. IV-A, liveness offsets), flattened into
// compact device tables (one copy for all networks of one shape and path). One CTA, or one
// warp, takes the next network from an atomic queue and runs its whole path: stage the leaves
// into the network's arena (planned orders), then for each step C = A (m x k) . B (n x k)^T
// written through the output offset maps. With exponent scaling each tensor counts as
// renormalised by an exact power of two chosen from its largest entry: the step's stores also
// take the maximum, and whoever reads the tensor multiplies by the power of two, so that a step
// has one pass and one barrier. The exponents are summed per network in an int64; the network's
// result is (value, log2 scale) and ln|Z| = ln|value| + log2 * ln 2 in FP64 on the host side. In
// the max-plus semiring (real, unscaled) a step is C = max_k (A + B) instead.
//
// What bounds it: latency, of the steps one after another (tens per network, most of them under
// 100 terms) and, in the few large steps, of the loads whose lanes are k floats apart. So
// small steps run one output per thread with no table and no division, steps of at least 8
// outputs per thread run 4 x 4 (complex: 4 x 2) outputs per thread with 16-byte loads, and the
// networks are queued by falling cost so that the large ones do not end last. 4096 Ising
// networks of 20-60 vertices: 3.98 -> 0.60 ms (0.89 ms in the caller's order and with 64
// registers a thread, 0.64 ms with 80, 0.60 with 128: the tiles want registers more than the
// small steps want warps), 0.58 with the step records in shared memory, 0.38 with run_panels;
// 1024 king's graphs of 4-7 a side, max-plus: 14.0 -> 1.8 -> 0.89 ms. A small step is now ~1300
// clocks: 200-300 for its record, 850 for an output, 250 for the maximum and the barrier.
// The CTA width (threads per network) and CTAs per SM are chosen by an autotuner that
// times the real batch; the launch (queue reset + kernel) can be replayed as a CUDA graph.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <numeric>
#include <string>
#include <unordered_map>
#include <vector>

#include <cuda_runtime.h>

#include "batch.h"
#include "kernels.h"
#include "tn_internal.h"

namespace tn {
namespace {

__device__ __forceinline__ float bpow2_neg(int e) {
  e = max(-126, min(127, e));
  return __int_as_float((127 - e) << 23);
}

// The threads that run one network: a whole CTA, or one warp.
template <bool WARP>
struct Team {
  static __device__ __forceinline__ int rank() { return WARP ? threadIdx.x & 31 : threadIdx.x; }
  static __device__ __forceinline__ int size() { return WARP ? 32 : blockDim.x; }
  static __device__ __forceinline__ void sync() {
    if (WARP) __syncwarp();
    else __syncthreads();
  }
};

// The offset of index x under a digit map of nd digits (arrays 16-byte aligned; places beyond nd
// are 0, so four are taken without a branch).
__device__ __forceinline__ int map_offset(const int32_t* ext, const int32_t* str, int nd, bool pow2, int x) {
  int off = 0;
  if (pow2) {
    const int4 e = *reinterpret_cast<const int4*>(ext), st = *reinterpret_cast<const int4*>(str);
    off = ((x >> (e.x & 31)) & (e.x >> 8)) * st.x + ((x >> (e.y & 31)) & (e.y >> 8)) * st.y +
          ((x >> (e.z & 31)) & (e.z >> 8)) * st.z + ((x >> (e.w & 31)) & (e.w >> 8)) * st.w;
#pragma unroll 1
    for (int d = 4; d < nd; ++d) off += ((x >> (ext[d] & 31)) & (ext[d] >> 8)) * str[d];
  } else {
    for (int d = nd - 1; d >= 0; --d) {
      const int w = ext[d];
      off += (x % w) * str[d];
      x /= w;
    }
  }
  return off;
}

// Output offset of row x (x < m) or of column x - m (x >= m) of step S.
__device__ __forceinline__ int step_offset(const BStep* S, int nr, int nc, bool pow2, int m, int x) {
  return x < m ? map_offset(S->rext, S->rstr, nr, pow2, x) : map_offset(S->cext, S->cstr, nc, pow2, x - m);
}

template <int KV>
__device__ __forceinline__ void load_k(const float* p, float s, float (&v)[KV]) {
  if constexpr (KV == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x * s, v[1] = x.y * s, v[2] = x.z * s, v[3] = x.w * s;
  } else if constexpr (KV == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x * s, v[1] = x.y * s;
  } else {
    v[0] = *p * s;
  }
}

// RM x RN outputs of one thread, each its own chain over k in order (so an output's bits do not
// depend on the tile it is computed in): rows a + ra[r], columns b + rb[c], KV terms per load.
template <bool MAXPLUS, int RM, int RN>
__device__ __forceinline__ void dot_init(float (&cr)[RM][RN], float (&ci)[RM][RN]) {
#pragma unroll
  for (int r = 0; r < RM; ++r)
#pragma unroll
    for (int c = 0; c < RN; ++c) {
      cr[r][c] = MAXPLUS ? __int_as_float(0xff800000) : 0.f;  // max-plus: its zero is -inf, its product +
      ci[r][c] = 0.f;
    }
}
template <bool CPLX, bool MAXPLUS, int RM, int RN, int KV>
__device__ __forceinline__ void dot_tile(const float* a, int ai, const int (&ra)[RM], const float* b, int bi,
                                         const int (&rb)[RN], int k, float sa, float sb, float (&cr)[RM][RN],
                                         float (&ci)[RM][RN]) {
#pragma unroll(RM * RN == 1 ? 4 : 1)
  for (int t = 0; t < k; t += KV) {
    float xr[RM][KV], xi[RM][KV];
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      load_k<KV>(a + ra[r] + t, sa, xr[r]);
      if (CPLX) load_k<KV>(a + ai + ra[r] + t, sa, xi[r]);
    }
#pragma unroll
    for (int c = 0; c < RN; ++c) {
      float yr[KV], yi[KV];
      load_k<KV>(b + rb[c] + t, sb, yr);
      if (CPLX) load_k<KV>(b + bi + rb[c] + t, sb, yi);
#pragma unroll
      for (int q = 0; q < KV; ++q)
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          if (CPLX) {
            cr[r][c] = fmaf(xr[r][q], yr[q], fmaf(-xi[r][q], yi[q], cr[r][c]));
            ci[r][c] = fmaf(xr[r][q], yi[q], fmaf(xi[r][q], yr[q], ci[r][c]));
          } else if (MAXPLUS) {
            cr[r][c] = fmaxf(cr[r][c], xr[r][q] + yr[q]);
          } else {
            cr[r][c] = fmaf(xr[r][q], yr[q], cr[r][c]);
          }
        }
    }
  }
}

// One step in the arena `ar` by the team; returns the largest output's bits (sign cleared), this
// thread's outputs only. RM x RN tiles are dealt to warps in patches of 32 >> bj by 1 << bj
// threads, a thread's rows tm apart and its columns tn apart, so that neighbouring threads read
// neighbouring rows. 1 x 1: output o to thread o, in order.
template <bool CPLX, bool MAXPLUS, bool WARP, int RM, int RN, int KV>
__device__ __forceinline__ int run_step(float* ar, const BStep* S, int m, int n, int k, int nr, int nc,
                                        bool pow2, int a, int b, int c, float sa, float sb, const int* tab) {
  int mx = 0;
  float cr[RM][RN], ci[RM][RN];
  auto store = [&](int off, float vr, float vi) {
    ar[c + off] = vr;
    float v = fabsf(vr);
    if (CPLX) {
      ar[c + m * n + off] = vi;
      v = fmaxf(v, fabsf(vi));
    }
    mx = max(mx, __float_as_int(v));
  };
  if constexpr (RM == 1) {
    const int nsh = (n & (n - 1)) == 0 ? 31 - __clz(n) : -1;
    for (int o = Team<WARP>::rank(); o < m * n; o += Team<WARP>::size()) {
      const int i = nsh >= 0 ? o >> nsh : o / n, j = o - i * n;
      const int ra[1] = {i * k}, rb[1] = {j * k};
      dot_init<MAXPLUS>(cr, ci);
      dot_tile<CPLX, MAXPLUS, 1, 1, KV>(ar + a, m * k, ra, ar + b, n * k, rb, k, sa, sb, cr, ci);
      store(map_offset(S->rext, S->rstr, nr, pow2, i) + map_offset(S->cext, S->cstr, nc, pow2, j), cr[0][0], ci[0][0]);
    }
  } else {
    const int tm = (m + RM - 1) / RM, tn = (n + RN - 1) / RN;
    const int bj = tn >= 8 ? 3 : tn >= 4 ? 2 : tn >= 2 ? 1 : 0;
    const int lane = threadIdx.x & 31;
    const int li = lane >> bj, lj = lane & ((1 << bj) - 1);
    const int pn = (tn + (1 << bj) - 1) >> bj, pm = (tm + (32 >> bj) - 1) >> (5 - bj);
    for (int p = Team<WARP>::rank() >> 5; p < pm * pn; p += Team<WARP>::size() >> 5) {
      const int pi = p / pn, pj = p - pi * pn;
      const int ti = (pi << (5 - bj)) + li, tj = (pj << bj) + lj;
      if (ti >= tm || tj >= tn) continue;
      int ra[RM], rb[RN];
#pragma unroll
      for (int r = 0; r < RM; ++r) ra[r] = min(ti + r * tm, m - 1) * k;
#pragma unroll
      for (int q = 0; q < RN; ++q) rb[q] = min(tj + q * tn, n - 1) * k;
      dot_init<MAXPLUS>(cr, ci);
      dot_tile<CPLX, MAXPLUS, RM, RN, KV>(ar + a, m * k, ra, ar + b, n * k, rb, k, sa, sb, cr, ci);
#pragma unroll
      for (int q = 0; q < RN; ++q) {
        const int j = tj + q * tn;
        if (j >= n) continue;
        const int oc = tab ? tab[m + j] : map_offset(S->cext, S->cstr, nc, pow2, j);
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          const int i = ti + r * tm;
          if (i < m) store((tab ? tab[i] : map_offset(S->rext, S->rstr, nr, pow2, i)) + oc, cr[r][q], ci[r][q]);
        }
      }
    }
  }
  return mx;
}

// A step of a network whose arena is in global memory: its operands' rows are k floats apart, and
// lanes that read their own rows touch a line each, eight times over. Here 32 terms of the rows of a
// (4 G) x 32 tile of outputs (G = threads / 8) are brought into shared memory by whole lines, and each
// thread's 4 x 4 outputs run over them, k in order as everywhere: the same bits. The rows are
// the larger operand's, 36 floats apart (a quarter warp's 16-byte reads then meet different
// banks). A 32 x 16 x 512 step was 88 us of its CTA and a 64 x 256 x 16 one 47: 4096 Ising networks
// 0.58 -> 0.38 ms, 1024 king's graphs 1.80 -> 0.89 ms.
constexpr int kPanelRow = 36;
__host__ __device__ constexpr int panel_floats(int threads) { return (threads / 2 + 32) * kPanelRow; }

template <bool MAXPLUS>
__device__ __forceinline__ int run_panels(float* ar, const BStep* S, int m, int n, int k, int nr, int nc, bool pow2,
                                          int a, int b, int c, float sa, float sb, const int* tab, float* panel) {
  const int tid = threadIdx.x, T = blockDim.x, G = T >> 3;
  const bool by_a = m >= n;
  const float* P = ar + (by_a ? a : b);
  const float* Q = ar + (by_a ? b : a);
  const float sp = by_a ? sa : sb, sq = by_a ? sb : sa;
  const int np = by_a ? m : n, nq = by_a ? n : m;
  const int ti = tid >> 3, tj = tid & 7;
  float* pq = panel + 4 * G * kPanelRow;
  int ra[4], rb[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    ra[r] = (ti + G * r) * kPanelRow;
    rb[r] = (tj + 8 * r) * kPanelRow;
  }
  int mx = 0;
  for (int p0 = 0; p0 < np; p0 += 4 * G)
    for (int q0 = 0; q0 < nq; q0 += 32) {
      float cr[4][4], ci[4][4];
      dot_init<MAXPLUS>(cr, ci);
      for (int t0 = 0; t0 < k; t0 += 32) {
        const int kc = min(32, k - t0), t = t0 + 4 * tj;
        __syncthreads();  // the panels' last reads
        if (4 * tj < kc) {
          for (int r = ti; r < 4 * G && p0 + r < np; r += G) {
            float v[4];
            load_k<4>(P + (p0 + r) * k + t, sp, v);
            *reinterpret_cast<float4*>(panel + r * kPanelRow + 4 * tj) = make_float4(v[0], v[1], v[2], v[3]);
          }
          for (int r = ti; r < 32 && q0 + r < nq; r += G) {
            float v[4];
            load_k<4>(Q + (q0 + r) * k + t, sq, v);
            *reinterpret_cast<float4*>(pq + r * kPanelRow + 4 * tj) = make_float4(v[0], v[1], v[2], v[3]);
          }
        }
        __syncthreads();
        dot_tile<false, MAXPLUS, 4, 4, 4>(panel, 0, ra, pq, 0, rb, kc, 1.f, 1.f, cr, ci);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int p = p0 + ti + G * x, q = q0 + tj + 8 * y;
          if (p >= np || q >= nq) continue;
          const int i = by_a ? p : q, j = by_a ? q : p;
          ar[c + (tab ? tab[i] + tab[m + j]
                      : map_offset(S->rext, S->rstr, nr, pow2, i) + map_offset(S->cext, S->cstr, nc, pow2, j))] = cr[x][y];
          mx = max(mx, __float_as_int(fabsf(cr[x][y])));
        }
    }
  return mx;
}

// CTAs of at most this many threads take the form with register tiles (128 registers a thread);
// wider ones, which the autotuner does not try, run one output per thread
constexpr int kTileThreads = 256;

// leaves above this many elements are staged by the whole team, the others by groups of 8 threads
constexpr int kGroupLeaf = 64;

template <bool CPLX, bool MAXPLUS, bool WARP, bool TILES>
__global__ void __launch_bounds__(TILES ? kTileThreads : 1024, TILES ? 2 : 1)
batch_kernel(const BNet* __restrict__ nets, const BLeaf* __restrict__ leaves, const BStep* __restrict__ steps,
             int32_t n_nets, const float* __restrict__ packed, float* arena, int32_t* queue, int32_t scaling,
             double* values, double* logs, int32_t smem_arena, int32_t tab_ints) {
  // dynamic shared memory: [arenas: smem_arena floats per team | offset tables: tab_ints per team]
  extern __shared__ __align__(16) float s_arena[];
  __shared__ int s_exp[kExpBytes / 4];  // the step outputs' largest exponents: ints, or bytes (+127) per warp
  __shared__ int s_net;
  __shared__ long long s_log;
  constexpr int kRec = sizeof(BStep) / 16;
  __shared__ int4 s_step[2][WARP ? 1 : kRec];  // this step's record and the next one's
  using T = Team<WARP>;
  constexpr int RM = 4, RN = CPLX ? 2 : 4;
  const int teams = WARP ? blockDim.x >> 5 : 1, team = WARP ? threadIdx.x >> 5 : 0;
  const int rank = T::rank(), size = T::size(), lane = threadIdx.x & 31;
  int* s_tab = reinterpret_cast<int*>(s_arena + smem_arena * teams) + team * tab_ints;
  const int exp_cap = WARP ? kExpBytes / teams : kExpBytes / 4;
  uint8_t* w_exp = reinterpret_cast<uint8_t*>(s_exp) + (WARP ? team * exp_cap : 0);
  while (true) {
    int w = 0;
    if (WARP) {
      if (lane == 0) w = atomicAdd(queue, 1);
      w = __shfl_sync(0xffffffffu, w, 0);
    } else {
      if (rank == 0) {
        s_net = atomicAdd(queue, 1);
        s_log = 0;
      }
      __syncthreads();
      w = s_net;
    }
    if (w >= n_nets) break;
    const BNet net = nets[w];
    // the network's arena: in shared memory when it fits the launch's shared-memory arena
    // (smem_arena floats per team), else its own slice of the global batch arena
    float* ar = net.arena_floats <= smem_arena ? s_arena + team * smem_arena : arena + net.arena;
    const float* in = packed + net.in * (CPLX ? 2 : 1);
    const BLeaf* L0 = leaves + net.leaf0;
    const BStep* S0 = steps + net.step0;
    const bool defer = net.n_steps <= exp_cap;
    long long lsum = 0;  // this thread's share of the exponents' sum
    if (!WARP && scaling)
      for (int i = rank; i < min(max(net.n_steps, 2), exp_cap); i += size) s_exp[i] = -127;
    if (!WARP && rank < kRec && net.n_steps > 0) s_step[0][rank] = __ldg(reinterpret_cast<const int4*>(S0) + rank);
    // Leaves (declared order -> planned order; complex64 -> planar), each scaled by its own exact
    // power of two: small ones by groups of 8 threads, whose own elements they scale
    bool big = false;
    for (int l0 = 0; l0 < net.n_leaves; l0 += size >> 3) {
      const int l = l0 + (rank >> 3), sub = lane & 7;
      int4 h = make_int4(0, 0, 0, 0);
      if (l < net.n_leaves) h = __ldg(reinterpret_cast<const int4*>(L0 + l));
      big = big || h.z > kGroupLeaf;
      const bool mine = h.z <= kGroupLeaf;
      int mx = 0;
      if (mine)
        for (int e = sub; e < h.z; e += 8) {
          const int src = h.x + map_offset(L0[l].ext, L0[l].sstride, h.w & 0xff, h.w < 0, e);
          if (CPLX) {
            const float2 v = reinterpret_cast<const float2*>(in)[src];
            ar[h.y + e] = v.x;
            ar[h.y + h.z + e] = v.y;
            mx = max(mx, __float_as_int(fmaxf(fabsf(v.x), fabsf(v.y))));
          } else {
            const float v = in[src];
            ar[h.y + e] = v;
            mx = max(mx, __float_as_int(fabsf(v)));
          }
        }
      if (!MAXPLUS && scaling) {
        for (int o = 4; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        int e = (mx >> 23) - 127;
        if (e < -126) e = 0;  // an all-zero leaf is left as is
        if (mine && e != 0) {
          const float sc = bpow2_neg(e);
          for (int i = sub; i < h.z; i += 8) {
            ar[h.y + i] *= sc;
            if (CPLX) ar[h.y + h.z + i] *= sc;
          }
          if (sub == 0) lsum += e;
        }
      }
    }
    // the largest exponent over the team, every thread's answer; slot: two taken in turn
    auto team_exp = [&](int mx, int slot) {
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (!WARP) {
        if (lane == 0) atomicMax(&s_exp[slot], (mx >> 23) - 127);
        __syncthreads();
        const int e = s_exp[slot];
        if (rank == 0) s_exp[slot ^ 1] = -127;  // read by nobody until the barrier after the scaling
        return e;
      }
      return (mx >> 23) - 127;
    };
    auto scale_in_place = [&](int off, int elems, int e) {
      if (e < -126) e = 0;
      if (e != 0) {
        const float sc = bpow2_neg(e);
        for (int i = rank; i < elems * (CPLX ? 2 : 1); i += size) ar[off + i] *= sc;
      }
      if (rank == 0) lsum += e;
      T::sync();
    };
    if (WARP) __syncwarp();
    if (WARP ? __any_sync(0xffffffffu, big) : __syncthreads_or(big)) {
      int turn = 0;
      for (int l = 0; l < net.n_leaves; ++l) {
        const int4 h = __ldg(reinterpret_cast<const int4*>(L0 + l));
        if (h.z <= kGroupLeaf) continue;
        int mx = 0;
        for (int e = rank; e < h.z; e += size) {
          const int src = h.x + map_offset(L0[l].ext, L0[l].sstride, h.w & 0xff, h.w < 0, e);
          if (CPLX) {
            const float2 v = reinterpret_cast<const float2*>(in)[src];
            ar[h.y + e] = v.x;
            ar[h.y + h.z + e] = v.y;
            mx = max(mx, __float_as_int(fmaxf(fabsf(v.x), fabsf(v.y))));
          } else {
            const float v = in[src];
            ar[h.y + e] = v;
            mx = max(mx, __float_as_int(fabsf(v)));
          }
        }
        if (!MAXPLUS && scaling) {
          const int e = team_exp(mx, turn);
          if (WARP) __syncwarp();
          scale_in_place(h.y, h.z, e);
          turn ^= 1;
        }
      }
      if (!WARP && scaling) {
        // the two slots back as the steps expect them
        T::sync();
        if (rank < 2) s_exp[rank] = -127;
      }
      T::sync();
    }
    for (int s = 0; s < net.n_steps; ++s) {
      // (a record read from L2 by every step cost it more than its arithmetic)
      const BStep* S = WARP ? S0 + s : reinterpret_cast<const BStep*>(s_step[s & 1]);
      const int4 h0 = reinterpret_cast<const int4*>(S)[0], h1 = reinterpret_cast<const int4*>(S)[1];
      int4 next;
      const bool fetch = !WARP && rank < kRec && s + 1 < net.n_steps;
      if (fetch) next = __ldg(reinterpret_cast<const int4*>(S0 + s + 1) + rank);
      const int m = h0.w, n = h1.x, k = h1.y, mn = m * n;
      const int nr = (h1.z >> 27) & 15, nc = h1.w >> 27;
      const bool pow2 = h1.z < 0;
      float sa = 1.f, sb = 1.f;
      if (!MAXPLUS && scaling && defer) {
        auto scale_of = [&](int id) {
          if (id == kBLeafId) return 1.f;
          const int e = WARP ? int(w_exp[id]) - 127 : s_exp[id];
          return e < -126 ? 1.f : bpow2_neg(e);  // an all-zero tensor is left as is
        };
        sa = scale_of(h1.z & kBLeafId);
        sb = scale_of(h1.w & kBLeafId);
      }
      int mx = 0;
      // (k deep enough for the panels to pay, and no more than half of a tile's rows empty)
      const bool panels = TILES && !WARP && !CPLX && ar != s_arena && smem_arena >= panel_floats(blockDim.x) &&
                          (k & 3) == 0 && k >= 16 && max(m, n) >= 16 && min(m, n) >= 8 && mn * (k >> 4) >= 16 * size;
      if (panels) {
        if constexpr (TILES && !WARP && !CPLX) {
          const int* tab = nullptr;
          if (m + n <= tab_ints) {
            for (int x = rank; x < m + n; x += size) s_tab[x] = step_offset(S, nr, nc, pow2, m, x);
            tab = s_tab;  // (complete at the panels' first barrier)
          }
          mx = run_panels<MAXPLUS>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, tab, s_arena);
        }
      } else if (rank - lane >= mn) {
        // no output for this warp
      } else if (TILES && m >= RM && n >= RN && mn >= 8 * size) {
        const int* tab = nullptr;
        if (m + n <= tab_ints) {
          for (int x = rank; x < m + n; x += size) s_tab[x] = step_offset(S, nr, nc, pow2, m, x);
          tab = s_tab;
          T::sync();
        }
        if constexpr (!TILES) {
        } else if ((k & 3) == 0 && !CPLX)
          mx = run_step<CPLX, MAXPLUS, WARP, RM, RN, CPLX ? 2 : 4>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa,
                                                                  sb, tab);
        else if ((k & 1) == 0)
          mx = run_step<CPLX, MAXPLUS, WARP, RM, RN, 2>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, tab);
        else
          mx = run_step<CPLX, MAXPLUS, WARP, RM, RN, 1>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, tab);
      } else if ((k & 3) == 0) {
        mx = run_step<CPLX, MAXPLUS, WARP, 1, 1, 4>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, nullptr);
      } else if ((k & 1) == 0) {
        mx = run_step<CPLX, MAXPLUS, WARP, 1, 1, 2>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, nullptr);
      } else {
        mx = run_step<CPLX, MAXPLUS, WARP, 1, 1, 1>(ar, S, m, n, k, nr, nc, pow2, h0.x, h0.y, h0.z, sa, sb, nullptr);
      }
      if (fetch) s_step[(s + 1) & 1][rank] = next;
      if (!MAXPLUS && scaling) {
        __syncwarp();
        if (defer) {
          mx = __reduce_max_sync(0xffffffffu, mx);
          if (lane == 0) {
            if (WARP) w_exp[s] = static_cast<uint8_t>(mx >> 23);
            else if (mx) atomicMax(&s_exp[s], (mx >> 23) - 127);
          }
        } else {
          const int e = team_exp(mx, s & 1);
          if (WARP) __syncwarp();
          scale_in_place(h0.z, mn, e);
          continue;
        }
      }
      T::sync();
    }
    float sr = 1.f;
    if (!MAXPLUS && scaling) {
      if (defer) {
        for (int i = rank; i < net.n_steps; i += size) {
          const int e = WARP ? int(w_exp[i]) - 127 : s_exp[i];
          lsum += e < -126 ? 0 : e;
        }
        if (net.n_steps > 0) {
          const int e = WARP ? int(w_exp[net.n_steps - 1]) - 127 : s_exp[net.n_steps - 1];
          if (e >= -126) sr = bpow2_neg(e);
        }
      }
      for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
      if (!WARP) {
        if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&s_log), static_cast<unsigned long long>(lsum));
        __syncthreads();
        lsum = s_log;
      }
    }
    if (rank == 0) {
      // scalar results (closed networks): value and log2 scale
      values[2 * (int64_t)net.index] = ar[net.root] * sr;
      values[2 * (int64_t)net.index + 1] = CPLX ? ar[net.root + net.root_size] * sr : 0.0;
      logs[net.index] = double(lsum) * 0.69314718055994530942;
    }
    T::sync();
  }
}

}  // namespace
}  // namespace tn

using namespace tn;

struct tn_batch_s {
  int32_t n_nets = 0;
  bool cplx = false, scaling = false, maxplus = false;
  std::vector<BNet> nets;
  std::vector<BLeaf> leaves;
  std::vector<BStep> steps;
  std::vector<int64_t> leaf_offset;  // packed input offset of every leaf (+ total)
  int64_t arena_floats = 0;
  char* dev = nullptr;               // tables + arena + queue
  BNet* d_nets = nullptr;
  BLeaf* d_leaves = nullptr;
  BStep* d_steps = nullptr;
  float* d_arena = nullptr;
  int32_t* d_queue = nullptr;
  int threads = 128, ctas_per_sm = 4, num_sms = 148;
  int nets_per_cta = 1;              // > 1: one warp per network, this many warps per CTA
  int32_t smem_arena = 0;            // shared-memory arena per network slot (floats; 0: none)
  int64_t max_arena_floats = 0;      // largest network arena
  int32_t tab_ints = 0;              // offset-table ints per network slot
  double flops = 0;
  // graph cache
  cudaGraphExec_t gexec = nullptr;
  const void* g_in = nullptr;
  void* g_vals = nullptr;
  void* g_logs = nullptr;
  cudaStream_t g_stream = nullptr;
};

namespace tn {

using BatchKernel = void (*)(const BNet*, const BLeaf*, const BStep*, int32_t, const float*, float*, int32_t*, int32_t,
                             double*, double*, int32_t, int32_t);
template <bool CPLX, bool MAXPLUS, bool WARP>
BatchKernel batch_form(bool tiles) {
  return tiles ? batch_kernel<CPLX, MAXPLUS, WARP, true> : batch_kernel<CPLX, MAXPLUS, WARP, false>;
}

cudaError_t launch_batch_kernel(const BNet* nets, const BLeaf* leaves, const BStep* steps, int32_t n_nets,
                                const void* packed, float* arena, int32_t* queue, bool cplx, bool scaling,
                                bool maxplus, int threads, int grid, double* values, double* logs,
                                cudaStream_t st, bool warp, int32_t smem_arena, int32_t tab_ints) {
  cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  const float* in = static_cast<const float*>(packed);
  const int sc = scaling ? 1 : 0;
  // dynamic shared memory: an arena and an offset table per CTA, or per warp in the warp form
  smem_arena &= ~63;  // arenas are multiples of 64 floats
  const int smem = (smem_arena + tab_ints) * 4 * (warp ? threads / 32 : 1);
  const bool tiles = threads <= kTileThreads;
  auto kernel = warp ? (cplx ? batch_form<true, false, true>(tiles)
                             : maxplus ? batch_form<false, true, true>(tiles) : batch_form<false, false, true>(tiles))
                     : (cplx ? batch_form<true, false, false>(tiles)
                             : maxplus ? batch_form<false, true, false>(tiles) : batch_form<false, false, false>(tiles));
  // (an allowance belongs to the current device, so each launch that needs one sets it;
  // always the largest, so launches of several threads do not meet in it)
  if (smem + kBatchStaticSmem > kDefaultSmem)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kMaxSmemPerCta) - kBatchStaticSmem);
  if (e != cudaSuccess) return e;
  kernel<<<grid, threads, smem, st>>>(nets, leaves, steps, n_nets, in, arena, queue, maxplus ? 0 : sc, values, logs,
                                      smem_arena, tab_ints);
  return cudaGetLastError();
}

// Replace the extents of a digit map by the digits' places where all are powers of two.
static bool digit_places(int32_t* ext, int n) {
  int sh = 0;
  for (int d = 0; d < n; ++d)
    if (ext[d] < 1 || (ext[d] & (ext[d] - 1)) != 0 || ext[d] >= 1 << 23) return false;
  for (int d = n - 1; d >= 0; --d) {
    const int32_t mask = ext[d] - 1;
    ext[d] = sh | mask << 8;
    sh += __builtin_popcount(static_cast<unsigned>(mask));
  }
  return true;
}

bool batch_template(const Plan& P, BatchTemplate& T, std::string& err) {
  if (P.n_slices != 1) {
    err = "sliced networks are not batched";
    return false;
  }
  if (!P.open_modes.empty()) {
    err = "open labels (closed networks only)";
    return false;
  }
  if (P.arena_bytes / 4 > (int64_t(1) << 30)) {
    err = "network too large for the batched kernel";
    return false;
  }
  auto foff = [&](int32_t t) { return static_cast<int32_t>(P.tensors[t].offset / 4); };
  T = BatchTemplate{};
  const int32_t root = P.n_leaves + (int32_t)P.steps.size() - 1;
  T.root = foff(root);
  T.root_size = (int32_t)P.tensors[root].size;
  for (int32_t t = 0; t < P.n_leaves; ++t) {
    const TensorRec& R = P.tensors[t];
    const LeafDesc& d = P.leafdesc[t];
    if (d.rank > kBMaxRank || R.split) {
      err = d.rank > kBMaxRank ? "leaf rank too large" : "split-BF16 operands (tensor-core steps)";
      return false;
    }
    BLeaf L{};
    L.src = static_cast<int32_t>(T.input_elems);
    L.dst = foff(t);
    L.size = (int32_t)R.size;
    for (int r = 0; r < d.rank; ++r) {
      L.ext[r] = (int32_t)d.ext[r];
      L.sstride[r] = (int32_t)d.sstride[r];
    }
    L.rank = d.rank | (digit_places(L.ext, d.rank) ? kBPow2 : 0);
    int64_t full = 1;
    for (int32_t x : R.decl) full *= P.extent[x];
    T.input_elems += full;
    T.leaves.push_back(L);
  }
  for (const StepRec& st : P.steps) {
    if (st.rows.n > kBMaxDims || st.cols.n > kBMaxDims || st.cls == TN_CLASS_TC) {
      err = st.cls == TN_CLASS_TC ? "tensor-core steps" : "output interleaving too fine";
      return false;
    }
    BStep S{};
    S.a = foff(st.a);
    S.b = foff(st.b);
    S.c = foff(st.out);
    S.m = (int32_t)st.m;
    S.n = (int32_t)st.n;
    S.k = (int32_t)st.k;
    for (int d = 0; d < st.rows.n; ++d) {
      S.rext[d] = (int32_t)st.rows.ext[d];
      S.rstr[d] = (int32_t)st.rows.stride[d];
    }
    for (int d = 0; d < st.cols.n; ++d) {
      S.cext[d] = (int32_t)st.cols.ext[d];
      S.cstr[d] = (int32_t)st.cols.stride[d];
    }
    int32_t rext[kBMaxDims], cext[kBMaxDims];
    std::copy(S.rext, S.rext + kBMaxDims, rext);
    std::copy(S.cext, S.cext + kBMaxDims, cext);
    const bool pow2 = digit_places(rext, st.rows.n) && digit_places(cext, st.cols.n);
    if (pow2) {
      std::copy(rext, rext + kBMaxDims, S.rext);
      std::copy(cext, cext + kBMaxDims, S.cext);
    }
    S.pa = (st.a < P.n_leaves ? kBLeafId : st.a - P.n_leaves) | st.rows.n << 27 | (pow2 ? kBPow2 : 0);
    S.pb = (st.b < P.n_leaves ? kBLeafId : st.b - P.n_leaves) | st.cols.n << 27;
    T.steps.push_back(S);
    T.max_tab = std::max<int32_t>(T.max_tab, static_cast<int32_t>(st.m + st.n));
    T.flops += (P.is_complex ? 8.0 : 2.0) * double(st.m) * double(st.n) * double(st.k);
  }
  T.arena_floats = (P.arena_bytes + 255) / 256 * 64;  // keep every arena 256-byte aligned
  return true;
}

}  // namespace tn

namespace {
tn_status launch_batch(tn_batch_s* B, const void* packed, double* values, double* logs, cudaStream_t st) {
  const bool warp = B->nets_per_cta > 1;
  const int64_t ctas_needed = warp ? (B->n_nets + B->nets_per_cta - 1) / B->nets_per_cta : B->n_nets;
  const int grid = std::min<int64_t>(ctas_needed, (int64_t)B->num_sms * B->ctas_per_sm);
  const int threads = warp ? 32 * B->nets_per_cta : B->threads;
  cudaError_t e = launch_batch_kernel(B->d_nets, B->d_leaves, B->d_steps, B->n_nets, packed, B->d_arena, B->d_queue,
                                      B->cplx, B->scaling, B->maxplus, threads, grid, values, logs, st, warp,
                                      B->smem_arena, B->tab_ints);
  if (e != cudaSuccess) {
    set_error(std::string("batch kernel launch: ") + cudaGetErrorString(e));
    return TN_ERR_CUDA;
  }
  return TN_OK;
}
}  // namespace

extern "C" {

tn_status tn_batch_plan(int32_t n_nets, const tn_network* nets, const tn_path* paths, tn_dtype_policy policy,
                        tn_batch_t* out) {
  if (n_nets <= 0 || !nets || !paths || !out) {
    set_error("tn_batch_plan: bad arguments");
    return TN_ERR_INVALID;
  }
  if (policy.prec != TN_C64_FP32_SIMT && policy.prec != TN_R32_FP32_SIMT) {
    set_error("tn_batch_plan: batched small networks run the FP32 form (C64_FP32_SIMT or R32_FP32_SIMT)");
    return TN_ERR_UNSUPPORTED;
  }
  auto B = std::make_unique<tn_batch_s>();
  B->n_nets = n_nets;
  B->cplx = policy.prec == TN_C64_FP32_SIMT;
  B->scaling = policy.exp_scaling != 0;
  B->maxplus = policy.semiring == TN_SEMIRING_MAXPLUS;
  if (B->maxplus && (B->cplx || B->scaling)) {
    set_error("tn_batch_plan: the max-plus semiring runs R32 without exponent scaling");
    return TN_ERR_UNSUPPORTED;
  }
  int64_t in_off = 0;
  std::unordered_map<std::string, std::pair<size_t, size_t>> tables;
  std::vector<double> cost;
  tn_dtype_policy hp = policy;
  hp.flags |= TN_PLAN_HOST_ONLY;
  hp.max_slice_batch = 1;
  for (int32_t w = 0; w < n_nets; ++w) {
    Plan P;
    std::string err;
    tn_status s = build_plan(&nets[w], &paths[w], nullptr, 0, hp, P, err);
    if (s != TN_OK) {
      set_error("network " + std::to_string(w) + ": " + err);
      return s;
    }
    if (!P.open_modes.empty()) {
      set_error("tn_batch_plan: network " + std::to_string(w) + " has open labels (closed networks only)");
      return TN_ERR_UNSUPPORTED;
    }
    drop_gate_runs(P);  // the batched kernel runs the steps one after another
    assign_workspace(P, 1, false);
    if (!P.workspace_ok) {
      set_error("tn_batch_plan: workspace self-check failed");
      return TN_ERR_INVALID;
    }
    BatchTemplate T;
    std::string why;
    if (!batch_template(P, T, why)) {
      set_error("tn_batch_plan: network " + std::to_string(w) + ": " + why);
      return TN_ERR_UNSUPPORTED;
    }
    BNet bn{};
    bn.arena = B->arena_floats;
    bn.index = w;
    // networks of one shape and path share their tables (which then stay in L2)
    std::string key(reinterpret_cast<const char*>(T.leaves.data()), T.leaves.size() * sizeof(BLeaf));
    key.append(reinterpret_cast<const char*>(T.steps.data()), T.steps.size() * sizeof(BStep));
    const auto [at, fresh] = tables.emplace(std::move(key), std::make_pair(B->leaves.size(), B->steps.size()));
    bn.leaf0 = (int32_t)at->second.first;
    bn.n_leaves = (int32_t)T.leaves.size();
    bn.step0 = (int32_t)at->second.second;
    bn.n_steps = (int32_t)T.steps.size();
    bn.root = T.root;
    bn.root_size = T.root_size;
    bn.arena_floats = static_cast<int32_t>(T.arena_floats);
    bn.in = in_off;
    for (const BLeaf& L : T.leaves) B->leaf_offset.push_back(in_off + L.src);
    if (fresh) {
      B->leaves.insert(B->leaves.end(), T.leaves.begin(), T.leaves.end());
      B->steps.insert(B->steps.end(), T.steps.begin(), T.steps.end());
    }
    in_off += T.input_elems;
    cost.push_back(T.flops);
    B->flops += T.flops;
    B->arena_floats += T.arena_floats;
    B->max_arena_floats = std::max(B->max_arena_floats, T.arena_floats);
    B->tab_ints = std::max(B->tab_ints, std::min(T.max_tab, kMaxTabInts));
    B->nets.push_back(bn);
  }
  B->leaf_offset.push_back(in_off);
  // the costliest networks first
  std::vector<int32_t> order(n_nets);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return cost[x] > cost[y]; });
  std::vector<BNet> queued;
  for (int32_t w : order) queued.push_back(B->nets[w]);
  B->nets.swap(queued);
  if ((policy.flags & TN_PLAN_HOST_ONLY) == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&B->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      set_error("tn_batch_plan: no CUDA device");
      return TN_ERR_CUDA;
    }
    auto al = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t b_nets = al(sizeof(BNet) * B->nets.size()), b_leaves = al(sizeof(BLeaf) * B->leaves.size());
    const size_t b_steps = al(sizeof(BStep) * std::max<size_t>(1, B->steps.size()));
    const size_t b_arena = al(sizeof(float) * B->arena_floats);
    const size_t total = b_nets + b_leaves + b_steps + b_arena + 256;
    void* mem = nullptr;
    if (cudaMalloc(&mem, total) != cudaSuccess) {
      cudaGetLastError();
      set_error("tn_batch_plan: cudaMalloc failed");
      return TN_ERR_OOM;
    }
    B->dev = static_cast<char*>(mem);
    B->d_nets = reinterpret_cast<BNet*>(B->dev);
    B->d_leaves = reinterpret_cast<BLeaf*>(B->dev + b_nets);
    B->d_steps = reinterpret_cast<BStep*>(B->dev + b_nets + b_leaves);
    B->d_arena = reinterpret_cast<float*>(B->dev + b_nets + b_leaves + b_steps);
    B->d_queue = reinterpret_cast<int32_t*>(B->dev + b_nets + b_leaves + b_steps + b_arena);
    if (cudaMemcpy(B->d_nets, B->nets.data(), sizeof(BNet) * B->nets.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(B->d_leaves, B->leaves.data(), sizeof(BLeaf) * B->leaves.size(), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        (!B->steps.empty() && cudaMemcpy(B->d_steps, B->steps.data(), sizeof(BStep) * B->steps.size(),
                                         cudaMemcpyHostToDevice) != cudaSuccess) ||
        uploads_done() != cudaSuccess) {
      cudaFree(mem);
      set_error("tn_batch_plan: table upload failed");
      return TN_ERR_CUDA;
    }
  }
  *out = B.release();
  return TN_OK;
}

tn_status tn_batch_info(tn_batch_t b, int64_t* leaf_offsets, double* flops, int32_t* threads,
                        int32_t* ctas_per_sm, int32_t* nets_per_cta, int32_t* smem_arena) {
  if (!b) {
    set_error("null batch");
    return TN_ERR_INVALID;
  }
  if (leaf_offsets) std::copy(b->leaf_offset.begin(), b->leaf_offset.end(), leaf_offsets);
  if (flops) *flops = b->flops;
  if (threads) *threads = b->threads;
  if (ctas_per_sm) *ctas_per_sm = b->ctas_per_sm;
  if (nets_per_cta) *nets_per_cta = b->nets_per_cta;
  if (smem_arena) *smem_arena = b->smem_arena;
  return TN_OK;
}

tn_status tn_batch_contract(tn_batch_t b, const void* packed_inputs, double* values, double* log_scales,
                            void* stream) {
  if (!b || !b->dev || !packed_inputs || !values || !log_scales) {
    set_error("tn_batch_contract: bad arguments (or a host-only batch)");
    return TN_ERR_INVALID;
  }
  return launch_batch(b, packed_inputs, values, log_scales, reinterpret_cast<cudaStream_t>(stream));
}

tn_status tn_batch_contract_graph(tn_batch_t b, const void* packed_inputs, double* values, double* log_scales,
                                  void* stream) {
  if (!b || !b->dev || !packed_inputs || !values || !log_scales) {
    set_error("tn_batch_contract_graph: bad arguments (or a host-only batch)");
    return TN_ERR_INVALID;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!b->gexec || b->g_in != packed_inputs || b->g_vals != values || b->g_logs != log_scales ||
      b->g_stream != st) {
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
    cudaStream_t cap = nullptr;
    if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) {
      set_error("graph capture stream");
      return TN_ERR_CUDA;
    }
    cudaGraph_t g = nullptr;
    tn_status s = TN_OK;
    if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) s = TN_ERR_CUDA;
    if (s == TN_OK) s = launch_batch(b, packed_inputs, values, log_scales, cap);
    cudaError_t e = cudaStreamEndCapture(cap, &g);
    if (s == TN_OK && e == cudaSuccess) e = cudaGraphInstantiate(&b->gexec, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    if (s != TN_OK || e != cudaSuccess) {
      cudaGetLastError();
      set_error(std::string("batch graph capture failed: ") + cudaGetErrorString(e));
      return TN_ERR_CUDA;
    }
    b->g_in = packed_inputs;
    b->g_vals = values;
    b->g_logs = log_scales;
    b->g_stream = st;
  }
  cudaError_t e = cudaGraphLaunch(b->gexec, st);
  if (e != cudaSuccess) {
    set_error(std::string("graph launch: ") + cudaGetErrorString(e));
    return TN_ERR_CUDA;
  }
  return TN_OK;
}

tn_status tn_batch_autotune(tn_batch_t b, const void* packed_inputs, double* values, double* log_scales,
                            void* stream) {
  if (!b || !b->dev) {
    set_error("tn_batch_autotune: bad batch");
    return TN_ERR_INVALID;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int cand_threads[] = {32, 64, 128, 256};
  const int cand_ctas[] = {2, 4, 8, 16};
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  float best = 1e30f;
  int bt = b->threads, bc = b->ctas_per_sm, bg = b->nets_per_cta;
  int32_t bs = b->smem_arena;
  // (threads per network, networks per CTA): a CTA per network at 32-256 threads, or a warp
  // per network with 4 or 8 warps per CTA
  struct Shape { int t, g; };
  std::vector<Shape> shapes;
  for (int t : cand_threads) shapes.push_back({t, 1});
  shapes.push_back({32, 4});
  shapes.push_back({32, 8});
  // shared-memory arena per network slot: none, or the largest that c CTAs of g slots fit
  // (networks above it keep their global arenas), no larger than the largest arena
  for (const Shape& sh : shapes)
    for (int c : cand_ctas)
      for (int sm = 0; sm < 2; ++sm) {
      const int cta_threads = sh.g > 1 ? 32 * sh.g : sh.t;
      if (cta_threads * c > 2048) continue;
      int64_t cap = 0;
      const int64_t per_slot = std::min<int64_t>(kSmemPerSm / (4 * sh.g * c), kMaxSmemPerCta / (4 * sh.g));
      if (per_slot < b->tab_ints) continue;  // the offset tables alone do not fit this shape
      if (sm) {
        cap = std::min<int64_t>(per_slot - b->tab_ints, b->max_arena_floats) / 64 * 64;
        if (cap < 64) continue;
      }
      b->threads = sh.t;
      b->nets_per_cta = sh.g;
      b->ctas_per_sm = c;
      b->smem_arena = static_cast<int32_t>(cap);
      float ms_best = 1e30f;
      for (int rep = 0; rep < 3; ++rep) {
        cudaEventRecord(e0, st);
        tn_status s = launch_batch(b, packed_inputs, values, log_scales, st);
        cudaEventRecord(e1, st);
        if (s != TN_OK || cudaEventSynchronize(e1) != cudaSuccess) {
          cudaEventDestroy(e0);
          cudaEventDestroy(e1);
          set_error("tn_batch_autotune: a candidate failed");
          return TN_ERR_CUDA;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms_best = std::min(ms_best, ms);
      }
      if (ms_best < best) {
        best = ms_best;
        bt = sh.t;
        bg = sh.g;
        bc = c;
        bs = b->smem_arena;
      }
    }
  b->threads = bt;
  b->nets_per_cta = bg;
  b->ctas_per_sm = bc;
  b->smem_arena = bs;
  if (b->gexec) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return TN_OK;
}

tn_status tn_batch_set_shape(tn_batch_t b, int32_t threads, int32_t ctas_per_sm, int32_t nets_per_cta,
                             int32_t smem_arena) {
  const bool warp = nets_per_cta > 1;
  const int cta_threads = warp ? 32 * nets_per_cta : threads;
  if (!b || ctas_per_sm < 1 || nets_per_cta < 1 || (warp && threads != 32) || cta_threads < 32 ||
      cta_threads > 1024 || cta_threads % 32 != 0 || cta_threads * ctas_per_sm > 2048 ||
      smem_arena < 0 || int64_t(smem_arena + b->tab_ints) * 4 * nets_per_cta > kMaxSmemPerCta ||
      int64_t(smem_arena + b->tab_ints) * 4 * nets_per_cta * ctas_per_sm > kSmemPerSm) {
    set_error("tn_batch_set_shape: bad launch shape");
    return TN_ERR_INVALID;
  }
  b->threads = threads;
  b->ctas_per_sm = ctas_per_sm;
  b->nets_per_cta = nets_per_cta;
  b->smem_arena = smem_arena;
  if (b->gexec) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
  }
  return TN_OK;
}

tn_status tn_batch_destroy(tn_batch_t b) {
  if (!b) return TN_OK;
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->dev) cudaFree(b->dev);
  delete b;
  return TN_OK;
}

}  // extern "C"
