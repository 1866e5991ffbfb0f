// Gate runs (sm_103a): consecutive big x small steps on one tensor, in one pass over it.
//
// A step whose small operand is square (k = n = 2, 4, 8, 16: gates on a state) only replaces bits
// of the big tensor's index: the k bits give way to as many n bits, every other bit moves to its
// place in the output. So a run of them is one fixed permutation of index bits ("wires") with a
// small matrix applied to some wires on the way. A tile holds all values of the wires that the
// run's gates act on and of the lowest few bits of the run's input and of its output, so that
// both are moved in whole sectors; a CTA loads it into shared memory, applies the gates in place
// and stores it. A leaf is read where the caller has it, instead of being staged in the planned
// order first; a run that ends the path writes the caller's FP64 output itself.
//
// Every output is summed over k in order with the FMAs of contract_stream_kernel: the same bits as
// a pass per step.
//
// What bounds it: the instructions of a tile's way through shared memory, no longer HBM. Four
// two-qubit gates on 26 qubits with the leaf's staging and the output's widening moved 6.5 GB in 1.21
// ms; the run moves 1.6 GB in 0.43 ms, with 5 instructions of 8 issue slots used: per element 64
// FMAs, 20 others for the gates, 35 for load, FP64 and store. A tile of 2^12 complex elements
// takes 32 KB, six CTAs of 128 threads an SM: some load or store while others compute, and a thread's
// share of 32 elements pays for its setup (256 threads: 0.54 -> 0.48 ms). Sixteen loads in flight
// and rounds in Gray code order: 0.48 -> 0.43. Measured and slower: tiles dealt to resident CTAs
// (their phases align: 0.84), two elements to a packed FMA (0.52-0.98: registers).
// Shared-memory addresses are linear over the wires (XOR): a tile wire above the bank bits also
// flips one of them, chosen so that the lanes of the load, of every gate and of the store meet
// different banks.
#include <cstdint>

#include <cuda_runtime.h>

#include "kernels.h"
#include "widen.cuh"

namespace tn {
namespace {

constexpr int kThreads = 128;
constexpr int kThreadBits = 7;
constexpr int kIters = 1 << (kGateTileBits - kThreadBits);

// An element of the tile at a byte address (real: y is not stored).
template <bool CPLX>
__device__ __forceinline__ float2 get(const char* tile, int at) {
  if constexpr (CPLX) return *reinterpret_cast<const float2*>(tile + at);
  else return make_float2(*reinterpret_cast<const float*>(tile + at), 0.f);
}
template <bool CPLX>
__device__ __forceinline__ void put(char* tile, int at, float2 v) {
  if constexpr (CPLX) *reinterpret_cast<float2*>(tile + at) = v;
  else *reinterpret_cast<float*>(tile + at) = v.x;
}

template <bool CPLX, int KB>
__device__ __forceinline__ void gate_pass(char* tile, const GateStep& g, const float2* mat, int t) {
  constexpr int K = 1 << KB;
  const int groups = 1 << (t - KB), tid = threadIdx.x;
  if (tid >= groups) return;
  int base0 = 0;
#pragma unroll
  for (int b = 0; b < kThreadBits; ++b) base0 ^= (tid >> b) & 1 ? g.rest[b] : 0;
  int ko[K];
#pragma unroll
  for (int q = 0; q < K; ++q) {
    ko[q] = 0;
#pragma unroll
    for (int b = 0; b < KB; ++b) ko[q] ^= (q >> b) & 1 ? g.wire[b] : 0;
  }
  float2 m[KB <= 2 ? K * K : 1];
  if constexpr (KB <= 2) {
#pragma unroll
    for (int i = 0; i < K * K; ++i) m[i] = mat[i];
  }
  const int rounds = groups > kThreads ? groups / kThreads : 1;
  int base = base0;
  // the rounds in Gray code order: one bit of the group's index changes from each to the next
  for (int i = 0; i < rounds; ++i) {
    if (i > 0) base ^= g.rest[kThreadBits + __ffs(i) - 1];
    float2 x[K];
#pragma unroll
    for (int q = 0; q < K; ++q) x[q] = get<CPLX>(tile, base ^ ko[q]);
#pragma unroll
    for (int j = 0; j < K; ++j) {
      float2 c = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const float2 y = KB <= 2 ? m[KB <= 2 ? j * K + q : 0] : mat[j * K + q];
        c.x = fmaf(x[q].x, y.x, c.x);
        if (CPLX) {
          c.x = fmaf(-x[q].y, y.y, c.x);
          c.y = fmaf(x[q].x, y.y, c.y);
          c.y = fmaf(x[q].y, y.x, c.y);
        }
      }
      put<CPLX>(tile, base ^ ko[j], c);
    }
  }
}

// What a round of the load or of the store adds to a thread's offset (bytes) and address.
struct __align__(16) Round {
  int64_t off;
  int at;
};

template <bool CPLX>
__global__ void __launch_bounds__(kThreads, 6) gate_run_kernel(const __grid_constant__ GateArgs a) {
  extern __shared__ __align__(16) char tile[];
  __shared__ Round s_in[kIters], s_out[kIters];
  __shared__ int64_t s_tile[2];
  const int t = a.t, tid = threadIdx.x;
  const int in_bytes = CPLX && a.interleaved ? 8 : 4, out_bytes = (a.widen ? 8 : 4) * (CPLX && a.widen ? 2 : 1);
  float2* mats = reinterpret_cast<float2*>(tile + ((CPLX ? 8 : 4) << t));
  for (int g = 0, o = 0; g < a.n_gates; ++g) {
    const int kk = 1 << (2 * a.gate[g].bits);
    for (int i = tid; i < kk; i += kThreads)
      mats[o + i] = make_float2(__ldg(a.gate[g].b + i), CPLX ? __ldg(a.gate[g].b + a.gate[g].b_plane + i) : 0.f);
    o += kk;
  }
  if (tid < kIters) {
    Round ri{0, 0}, ro{0, 0};
#pragma unroll
    for (int b = kThreadBits; b < kGateTileBits; ++b)
      if ((tid >> (b - kThreadBits)) & 1) {
        ri.off += a.in_off[b] * in_bytes;
        ro.off += a.out_off[b] * out_bytes;
        ri.at ^= a.in_addr[b];
        ro.at ^= a.out_addr[b];
      }
    s_in[tid] = ri;
    s_out[tid] = ro;
  }
  if (tid < 32) {  // the tile's offsets
    int64_t x = 0, y = 0;
    if (tid < a.outer && (blockIdx.x >> tid) & 1) {
      x = a.in_outer[tid];
      y = a.out_outer[tid];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (tid == 0) {
      s_tile[0] = x;
      s_tile[1] = y;
    }
  }
  int64_t in = 0, out = 0;
  int ia = 0, oa = 0;
#pragma unroll
  for (int b = 0; b < kThreadBits; ++b)
    if ((tid >> b) & 1) {
      in += a.in_off[b];
      out += a.out_off[b];
      ia ^= a.in_addr[b];
      oa ^= a.out_addr[b];
    }
  __syncthreads();
  const char* src = reinterpret_cast<const char*>(a.in) + (in + s_tile[0]) * in_bytes;
  char* dst = static_cast<char*>(a.out) + (out + s_tile[1]) * out_bytes;
  const int iters = 1 << (t - kThreadBits);
  auto fetch = [&](int i) {
    const char* p = src + s_in[i].off;
    if (!CPLX) return make_float2(__ldg(reinterpret_cast<const float*>(p)), 0.f);
    if (a.interleaved) return __ldg(reinterpret_cast<const float2*>(p));
    return make_float2(__ldg(reinterpret_cast<const float*>(p)), __ldg(reinterpret_cast<const float*>(p) + a.in_plane));
  };
  constexpr int U = 16;  // elements in flight per thread
  if (iters >= U) {
    for (int i0 = 0; i0 < iters; i0 += U) {
      float2 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = fetch(i0 + u);
#pragma unroll
      for (int u = 0; u < U; ++u) put<CPLX>(tile, ia ^ s_in[i0 + u].at, v[u]);
    }
  } else {
#pragma unroll 2
    for (int i = 0; i < iters; ++i) put<CPLX>(tile, ia ^ s_in[i].at, fetch(i));
  }
  __syncthreads();
  for (int g = 0, o = 0; g < a.n_gates; ++g) {
    const GateStep& s = a.gate[g];
    if (s.bits == 1) gate_pass<CPLX, 1>(tile, s, mats + o, t);
    else if (s.bits == 2) gate_pass<CPLX, 2>(tile, s, mats + o, t);
    else if (s.bits == 3) gate_pass<CPLX, 3>(tile, s, mats + o, t);
    else gate_pass<CPLX, 4>(tile, s, mats + o, t);
    o += 1 << (2 * s.bits);
    __syncthreads();
  }
#pragma unroll 4
  for (int i = 0; i < iters; ++i) {
    const Round r = s_out[i];
    const float2 v = get<CPLX>(tile, oa ^ r.at);
    char* p = dst + r.off;
    if (!a.widen) {
      *reinterpret_cast<float*>(p) = v.x;
      if (CPLX) reinterpret_cast<float*>(p)[a.out_plane] = v.y;
    } else if (CPLX) {
      *reinterpret_cast<double2*>(p) = f64_of_f32(v);
    } else {
      *reinterpret_cast<double*>(p) = f64_of_f32(v.x);
    }
  }
  if (a.log_scale && blockIdx.x == 0 && tid == 0) *a.log_scale = 0.0;
}

}  // namespace

template <bool CPLX>
static cudaError_t launch(const GateArgs& a, cudaStream_t st) {
  constexpr int elem = CPLX ? 8 : 4;
  constexpr int fixed = 2 * kIters * int(sizeof(Round)) + 2 * int(sizeof(int64_t));  // the kernel's own arrays
  int bytes = elem << a.t;
  for (int g = 0; g < a.n_gates; ++g) bytes += int(sizeof(float2)) << (2 * a.gate[g].bits);
  // (an allowance belongs to the current device, so each launch that needs one sets it;
  // always the largest, so launches of several threads do not meet in it)
  if (bytes + fixed > kDefaultSmem) {
    const cudaError_t e = cudaFuncSetAttribute(gate_run_kernel<CPLX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (elem << kGateTileBits) + kGateMaxRun * 256 * int(sizeof(float2)));
    if (e != cudaSuccess) return e;
  }
  gate_run_kernel<CPLX><<<1u << a.outer, kThreads, bytes, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_gate_run(const GateArgs& a, bool cplx, cudaStream_t st) {
  return cplx ? launch<true>(a, st) : launch<false>(a, st);
}

}  // namespace tn
