// Step chains (sm_103a): a run of tiny pairwise steps in one launch of one thread-block cluster.
//
// What bounds it: latency. A step is a few hundred outputs of a few terms, so what counts is how
// many times the launch waits for one step's results to be visible to the next. The steps of a
// run are a forest, a few levels deep (the 4x4 kicked Ising's 702 steps: 9 levels), so the plan
// sorts them by level and cuts each level's outputs into tasks of a few outputs per lane, one per
// warp of the cluster; the cluster barrier between levels orders a level's stores and scale
// records before the next level's loads. Each output is one lane's, summed over k in order with
// the FMAs of contract_simt_kernel: the same bits as a launch per step.
// A warp's task, its step's descriptor and the level bounds are fetched one, two and three levels
// ahead, so a level costs its operands' loads, its stores and the barrier.
// A run of one level needs no barrier and takes as many CTAs as give each lane one output.
// Measured (GB300): the 702 steps 1036 us in one CTA step after step (1.5 us each) -> 40 us; 27
// steps of one level (110592 outputs) 284 -> 33 us on one cluster -> ~8 us on 216 CTAs; the
// 12-qubit amplitude's 57 steps (12 levels) 84 -> 26 -> 19.5 us, the last by taking branches out
// of a lane's chain: a level was ~2000 clocks for 2 terms and 300 more for every 4, nearly all of
// it branches and dependent loads of the dims, and is ~1500 and 60 now. (Software-pipelined or
// 16-term groups were slower: spills, and instructions that one CTA runs once cost their fetch.)
#include <atomic>
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "kernels.h"
#include "scale.cuh"
#include "split_bf16.cuh"
#include "pdl.cuh"

namespace tn {
namespace {

constexpr int kChainThreads = 512;
constexpr int kChainWarps = kChainThreads / 32;
constexpr int kStepWords = sizeof(ChainStep) / 4;
constexpr int kLaneWords = (kStepWords + 31) / 32;
static_assert(offsetof(ChainStep, ext) % 16 == 0 && offsetof(ChainStep, stride) % 16 == 0 && kMaxDims % 4 == 0,
              "four places per 16-byte load");
static_assert(sizeof(ChainStep) % 16 == 0, "ChainStep copied as 32-bit words, table entries 16-byte aligned");

// every CTA of the cluster (the grid): the stores and atomics before it are visible to the loads after it
__device__ __forceinline__ void level_barrier() {
  __syncwarp();
  if (gridDim.x == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// Offset of index i under the nd merged dims of one side of a step (last fastest). Extents that are
// all powers of two come as places (shift << 24 | mask), whose digits do not wait for one
// another; a place beyond nd is 0, so four are taken without a branch. Else as 0xff << 24 | extent.
__device__ __forceinline__ int dims_offset(const uint32_t* ext, const int32_t* stride, int nd, uint32_t i) {
  const uint4 e = *reinterpret_cast<const uint4*>(ext);
  int off = 0;
  if (e.x >> 24 != 0xffu) {
    const int4 st = *reinterpret_cast<const int4*>(stride);
    off = static_cast<int>((i >> (e.x >> 24)) & e.x & 0xffffffu) * st.x +
          static_cast<int>((i >> (e.y >> 24)) & e.y & 0xffffffu) * st.y +
          static_cast<int>((i >> (e.z >> 24)) & e.z & 0xffffffu) * st.z +
          static_cast<int>((i >> (e.w >> 24)) & e.w & 0xffffffu) * st.w;
#pragma unroll 1
    for (int d = 4; d < nd; ++d) off += static_cast<int>((i >> (ext[d] >> 24)) & ext[d] & 0xffffffu) * stride[d];
  } else {
#pragma unroll 1
    for (int d = nd - 1; d >= 0; --d) {
      const uint32_t x = ext[d] & 0xffffffu, q = i / x;
      off += static_cast<int>(i - q * x) * stride[d];
      i = q;
    }
  }
  return off;
}

// Bring p's sector into L1 (no value is waited for).
__device__ __forceinline__ void touch(const float* p) {
  float x;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(p) : "memory");
}

template <bool CPLX, bool MAXPLUS>
__device__ __forceinline__ void add_term(float xr, float xi, float yr, float yi, float sa, float sb, float& accr,
                                         float& acci) {
  const float vr = xr * sa, wr = yr * sb;
  if (CPLX) {
    const float vi = xi * sa, wi = yi * sb;
    accr = fmaf(vr, wr, accr);
    accr = fmaf(-vi, wi, accr);
    acci = fmaf(vr, wi, acci);
    acci = fmaf(vi, wr, acci);
  } else if (MAXPLUS) {
    accr = fmaxf(accr, vr + wr);
  } else {
    accr = fmaf(vr, wr, accr);
  }
}

// One task: outputs first .. first + count - 1 of batch entry b of step S, a lane per output.
template <bool CPLX, bool MAXPLUS>
__device__ __forceinline__ void run_task(const ChainStep& S, const ChainTask& t, int lane) {
  const float kZero = MAXPLUS ? __int_as_float(0xff800000) : 0.f;
  constexpr int U = CPLX ? 4 : 8;  // terms whose loads are in flight together
  const int b = t.b;
  float sa = 1.f, sb = 1.f;
  ScaleRec *ra = nullptr, *rb = nullptr, *rc = nullptr;
  if (S.recs) {
    ra = S.recs + S.rec_a + (S.a_bstride ? b : 0);
    rb = S.recs + S.rec_b + (S.b_bstride ? b : 0);
    rc = S.recs + S.rec_c + (S.c_bstride ? b : 0);
    sa = pow2_neg(scale_exp(ra));
    sb = pow2_neg(scale_exp(rb));
  }
  const float* A = S.A + b * S.a_bstride;
  const float* B = S.B + b * S.b_bstride;
  float* C = S.C + b * S.c_bstride;
  const int k = S.k;
  // rows of a multiple of four terms start 16-byte aligned (tensors do at 256), of two at 8
  const int bits = k | S.a_plane | S.b_plane | S.a_bstride | S.b_bstride;
  const int vec = (bits & 3) == 0 ? 4 : k == 2 && (bits & 1) == 0 ? 2 : 1;
  int lmax = -127;
  for (int idx = t.first + lane; idx < t.first + t.count; idx += 32) {
    const int r = S.n_shift >= 0 ? idx >> S.n_shift : idx / S.n, c = idx - r * S.n;
    const float* ar = A + r * k;
    const float* br = B + c * k;
    float accr = kZero, acci = kZero;
    if (vec == 4) {
      // whole groups of four terms: no branches but the loop's (a lone warp waits for each). Deep
      // rows: every 32-byte sector is asked for before the first is waited for
#pragma unroll 1
      for (int k0 = 8; k0 < k; k0 += 8) {
        touch(ar + k0);
        touch(br + k0);
        if (CPLX) {
          touch(ar + S.a_plane + k0);
          touch(br + S.b_plane + k0);
        }
      }
#pragma unroll 1
      for (int k0 = 0; k0 < k; k0 += 4) {
        const float4 x = *reinterpret_cast<const float4*>(ar + k0), y = *reinterpret_cast<const float4*>(br + k0);
        float4 u{}, w{};
        if (CPLX) {
          u = *reinterpret_cast<const float4*>(ar + S.a_plane + k0);
          w = *reinterpret_cast<const float4*>(br + S.b_plane + k0);
        }
        add_term<CPLX, MAXPLUS>(x.x, u.x, y.x, w.x, sa, sb, accr, acci);
        add_term<CPLX, MAXPLUS>(x.y, u.y, y.y, w.y, sa, sb, accr, acci);
        add_term<CPLX, MAXPLUS>(x.z, u.z, y.z, w.z, sa, sb, accr, acci);
        add_term<CPLX, MAXPLUS>(x.w, u.w, y.w, w.w, sa, sb, accr, acci);
      }
    } else if (vec == 2) {
      const float2 x = *reinterpret_cast<const float2*>(ar), y = *reinterpret_cast<const float2*>(br);
      float2 u{}, w{};
      if (CPLX) {
        u = *reinterpret_cast<const float2*>(ar + S.a_plane);
        w = *reinterpret_cast<const float2*>(br + S.b_plane);
      }
      add_term<CPLX, MAXPLUS>(x.x, u.x, y.x, w.x, sa, sb, accr, acci);
      add_term<CPLX, MAXPLUS>(x.y, u.y, y.y, w.y, sa, sb, accr, acci);
    } else {
#pragma unroll 1
      for (int k0 = 0; k0 < k; k0 += U) {
        float xr[U], yr[U], xi[U], yi[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (k0 + u >= k) break;
          xr[u] = ar[k0 + u];
          yr[u] = br[k0 + u];
          if (CPLX) {
            xi[u] = ar[S.a_plane + k0 + u];
            yi[u] = br[S.b_plane + k0 + u];
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (k0 + u >= k) break;
          add_term<CPLX, MAXPLUS>(xr[u], xi[u], yr[u], yi[u], sa, sb, accr, acci);
        }
      }
    }
    const int off = dims_offset(S.ext, S.stride, S.nr, r) + dims_offset(S.ext + kMaxDims, S.stride + kMaxDims, S.nc, c);
    if (CPLX) store_cplx(C, S.c_plane, off, accr, acci, S.c_split);
    else C[off] = accr;
    if (S.recs) lmax = max(lmax, exp_of(CPLX ? fmaxf(fabsf(accr), fabsf(acci)) : fabsf(accr)));
  }
  if (S.recs) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lmax = max(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if (lane == 0) {
      atomicMax(&rc->emax, lmax);
      if (t.first == 0) rc->log2 = ra->log2 + rb->log2 + scale_exp(ra) + scale_exp(rb);
    }
  }
}

template <bool CPLX, bool MAXPLUS>
__global__ void __launch_bounds__(kChainThreads) contract_chain_kernel(const ChainStep* __restrict__ steps,
                                                                       const ChainTask* __restrict__ tasks,
                                                                       const int32_t* __restrict__ levels,
                                                                       int32_t n_levels, int32_t nb,
                                                                       int32_t skip_unbatched) {
  static_assert(!(CPLX && MAXPLUS), "the max-plus semiring is real");
  __shared__ ChainStep s_step[kChainWarps];
  pdl_wait();
  pdl_next();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w = blockIdx.x * kChainWarps + warp, W = gridDim.x * kChainWarps;
  ChainStep& S = s_step[warp];
  // level l: bounds, this warp's first task and its step's words; each fetched a level after
  // the one it depends on
  auto bound = [&](int l) { return __ldg(levels + (l < n_levels ? l : n_levels)); };
  auto task_at = [&](int t, int end) {
    ChainTask x{0, 0, 0, 0};
    if (t < end) {
      const int4 v = __ldg(reinterpret_cast<const int4*>(tasks + t));
      x = ChainTask{v.x, v.y, v.z, v.w};
    }
    return x;
  };
  auto fetch = [&](const ChainTask& t, uint32_t (&v)[kLaneWords]) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(steps + t.step);
#pragma unroll
    for (int i = 0; i < kLaneWords; ++i) v[i] = t.count && lane + 32 * i < kStepWords ? __ldg(src + lane + 32 * i) : 0u;
  };
  auto publish = [&](const uint32_t (&v)[kLaneWords]) {
    __syncwarp();  // the previous task's reads of the slot
#pragma unroll
    for (int i = 0; i < kLaneWords; ++i)
      if (lane + 32 * i < kStepWords) reinterpret_cast<uint32_t*>(&S)[lane + 32 * i] = v[i];
    __syncwarp();
  };
  auto run = [&](const ChainTask& t) {
    // a later pass keeps the slice-invariant steps' results; a short one has fewer entries
    if (S.batched ? t.b < nb : !skip_unbatched) run_task<CPLX, MAXPLUS>(S, t, lane);
  };
  int b0 = bound(0), b1 = bound(1), b2 = bound(2), b3 = bound(3);
  ChainTask t0 = task_at(b0 + w, b1), t1 = task_at(b1 + w, b2);
  uint32_t v[kLaneWords];
  fetch(t0, v);
  for (int l = 0; l < n_levels; ++l) {
    if (t0.count) publish(v);
    const int b4 = bound(l + 4);
    const ChainTask t2 = task_at(b2 + w, b3);
    fetch(t1, v);
    if (t0.count) run(t0);
    for (int t = b0 + w + W; t < b1; t += W) {
      const ChainTask x = task_at(t, b1);
      uint32_t u[kLaneWords];
      fetch(x, u);
      publish(u);
      run(x);
    }
    if (l + 1 < n_levels) level_barrier();
    b0 = b1;
    b1 = b2;
    b2 = b3;
    b3 = b4;
    t0 = t1;
    t1 = t2;
  }
}

// kChainMaxCtas if the kernel may take and the device has room for so large a cluster, else 8. The
// allowance (clusters above 8 are not portable) belongs to the current device, so each
// launch that needs it sets it; the room is the device's, asked for once.
template <bool CPLX, bool MAXPLUS>
int largest_cluster() {
  auto kern = contract_chain_kernel<CPLX, MAXPLUS>;
  int dev = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 8;
  }
  constexpr int kKnown = 64;
  static std::atomic<int> known[kKnown];
  const int slot = dev < kKnown ? dev : -1;
  int most = slot >= 0 ? known[slot].load(std::memory_order_relaxed) : 0;
  if (most > 0) return most;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kChainMaxCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(kChainMaxCtas);
  cfg.blockDim = dim3(kChainThreads);
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  most = 8;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) cudaGetLastError();
  else if (n >= 1) most = kChainMaxCtas;
  if (slot >= 0) known[slot].store(most, std::memory_order_relaxed);
  return most;
}

template <bool CPLX, bool MAXPLUS>
cudaError_t launch(const ChainStep* steps, const ChainTask* tasks, const int32_t* levels, int32_t n_levels,
                   int32_t ctas, int32_t nb, bool skip_unbatched, cudaStream_t st) {
  auto kern = contract_chain_kernel<CPLX, MAXPLUS>;
  const int most = n_levels > 1 && ctas > 8 ? largest_cluster<CPLX, MAXPLUS>() : 8;
  // one level: no barrier, so no cluster and no limit on the CTAs
  const int c = n_levels == 1 || ctas < most ? ctas : most;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = static_cast<unsigned>(c);
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(c));
  cfg.blockDim = dim3(kChainThreads);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = n_levels == 1 ? 1 : 2;
  return cudaLaunchKernelEx(&cfg, kern, steps, tasks, levels, n_levels, nb, static_cast<int32_t>(skip_unbatched));
}

}  // namespace

cudaError_t launch_contract_chain(const ChainStep* steps, const ChainTask* tasks, const int32_t* levels,
                                  int32_t n_levels, int32_t ctas, int32_t nb, bool skip_unbatched, bool cplx,
                                  bool maxplus, cudaStream_t st) {
  if (cplx) return launch<true, false>(steps, tasks, levels, n_levels, ctas, nb, skip_unbatched, st);
  if (maxplus) return launch<false, true>(steps, tasks, levels, n_levels, ctas, nb, skip_unbatched, st);
  return launch<false, false>(steps, tasks, levels, n_levels, ctas, nb, skip_unbatched, st);
}

}  // namespace tn
