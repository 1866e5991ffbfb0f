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
// 12-qubit amplitude's 57 steps (12 levels) 84 -> 29 us.
#include <cstdint>

#include <cuda_runtime.h>

#include "kernels.h"
#include "scale.cuh"
#include "split_bf16.cuh"

namespace tn {
namespace {

constexpr int kChainThreads = 512;
constexpr int kChainWarps = kChainThreads / 32;
constexpr int kStepWords = sizeof(ChainStep) / 4;
constexpr int kLaneWords = (kStepWords + 31) / 32;
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

// Offset of index i under the merged dims d0 .. d1 - 1 of a step (last fastest): extents packed
// with their log2 (0xff: not a power of two), strides in elements.
__device__ __forceinline__ int dims_offset(const ChainStep& S, int d0, int d1, uint32_t i) {
  int off = 0;
  for (int d = d1 - 1; d >= d0; --d) {
    const uint32_t e = S.ext[d] & 0xffffffu, sh = S.ext[d] >> 24;
    uint32_t q, r;
    if (sh != 0xffu) {
      q = i >> sh;
      r = i & (e - 1u);
    } else {
      q = i / e;
      r = i - q * e;
    }
    off += static_cast<int>(r) * S.stride[d];
    i = q;
  }
  return off;
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
  int lmax = -127;
  for (int idx = t.first + lane; idx < t.first + t.count; idx += 32) {
    const int r = S.n_shift >= 0 ? idx >> S.n_shift : idx / S.n, c = idx - r * S.n;
    const float* ar = A + r * k;
    const float* br = B + c * k;
    float accr = kZero, acci = kZero;
    for (int k0 = 0; k0 < k; k0 += U) {
      float xr[U], yr[U], xi[CPLX ? U : 1], yi[CPLX ? U : 1];
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
        const float vr = xr[u] * sa, wr = yr[u] * sb;
        if (CPLX) {
          const float vi = xi[u] * sa, wi = yi[u] * sb;
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
    }
    const int off = dims_offset(S, 0, S.nr, r) + dims_offset(S, kMaxDims, kMaxDims + S.nc, c);
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

template <bool CPLX, bool MAXPLUS>
cudaError_t launch(const ChainStep* steps, const ChainTask* tasks, const int32_t* levels, int32_t n_levels,
                   int32_t ctas, int32_t nb, bool skip_unbatched, cudaStream_t st) {
  auto kern = contract_chain_kernel<CPLX, MAXPLUS>;
  // clusters of 16 need the non-portable size and room for one on the device
  static const int most = [kern] {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return 8;
    }
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
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return 8;
    }
    return static_cast<int>(kChainMaxCtas);
  }();
  // one level: no barrier, so no cluster and no limit on the CTAs
  const int c = n_levels == 1 || ctas < most ? ctas : most;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = static_cast<unsigned>(c);
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(c));
  cfg.blockDim = dim3(kChainThreads);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = n_levels == 1 ? 0 : 1;
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
