// Tables of the batched small-network engine (batch.cu), shared with the serve loop,
// which packs compatible small requests into one launch of the same kernel.
#pragma once

#include <algorithm>
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "tn_internal.h"

namespace tn {

constexpr int kBMaxDims = 8;    // merged offset dims per side in the batch tables
constexpr int kBMaxRank = 8;    // planned leaf rank in the batch tables

// Mixed-radix digit maps (planned positions of a leaf, merged dims of a step's rows and
// columns): digit d of an index times its stride, summed. When every extent is a power of two
// (and below 2^23) ext[d] holds the digit's place instead, shift | (extent - 1) << 8, so that a
// digit costs a shift and a mask and does not wait for the one before it.
struct alignas(16) BLeaf {
  int32_t src;                  // element offset in the network's own inputs
  int32_t dst;                  // float offset in the network's arena (real plane)
  int32_t size;
  int32_t rank;                 // planned positions | kBPow2
  int32_t ext[kBMaxRank];
  int32_t sstride[kBMaxRank];   // declared stride of each planned position
};

struct alignas(16) BStep {
  int32_t a, b, c;              // float offsets in the arena (real planes; imaginary ones follow them)
  int32_t m, n, k;
  int32_t pa, pb;               // producing step (kBLeafId: a leaf) | row / column dims << 27 (pa: | kBPow2)
  int32_t rext[kBMaxDims], rstr[kBMaxDims];
  int32_t cext[kBMaxDims], cstr[kBMaxDims];
};
constexpr int32_t kBPow2 = INT32_MIN;           // the map's extents are all powers of two
constexpr int32_t kBLeafId = (1 << 27) - 1;

struct BNet {
  int64_t arena;                // float offset of the network's arena in the batch arena
  int64_t in;                   // element offset of its inputs in the packed input buffer
  int32_t leaf0, n_leaves;      // index range in the leaf table
  int32_t step0, n_steps;       // index range in the step table
  int32_t root, root_size;      // float offset and size of the result tensor
  int32_t arena_floats;         // size of the network's arena
  int32_t index;                // row of its results
};

// One network's tables, offsets relative to the network itself (arena floats from 0,
// leaf sources from 0 in the network's own packed inputs, leaf and step indices from 0).
struct BatchTemplate {
  std::vector<BLeaf> leaves;
  std::vector<BStep> steps;
  int64_t arena_floats = 0;     // 256-byte aligned
  int64_t input_elems = 0;      // elements of the network's packed inputs
  int32_t root = 0, root_size = 0;
  int32_t max_tab = 0;          // largest m + n of its steps (the offset table it needs)
  double flops = 0;
};

// offset-table entries per network slot at most (steps with larger m + n compute offsets
// element by element)
constexpr int32_t kMaxTabInts = 4096;

// Step outputs whose exponents a team keeps (bytes of shared memory per CTA / per warp's share):
// networks with more steps renormalise each output in place.
constexpr int kExpBytes = 2048;
// the kernel's static shared memory at most: the exponents, two step records, scalars
constexpr int kBatchStaticSmem = kExpBytes + 2 * int(sizeof(BStep)) + 64;

constexpr int64_t kMaxSmemPerCta = 227 * 1024;  // dynamic shared memory one CTA may take
constexpr int64_t kSmemPerSm = 224 * 1024;      // what the SM's resident CTAs share (with headroom)

// Floats of the shared-memory arena of a packed launch's CTAs, per_sm of them on an SM together with
// their offset tables: an SM's 228 KB hold, per CTA, 1 KB of the system's and the static part too.
inline int32_t pack_arena_floats(int per_sm, int32_t tab_ints, int64_t max_arena) {
  const int64_t share = std::min(int64_t(228 * 1024) / per_sm - 1024, kMaxSmemPerCta) - kBatchStaticSmem;
  return static_cast<int32_t>(std::max<int64_t>(0, std::min(share / 256 * 64 - tab_ints, max_arena)));
}

// Tables of a closed, unsliced network from its plan (workspace assigned for one copy, no
// tensor-core steps); false with a reason when the batched kernel cannot run it.
bool batch_template(const Plan& P, BatchTemplate& T, std::string& err);

// Launch the persistent kernel over n_nets networks (queue reset included): a CTA of
// `threads` per network, or with `warp` a warp per network (threads = 32 x warps per CTA).
// smem_arena > 0: a network whose arena holds at most smem_arena floats runs in a
// shared-memory arena of that size (one per CTA, or per warp), the others in `arena`.
// tab_ints > 0: each slot also gets a shared-memory table of that many ints for the output
// offsets of a step's rows and columns (steps with m + n above it compute them per element).
cudaError_t launch_batch_kernel(const BNet* nets, const BLeaf* leaves, const BStep* steps, int32_t n_nets,
                                const void* packed, float* arena, int32_t* queue, bool cplx, bool scaling,
                                bool maxplus, int threads, int grid, double* values, double* logs,
                                cudaStream_t st, bool warp = false, int32_t smem_arena = 0, int32_t tab_ints = 0);

}  // namespace tn
