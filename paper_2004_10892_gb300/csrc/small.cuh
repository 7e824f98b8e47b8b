// small.cuh -- a whole small plan in one kernel (k_small): a thread-block
// cluster contracts one item (slice, or bitstring and slice) from the gate
// tensors to its amplitude.
#pragma once
#include <cuda_runtime.h>

#include "program.hpp"

namespace tnq {

struct LeafDev {
  float2 val[4];      // entries when nv <= 2: (a, b) at a + 2b
  long long tab;      // nv > 2 (general networks): element offset of the 2^nv entries in the leaf value table
  long long off;      // element offset in the arena
  int nv;             // tensor variables (binary; entry index sum_x a_x 2^x)
  int n_free;         // leaf rank
  int dep;            // item-dependent in this configuration
  int pad;
  signed char vkind[LEAF_VMAX];  // 0 free, 1 fixed to 0 (input wire), 2 output bit, 3 sliced
  short varg[LEAF_VMAX];         // free: bit in the leaf; output: qubit; sliced: j
};

// Entry a of a leaf: inline for gates, from the value table for general tensors.
__device__ __forceinline__ float2 leaf_entry(const LeafDev& L, const float2* __restrict__ vals, int a) {
  return L.nv <= 2 ? L.val[a] : vals[L.tab + a];
}

constexpr int STPB = 512;               // threads per block
constexpr int SMALL_SHARED = 1 << 30;   // tensor offsets with this bit lie in shared memory
constexpr int SMALL_WORDS = 128;        // 32-bit words of a bitstring passed with the launch

// One input of a bucket. Its variables are the output's under `mask` (in the
// same order) above the eliminated one at bit 0: output entry b is entry
// compress(b, mask) of it; mv are the five shift masks of that compression.
struct SmallIn {
  int off;
  int meta;            // producing bucket (its scale), -1: gate tensor
  unsigned mask, mv[5];
};

// A gate tensor of at most two variables, restricted to the item's values.
struct SmallLeaf {
  float2 val[4];       // entry (a, b) at a + 2b
  int off;
  short n_free;        // variables that stay
  signed char kind[2];  // per gate variable: 0 free, 1 fixed to 0, 2 output bit, 3 sliced
  short arg[2];        // free: bit in the leaf; output: qubit; sliced: bit of the slice
  int pad;
};
static_assert(sizeof(SmallLeaf) == 48, "copied in 16-byte units");

struct SmallOp {
  int out;             // offset of the result
  int first;           // first entry within its level
  int bits;            // output variables
  int in0, nin;        // inputs, in the order they are multiplied
  int sum;             // 1: sum over bit 0 of every input (Eq. 2), 0: product only
  int split;           // 0: one product, added over the two values; else the first `split` inputs (one or two) are a
                       // product of their own, times which the others' is summed by FMAs (k_group's arithmetic)
};

// Buckets that depend on earlier levels only.
struct SmallLevel {
  int op0, nop, entries;
  int wide;            // 1: the whole cluster, 0: its first block
};

struct SmallArgs {
  const float4* tables;          // SmallIn, SmallLeaf, SmallLevel, SmallOp arrays, each on a 16-byte boundary
  const LeafDev* leaves;         // gate tensors of more than two variables (general networks)
  const LeafDev* scalars;
  const int* inout;
  const int2* finals;            // (offset, bucket)
  const float2* vals;
  float2* arena;                 // global part, per item
  double2* res;
  const unsigned* bits;          // bitstrings; null: the one in `words`
  unsigned long long item_base, bstr_base;
  long long arena_elems;         // per item
  int n_ops, n_ins, n_levels, n_small, n_leaves, n_scalars, n_inout, n_finals, smem_elems;
  int mode, p, n_words, scale_exp, scale_half;
  unsigned words[SMALL_WORDS];
};

// Bytes of the tables, and dynamic shared memory of one block (tensors, tables, maxima).
inline size_t small_tables_bytes(const SmallArgs& a) {
  auto up = [](size_t b) { return (b + 15) / 16 * 16; };
  return up((size_t)a.n_ins * sizeof(SmallIn)) + up((size_t)a.n_small * sizeof(SmallLeaf)) +
         up((size_t)a.n_levels * sizeof(SmallLevel)) + up((size_t)a.n_ops * sizeof(SmallOp));
}
inline size_t small_smem(const SmallArgs& a) {
  return (size_t)(a.smem_elems + 2) * 8 + small_tables_bytes(a) + ((size_t)a.n_ops + 1) * 4;
}
constexpr size_t SMALL_SMEM_MAX = 200 * 1024;
// Most clusters of `cluster` blocks that the device holds at once.
cudaError_t small_resident(const SmallArgs& a, int cluster, int* clusters);
// Contracts n_items items with `cluster` blocks each.
cudaError_t small_launch(const SmallArgs& a, int n_items, int cluster, cudaStream_t s);

}  // namespace tnq
