// pair.cuh -- a fused chain of buckets as a register-tiled product of its two
// large tensors (k_pair), optionally times a third one.
//
// A chain's result is out[o] = sum_K A B C prod_g g over the chain's
// eliminated variables K (Eq. 2 applied m times, regrouped; m = 1: a single
// bucket), with large tensors A and B that both hold the first eliminated
// variable u_0, at most one other large tensor C, and small tensors g, each of
// which has its variables among A's or among B's and is folded into that one.
// With K2 = K & vars(C) and K1 = K - K2:
//   out[o] = sum_K2 C[K2, o] (sum_K1 A[K1, K2, o] B[K1, K2, o]).
// With one large tensor only (B) the small tensors' product takes A's place.
// A GEMM chain of mostly padding comes here too; in 3xBF16 it keeps that
// precision's sums (`split`).
#pragma once
#include <cuda_runtime.h>

namespace tnq {

constexpr int PTB = 8;              // log2 threads per k_pair block
constexpr int PTPB = 1 << PTB;
constexpr int PRX_MAX = 2;          // register tile: up to 2^2 entries along A's variables ...
constexpr int PRY_MAX = 3;          // ... x 2^2 or 2^3 along B's
constexpr int PE_MAX = 13;          // staged (u = 0, u = 1) pairs of one operand: at most 2^13
constexpr int PF_MAX = 7;           // fold table of one operand: at most 2^8 pairs
constexpr int PIN_MAX = 16;         // tensors a chain reads
constexpr int PH_MAX = 32;          // tile bits
constexpr int PL_MAX = 3;            // output variables of a thread's loop
constexpr int PK_MAX = 5;           // eliminated variables of one loop
constexpr int PAIR_SMEM_TWO = 98 * 1024;   // two stages of one block's operands, so that two blocks fit an SM
constexpr int PAIR_SMEM_MAX = 200 * 1024;  // ... or one

// One tensor that the chain reads from memory.
struct PIn {
  const float2* ptr;
  long long istride;            // per item (0 if item-invariant)
  int meta;                     // meta row (-1: gate tensor, unit scale)
  int dep;
};

// A staged operand. Its local entries are enumerated as pairs over its bit 0
// by an index e (bits by increasing memory stride, so that consecutive threads
// read consecutive memory); bit i of e adds g[i] to the global offset
// (elements) and f[i] to the fold table's index, and is d[i] of the
// shared-memory slot (bytes): slots are combined with XOR, since they
// are swizzled (pair_params). Tile bit i adds h[i] and fh[i], bit i of the chunk gch[i] and fch[i].
struct POp {
  int gin;
  int ebits;
  int g[PE_MAX], d[PE_MAX], f[PE_MAX];
  int h[PH_MAX], fh[PH_MAX];
  int gch[2], fch[2];
  int base, size;               // bytes: its first stage (a multiple of size; the second follows it), a stage (a power of two)
};

// Small tensors folded into one operand: table of (u_0 = 0, u_0 = 1) pairs
// over the other variables that they hold, tile variables included: it depends
// on the item alone.
struct PFold {
  int n, nf;                    // tensors, table index bits
  int gin[PIN_MAX], ustride[PIN_MAX];
  int fs[PIN_MAX][PF_MAX];      // element stride of table index bit b
};

struct PairParams {
  PIn gin[PIN_MAX];
  POp a, b, c;                  // a.gin < 0: B alone; c.gin < 0: no third tensor
  PFold fa, fb;
  float2* out;
  long long out_istride;
  int out_h[PH_MAX];            // per tile bit
  int ta[PTB], tb[PTB], tc[PTB], to[PTB];  // thread bits: slots of a, b, c; output offset
  int xa[PRX_MAX], xc[PRX_MAX], xo[PRX_MAX];   // register bits along A: slots of a and c, output offset (0 for a K2 bit)
  int yb[PRY_MAX], yc[PRY_MAX], yo[PRY_MAX];   // register bits along B
  int rx, ry;                   // register bits along A / B
  int c_u0;                     // 1: C holds u_0 (K2 then includes it)
  int split;                    // 1: 3xBF16 (two large tensors only): operands as bf16 hi + lo, without lo times lo
  int nl, la[PL_MAX], lb[PL_MAX], lc[PL_MAX], lo[PL_MAX];  // a thread's loop over outputs
  int ft[PTB], yf[PRY_MAX], k1f[PK_MAX];        // B alone: the fold table's index instead of A's slots
  int n1, k1a[PK_MAX], k1b[PK_MAX];                // K1 without u_0 and the chunk's variable: slots of a and b
  int n2, k2a[PK_MAX], k2b[PK_MAX], k2c[PK_MAX];   // K2 outside the register tile
  int nkx, nky;                 // K2 bits among the register bits along A / B (the low ones)
  int n_ch;                     // chunks of a tile: one summed variable (2) or two (4) split off, or none (1)
  int n_h, n_gin, out_meta, out_dep, B;
  int smem;                     // dynamic shared memory bytes
  int* meta_e;
  unsigned* meta_m;
  const int* n_items;           // valid items of the batch (device; null: the batch is one item)
};

// Blocks of k_pair that fit the device at once for this shape; 0 and *err on failure.
int pair_grid(const PairParams& p, cudaError_t* err);
// Launches the chain over n_tiles tiles (item, tile variables).
void pair_launch(const PairParams& p, long long n_tiles, int grid, cudaStream_t s);

}  // namespace tnq
