// pair.cu -- k_pair: a fused chain of buckets as a register-tiled contraction
// (see pair.cuh).
#include <cuda_bf16.h>

#include "device_util.cuh"
#include "pair.cuh"

namespace tnq {

// Fold table entry e of one operand: the product of its small tensors at u_0 =
// 0 and 1, each times its scale, starting from (f, 0).
__device__ __forceinline__ float4 fold_entry(const PairParams& P, const PFold& F, int e, long long item, float f,
                                             const float* scale) {
  float2 p0 = make_float2(f, 0.f), p1 = p0;
  for (int j = 0; j < F.n; ++j) {
    const PIn& g = P.gin[F.gin[j]];
    const float2* q = g.ptr + (g.dep ? item * g.istride : 0ll);
#pragma unroll
    for (int i = 0; i < PF_MAX; ++i)
      if (i < F.nf && ((e >> i) & 1)) q += F.fs[j][i];
    const float s = scale[F.gin[j]];
    const float2 v0 = __ldg(q), v1 = __ldg(q + F.ustride[j]);
    p0 = cmul(p0, make_float2(v0.x * s, v0.y * s));
    p1 = cmul(p1, make_float2(v1.x * s, v1.y * s));
  }
  return make_float4(p0.x, p0.y, p1.x, p1.y);
}

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cfma(float2& r, float2 a, float2 b) {
  r.x = fmaf(a.x, b.x, r.x);
  r.y = fmaf(a.x, b.y, r.y);
  r.x = fmaf(-a.y, b.y, r.x);
  r.y = fmaf(a.y, b.x, r.y);
}

// r += a b over the pair's two values
__device__ __forceinline__ void cfma2(float2& r, float4 a, float4 b) {
  r.x = fmaf(a.x, b.x, r.x);
  r.y = fmaf(a.x, b.y, r.y);
  r.x = fmaf(-a.y, b.y, r.x);
  r.y = fmaf(a.y, b.x, r.y);
  r.x = fmaf(a.z, b.z, r.x);
  r.y = fmaf(a.z, b.w, r.y);
  r.x = fmaf(-a.w, b.w, r.x);
  r.y = fmaf(a.w, b.z, r.y);
}

// 3xBF16 as the GEMM packs it: x = hi + lo, two roundings to bf16. hi + lo is a
// float itself, so an operand is staged as that sum, and of a product a b the
// GEMM's three terms are a b - lo(a) lo(b).
__device__ __forceinline__ float2 bf16_lo(float2 x) {
  const float2 h = __bfloat1622float2(__float22bfloat162_rn(x));
  return make_float2(x.x - h.x, x.y - h.y);
}
__device__ __forceinline__ float2 bf16_split(float2 x) {
  const float2 h = __bfloat1622float2(__float22bfloat162_rn(x));
  const float2 l = __bfloat1622float2(__float22bfloat162_rn(make_float2(x.x - h.x, x.y - h.y)));
  return make_float2(h.x + l.x, h.y + l.y);
}
template <class F>
__device__ __forceinline__ float4 both(F f, float4 v, float sign = 1.f) {  // f of the pair's two values
  const float2 a = f(make_float2(v.x, v.y)), b = f(make_float2(v.z, v.w));
  return make_float4(sign * a.x, sign * a.y, sign * b.x, sign * b.y);
}

// Persistent: a block loops over tiles (item, tile variables), a tile over one,
// two or four chunks of its summed values. Two stages: while a chunk is computed,
// the next one's part of A, B (and C) comes in by cp.async; each thread then
// multiplies what it copied by the fold tables in place, and after one barrier
// every thread computes 4 x 2^RY register tiles: per pair of summed values 4 + 2^RY
// 16-byte shared loads feed 32 x 2^RY FMAs. Shared memory delivers 128 bytes a
// cycle to registers, so 4 x 4 needs all of it at the full FMA rate and 4 x 8
// three quarters.
//
// What bounds it, and GB300 figures against the bucket-by-bucket chain kernel
// (k_group) that ran these chains:
//  * two tensors: the FMA pipe (78 TFLOP/s measured). 5 buckets, bag 28, 32
//    items: 12.9 -> 1.97 ms, 72 TFLOP/s.
//  * three: issue slots (68 % busy, 62 % of them FMAs; 128 registers hold two
//    blocks an SM, and three of the 4 x 8 forms with C spill 5 to 41 words to
//    fit them) and the reads of C, each used once. 3 buckets, bag 28, 64 items:
//    19.9 -> 5.57 ms, 36 TFLOP/s.
//  * one: memory. A bucket of bag 23, 32 items: 4.0 -> 5.5 TB/s (k_bucket
//    before); 5 buckets, bag 22: 3.5 -> 5.2 TB/s of a copy's 6.8.
//  * 3xBF16 chains of mostly padding: memory too; eight instructions a value
//    for its low part. One row, 64 columns, K = 32, bag 25, 8 items: 4.11 (the
//    padded GEMM) -> 0.66 ms, 0.49 in plain FP32.
// Slower: register double buffering by halves of a pair (8-byte reads at a
// 16-byte stride cost twice the cycles, 2.28 -> 2.85 ms on the first); no
// faster: three or four stages.
// CM: 0 no C, 1 C without u_0 (its bit 0 is B's register bit 0), 2 C with u_0,
// 3 B alone: B comes through shared memory only to be read in consecutive
// pieces, and is multiplied by the small tensors' product as it is summed.
// SPLIT: 3xBF16 (CM 0 only).
template <int RX, int RY, int NKX, int NKY, int CM, bool SPLIT = false>
__global__ void __launch_bounds__(PTPB, 2) k_pair(const __grid_constant__ PairParams P, long long n_tiles) {
  extern __shared__ float4 sm[];
  constexpr bool HASC = CM == 1 || CM == 2, ONE = CM == 3;
  constexpr int NOP = HASC ? 3 : 2, OP0 = ONE ? 1 : 0;
  constexpr int RING = 4;  // a thread is at most one barrier ahead: what it writes is two tiles ahead
  __shared__ float4 s_fa[2][1 << PF_MAX], s_fb[2][1 << PF_MAX];  // by item, alternating
  __shared__ int4 s_it[NOP][1 << (PE_MAX - PTB)];  // staging iteration: global offset, slot, fold index
  __shared__ int4 s_k2[1 << PK_MAX];               // K2 outside the register tile: slots of a, b, c
  __shared__ int4 s_l[1 << PL_MAX];                // a thread's loop: slots of a, b, c, output offset
  __shared__ int2 s_k1[1 << PK_MAX];               // K1 pairs of a chunk: slots of a, b
  __shared__ int s_hstr[6][PH_MAX];
  __shared__ const float2* s_src[RING][3];
  __shared__ float2* s_out[RING];
  __shared__ int s_fold[RING][2];
  __shared__ float s_sc[PIN_MAX];  // scales of an item's inputs, and their exponents
  __shared__ int s_m[PIN_MAX];
  __shared__ float s_mul[2][4];    // per operand: scale of its staged entries; [3]: 1 when none is needed
  __shared__ int s_e[RING][PIN_MAX];
  __shared__ float s_red[PTPB / 32];
  constexpr int NX = 1 << RX, NY = 1 << RY;
  const int t = threadIdx.x, lane = t & 31;
  const POp* ops[3] = {&P.a, &P.b, &P.c};
  if (P.out_dep && P.n_items) n_tiles = (long long)*P.n_items << P.n_h;
  if (blockIdx.x >= n_tiles) return;
  // ---- tables that every tile uses
  if (t < PH_MAX) {
    s_hstr[0][t] = !ONE && t < P.n_h ? P.a.h[t] : 0;
    s_hstr[1][t] = t < P.n_h ? P.b.h[t] : 0;
    s_hstr[2][t] = HASC && t < P.n_h ? P.c.h[t] : 0;
    s_hstr[3][t] = t < P.n_h ? P.out_h[t] : 0;
    s_hstr[4][t] = t < P.n_h ? P.a.fh[t] : 0;
    s_hstr[5][t] = t < P.n_h ? P.b.fh[t] : 0;
    int4 v = make_int4(0, 0, 0, 0);
    for (int i = 0; i < P.n2; ++i)
      if ((t >> i) & 1) {
        v.x ^= P.k2a[i];
        v.y ^= P.k2b[i];
        v.z ^= P.k2c[i];
      }
    s_k2[t] = v;
    int2 w = make_int2(0, 0);
    for (int i = 0; i < P.n1; ++i)
      if ((t >> i) & 1) {
        w.x ^= ONE ? P.k1f[i] : P.k1a[i];
        w.y ^= P.k1b[i];
      }
    s_k1[t] = w;
  }
  if (t < (1 << PL_MAX)) {
    int4 v = make_int4(0, 0, 0, 0);
    for (int i = 0; i < P.nl; ++i)
      if ((t >> i) & 1) {
        v.x ^= P.la[i];
        v.y ^= P.lb[i];
        v.z ^= P.lc[i];
        v.w += P.lo[i];
      }
    s_l[t] = v;
  }
  int tg[NOP], td[NOP], tf[NOP];  // this thread's part of the staging offsets
#pragma unroll
  for (int o = OP0; o < NOP; ++o) {
    const POp& O = *ops[o];
    tg[o] = tf[o] = td[o] = 0;
#pragma unroll
    for (int i = 0; i < PTB; ++i)
      if (i < O.ebits && ((t >> i) & 1)) {
        tg[o] += O.g[i];
        td[o] ^= O.d[i];
        tf[o] += O.f[i];
      }
    const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
    if (t < nit) {
      int4 v = make_int4(0, 0, 0, 0);
      for (int i = PTB; i < O.ebits; ++i)
        if ((t >> (i - PTB)) & 1) {
          v.x += O.g[i];
          v.y ^= O.d[i];
          v.z += O.f[i];
        }
      s_it[o][t] = v;
    }
  }
  int ra = 0, rb = 0, rc = 0, ro = 0;  // this thread's register tile
#pragma unroll
  for (int i = 0; i < PTB; ++i)
    if ((t >> i) & 1) {
      ra ^= ONE ? P.ft[i] : P.ta[i];
      rb ^= P.tb[i];
      if (HASC) rc ^= P.tc[i];
      ro += P.to[i];
    }
  const bool fold_a = P.fa.n > 0;
  const unsigned sm0 = (unsigned)__cvta_generic_to_shared(sm);
  char* smb = reinterpret_cast<char*>(sm);
  __syncthreads();

  // pointers and fold offsets of a tile: one warp per value, lane i adds tile bit i's stride
  auto tile_setup = [&](long long tile, int slot) {
    const long long item = tile >> P.n_h;
    const int h = (int)(tile & ((1ll << P.n_h) - 1ll));
    const int w = t >> 5;
    if (w >= 6) return;
    const int v = __reduce_add_sync(0xffffffffu, ((h >> lane) & 1) ? s_hstr[w][lane] : 0);
    if (lane) return;
    if (w < NOP) {
      if (w < OP0) return;
      const PIn& g = P.gin[w == 0 ? P.a.gin : (w == 1 ? P.b.gin : P.c.gin)];
      s_src[slot][w] = g.ptr + (g.dep ? item * g.istride : 0ll) + v;
    } else if (w == 3) {
      s_out[slot] = P.out + (P.out_dep ? item * P.out_istride : 0ll) + v;
    } else if (w >= 4) {
      s_fold[slot][w - 4] = v;
    }
  };
  // Exponents, scales and fold tables of an item. Every input counts with its
  // own power of two, as in k_bucket: their product would leave FP32's range at
  // two inputs of 2^-64. A folded tensor's goes into its table, and an operand's
  // into B's while it is below 2^PAIR_SCALE (no work then: three of them fit the
  // table's range); beyond, the operand's staged entries are multiplied by it.
  // One operand alone keeps its scale in the table, up to 2^PAIR_ONE.
  constexpr int PAIR_SCALE = 20, PAIR_ONE = 100;
  auto item_setup = [&](long long item, int n) {
    if (t < P.n_gin) {
      const PIn& g = P.gin[t];
      int m = 0, e = 0;
      float f = 1.f;
      if (g.meta >= 0) {
        const long long row = (long long)g.meta * P.B + (g.dep ? item : 0ll);
        f = scale_of_max(P.meta_m[row], &m);
        if (ONE && t == P.b.gin) m = max(-PAIR_ONE, min(PAIR_ONE, m));
        e = P.meta_e[row] + m;
      }
      s_sc[t] = f;
      s_m[t] = m;
      s_e[n % RING][t] = e;
    }
    __syncthreads();
    int in_table = 0;
    float mul[3] = {1.f, 1.f, 1.f};
#pragma unroll
    for (int o = OP0; o < NOP; ++o) {
      const int j = ops[o]->gin;
      if (ONE || abs(s_m[j]) <= PAIR_SCALE) in_table += s_m[j];
      else mul[o] = s_sc[j];
    }
    if (t < (1 << P.fb.nf))
      s_fb[n & 1][t] = fold_entry(P, P.fb, t, item, __int_as_float((127 - in_table) << 23), s_sc);
    if (fold_a && t < (1 << P.fa.nf)) s_fa[n & 1][t] = fold_entry(P, P.fa, t, item, 1.f, s_sc);
    if (t == 0) {
      for (int o = 0; o < 3; ++o) s_mul[n & 1][o] = mul[o];
      s_mul[n & 1][3] = mul[0] == 1.f && mul[1] == 1.f && mul[2] == 1.f ? 1.f : 0.f;
    }
  };
  auto issue = [&](int slot, int chunk, int buf) {
#pragma unroll
    for (int o = OP0; o < NOP; ++o) {
      const POp& O = *ops[o];
      const float2* src = s_src[slot][o] + tg[o] + ((chunk & 1) ? O.gch[0] : 0) + ((chunk & 2) ? O.gch[1] : 0);
      const int at = td[o] ^ (O.base + (buf ? O.size : 0));
      const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
      if (O.ebits >= PTB || t < (1 << O.ebits))
        for (int it = 0; it < nit; ++it) {
          const int4 k = s_it[o][it];
          cp_async16(sm0 + (unsigned)(at ^ k.y), src + k.x);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // multiplies the pairs this thread copied by their operands' scales (out of the ordinary: see item_setup)
  auto rescale = [&](int buf, int n) {
#pragma unroll
    for (int o = OP0; o < NOP; ++o) {
      const POp& O = *ops[o];
      const float f = s_mul[n & 1][o];
      const int at = td[o] ^ (O.base + (buf ? O.size : 0));
      const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
      if (f != 1.f && (O.ebits >= PTB || t < (1 << O.ebits))) {
#pragma unroll 1
        for (int it = 0; it < nit; ++it) {
          float4& v = *reinterpret_cast<float4*>(smb + (at ^ s_it[o][it].y));
          v = make_float4(v.x * f, v.y * f, v.z * f, v.w * f);
        }
      }
    }
  };
  // multiplies the pairs this thread copied by the fold tables
  auto fold = [&](int slot, int chunk, int buf, int n) {
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const bool folded = o == 1 || fold_a;
      if (!SPLIT && !folded) continue;
      const POp& O = *ops[o];
      const float4* ft = (o == 0 ? s_fa[n & 1] : s_fb[n & 1]) + tf[o] + s_fold[slot][o] +
                         ((chunk & 1) ? O.fch[0] : 0) + ((chunk & 2) ? O.fch[1] : 0);
      const int at = td[o] ^ (O.base + (buf ? O.size : 0));
      const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
      if (O.ebits >= PTB || t < (1 << O.ebits)) {
#pragma unroll 2
        for (int it = 0; it < nit; ++it) {
          const int4 k = s_it[o][it];
          float4& dst = *reinterpret_cast<float4*>(smb + (at ^ k.y));
          float4 v = dst;
          if (folded) {
            const float4 f = ft[k.z];
            const float2 v0 = cmul(make_float2(v.x, v.y), make_float2(f.x, f.y));
            const float2 v1 = cmul(make_float2(v.z, v.w), make_float2(f.z, f.w));
            v = make_float4(v0.x, v0.y, v1.x, v1.y);
          }
          dst = SPLIT ? both(bf16_split, v) : v;
        }
      }
    }
  };
  float tmax = 0.f;
  auto flush = [&](long long item) {
    float m = tmax;
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __syncthreads();
    if (lane == 0) s_red[t >> 5] = m;
    __syncthreads();
    if (t == 0) {
      float b = 0.f;
      for (int w = 0; w < PTPB / 32; ++w) b = fmaxf(b, s_red[w]);
      if (b > 0.f) atomic_max_pos(&P.meta_m[(long long)P.out_meta * P.B + (P.out_dep ? item : 0ll)], b);
    }
    tmax = 0.f;
  };

  int n_item = 0, buf = 0;
  tile_setup(blockIdx.x, 0);
  item_setup((long long)blockIdx.x >> P.n_h, 0);
  __syncthreads();
  issue(0, 0, 0);
  int slot = 0;
  constexpr int XO = NX >> NKX, YO = NY >> NKY;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, slot = (slot + 1) % RING) {
    const long long item = tile >> P.n_h, next = tile + gridDim.x;
    const bool more = next < n_tiles;
    const bool new_item = more && (next >> P.n_h) != item;
    float2 x[NX][NY];  // sums of A B
    auto zero = [&] {
#pragma unroll
      for (int i = 0; i < NX; ++i)
#pragma unroll
        for (int j = 0; j < NY; ++j) x[i][j] = make_float2(0.f, 0.f);
    };
    for (int c = 0; c < P.n_ch; ++c) {
      const bool last = c + 1 == P.n_ch;
      if (last && more) {
        tile_setup(next, (slot + 1) % RING);
        if (new_item) item_setup(next >> P.n_h, n_item + 1);
      }
      const bool odd = !ONE && s_mul[n_item & 1][3] == 0.f;  // (fetched while the copies arrive)
      asm volatile("cp.async.wait_all;" ::: "memory");
      if (odd) rescale(buf, n_item);
      if constexpr (!ONE) fold(slot, c, buf, n_item);
      __syncthreads();  // the chunk is staged, and every thread is done with the other stage
      if (!last) issue(slot, c + 1, buf ^ 1);
      else if (more) issue((slot + 1) % RING, 0, buf ^ 1);
      // slots are byte offsets and stages aligned, so an address is one XOR
      const char* pa = ONE ? reinterpret_cast<const char*>(s_fb[n_item & 1] + s_fold[slot][1] +
                                                           ((c & 1) ? P.b.fch[0] : 0) + ((c & 2) ? P.b.fch[1] : 0))
                           : smb;
      const int ca = ONE ? ra : ra ^ (P.a.base + (buf ? P.a.size : 0)), cb = rb ^ (P.b.base + (buf ? P.b.size : 0));
      const int cc = HASC ? rc ^ (P.c.base + (buf ? P.c.size : 0)) : 0;
      auto quad = [](const char* p, int at) { return *reinterpret_cast<const float4*>(p + at); };
      auto elem = [](const char* p, int at) { return *reinterpret_cast<const float2*>(p + at); };
      float2* dst = s_out[slot] + ro;
      const int n1 = 1 << P.n1;
      auto off_x = [&](int i, const int* w) { return ((i & 1) ? w[0] : 0) ^ ((i & 2) ? w[1] : 0); };
      auto off_y = [&](int j, const int* w) {
        return ((j & 1) ? w[0] : 0) ^ ((j & 2) ? w[1] : 0) ^ (RY > 2 && (j & 4) ? w[2] : 0);
      };
      auto products = [&](int oa, int ob) {
#pragma unroll 1
        for (int q = 0; q < n1; ++q) {
          const int2 k = s_k1[q];
          const int qa = oa ^ k.x, qb = ob ^ k.y;
          float4 va[NX], la[SPLIT ? NX : 1];
#pragma unroll
          for (int i = 0; i < NX; ++i) {
            if (!ONE) va[i] = quad(pa, qa ^ off_x(i, P.xa));
            if constexpr (SPLIT) la[i] = both(bf16_lo, va[i], -1.f);
          }
#pragma unroll
          for (int j = 0; j < NY; ++j) {
            const float4 vb = quad(smb, qb ^ off_y(j, P.yb));
#pragma unroll
            for (int i = 0; i < NX; ++i) cfma2(x[i][j], ONE ? quad(pa, qa ^ off_y(j, P.yf)) : va[i], vb);
            if constexpr (SPLIT) {
              const float4 lb = both(bf16_lo, vb);
#pragma unroll
              for (int i = 0; i < NX; ++i) cfma2(x[i][j], la[i], lb);
            }
          }
        }
      };
      auto half_products = [&](int oa, int ob, int h) {  // u_0 = h alone
#pragma unroll 1
        for (int q = 0; q < n1; ++q) {
          const int2 k = s_k1[q];
          const int qa = oa ^ k.x ^ 8 * h, qb = ob ^ k.y ^ 8 * h;
          float2 va[NX];
#pragma unroll
          for (int i = 0; i < NX; ++i) va[i] = elem(smb, qa ^ off_x(i, P.xa));
#pragma unroll
          for (int j = 0; j < NY; ++j) {
            const float2 vb = elem(smb, qb ^ off_y(j, P.yb));
#pragma unroll
            for (int i = 0; i < NX; ++i) cfma(x[i][j], va[i], vb);
          }
        }
      };
      auto store = [&](int i, int j, float2 r, int lo) {
        const int ri = i << NKX, rj = j << NKY;
        dst[lo + ((ri & 1) ? P.xo[0] : 0) + ((ri & 2) ? P.xo[1] : 0) + ((rj & 1) ? P.yo[0] : 0) +
            ((rj & 2) ? P.yo[1] : 0) + (RY > 2 && (rj & 4) ? P.yo[2] : 0)] = r;
        tmax = fmaxf(tmax, fmaxf(fabsf(r.x), fabsf(r.y)));
      };
      const int nl = 1 << P.nl;
#pragma unroll 1
      for (int l = 0; l < nl; ++l) {
        const int4 lv = s_l[l];
        if constexpr (HASC) {
          float2 acc[XO][YO];
#pragma unroll
          for (int i = 0; i < XO; ++i)
#pragma unroll
            for (int j = 0; j < YO; ++j) acc[i][j] = make_float2(0.f, 0.f);
          const int n2 = 1 << P.n2;
#pragma unroll 1
          for (int q2 = 0; q2 < n2; ++q2) {
            const int4 k2 = s_k2[q2];
            const int oc = cc ^ lv.z ^ k2.z;
            if constexpr (CM == 2) {
#pragma unroll 1
              for (int h = 0; h < 2; ++h) {
                zero();
                half_products(ca ^ lv.x ^ k2.x, cb ^ lv.y ^ k2.y, h);
#pragma unroll
                for (int i = 0; i < NX; ++i)
#pragma unroll
                  for (int j = 0; j < NY; ++j)
                    cfma(acc[i >> NKX][j >> NKY], x[i][j], elem(smb, oc ^ 8 * h ^ off_x(i, P.xc) ^ off_y(j, P.yc)));
              }
            } else {
              zero();
              products(ca ^ lv.x ^ k2.x, cb ^ lv.y ^ k2.y);
              // times C, summed over the K2 register bits (C's bit 0 is B's register bit 0)
#pragma unroll
              for (int i = 0; i < NX; ++i)
#pragma unroll
                for (int j = 0; j < NY; j += 2) {
                  const float4 v = quad(smb, oc ^ off_x(i, P.xc) ^ off_y(j, P.yc));  // (yc[0] is 0: the pair's own bit)
                  const float2 u = x[i][j], w = x[i][j + 1];
                  cfma2(acc[i >> NKX][j >> NKY], make_float4(u.x, u.y, w.x, w.y), v);
                }
            }
          }
#pragma unroll
          for (int i = 0; i < XO; ++i)
#pragma unroll
            for (int j = 0; j < YO; ++j) store(i, j, acc[i][j], lv.w);
        } else {
          if (c == 0) zero();
          products(ca ^ lv.x, cb ^ lv.y);
          if (last) {
#pragma unroll
            for (int i = 0; i < NX; ++i)
#pragma unroll
              for (int j = 0; j < NY; ++j) store(i, j, x[i][j], lv.w);
          }
        }
      }
      buf ^= 1;
    }
    if (t == 0 && (tile & ((1ll << P.n_h) - 1ll)) == 0) {
      int e = 0;
      for (int j = 0; j < P.n_gin; ++j) e += s_e[n_item % RING][j];
      P.meta_e[(long long)P.out_meta * P.B + (P.out_dep ? item : 0ll)] = e;
    }
    if (new_item || !more) flush(item);
    n_item += new_item;
  }
}

using PairKernel = void (*)(PairParams, long long);
static PairKernel pair_kernel(const PairParams& p) {
  if (p.split) {
    if (p.rx == 2) return k_pair<2, 2, 0, 0, 0, true>;
    if (p.rx) return k_pair<1, 3, 0, 0, 0, true>;
    return p.ry > 1 ? k_pair<0, 3, 0, 0, 0, true> : k_pair<0, 1, 0, 0, 0, true>;
  }
  if (p.a.gin < 0) return p.ry > 1 ? k_pair<0, 3, 0, 0, 3> : k_pair<0, 1, 0, 0, 3>;
  if (p.c.gin < 0) {
    if (p.rx == 2) return p.ry > 2 ? k_pair<2, 3, 0, 0, 0> : k_pair<2, 2, 0, 0, 0>;
    if (p.rx) return k_pair<1, 3, 0, 0, 0>;
    return p.ry > 1 ? k_pair<0, 3, 0, 0, 0> : k_pair<0, 1, 0, 0, 0>;
  }
  if (p.ry > 2) switch (p.nkx * 3 + p.nky) {
    case 1: return k_pair<2, 3, 0, 1, 1>;
    case 2: return k_pair<2, 3, 0, 2, 1>;
    case 4: return k_pair<2, 3, 1, 1, 1>;
    case 5: return k_pair<2, 3, 1, 2, 1>;
    case 7: return k_pair<2, 3, 2, 1, 1>;
    default: return k_pair<2, 3, 2, 2, 1>;
  }
  switch ((p.c_u0 * 3 + p.nkx) * 3 + p.nky) {
    case 1: return k_pair<2, 2, 0, 1, 1>;
    case 2: return k_pair<2, 2, 0, 2, 1>;
    case 4: return k_pair<2, 2, 1, 1, 1>;
    case 5: return k_pair<2, 2, 1, 2, 1>;
    case 7: return k_pair<2, 2, 2, 1, 1>;
    case 8: return k_pair<2, 2, 2, 2, 1>;
    case 9: return k_pair<2, 2, 0, 0, 2>;
    case 10: return k_pair<2, 2, 0, 1, 2>;
    case 11: return k_pair<2, 2, 0, 2, 2>;
    case 13: return k_pair<2, 2, 1, 1, 2>;
    case 14: return k_pair<2, 2, 1, 2, 2>;
    default: return k_pair<2, 2, 2, 2, 2>;
  }
}

int pair_grid(const PairParams& p, cudaError_t* err) {
  const PairKernel k = pair_kernel(p);
  int dev = 0, sms = 0, per_sm = 0;
  if ((*err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, PAIR_SMEM_MAX)) != cudaSuccess ||
      (*err = cudaGetDevice(&dev)) != cudaSuccess ||
      (*err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (*err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, PTPB, p.smem)) != cudaSuccess)
    return 0;
  return sms * (per_sm > 0 ? per_sm : 1);
}

void pair_launch(const PairParams& p, long long n_tiles, int grid, cudaStream_t s) {
  const long long g = n_tiles < grid ? n_tiles : grid;
  pair_kernel(p)<<<(unsigned)g, PTPB, p.smem, s>>>(p, n_tiles);
}

}  // namespace tnq
