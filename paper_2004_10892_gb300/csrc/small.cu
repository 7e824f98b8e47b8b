// small.cu -- k_small: every bucket of a small plan in one launch (small.cuh).
//
// A plan of 2^4 to 2^18-entry buckets is bound by latency: as separate
// launches (one per level and per larger bucket) it waits for each launch and
// for its chain of dependent loads. Here one block runs the levels of few
// entries with its tensors in shared memory, one __syncthreads per level, and
// a cluster shares the wide levels through global memory (L2), one cluster
// barrier per level. Every item recomputes what does not depend on it: that
// costs no latency.
//
// GB300, a whole call from the host, before (a captured graph, or direct
// launches in the allocation-free call) and now: 4x4 depth 16 amplitude 141 ->
// 54 us; 5x5 depth 20 without allocations 305 -> 105 us; 16 slices of 6x6 depth
// 24 (6.3e7 flops) 277 -> 148 us; a 6x6 network of three-valued indices 379 ->
// 287 us. What is left: about 1600 cycles for a level of one entry (index
// arithmetic, dependent loads, the barrier), and for levels of 2^16 entries
// and more the 64 bytes a cycle that each of the cluster's SMs gets from L2.
#include <cooperative_groups.h>

#include "device_util.cuh"
#include "small.cuh"

namespace cg = cooperative_groups;

namespace tnq {

constexpr int SMALL_ALL = 9;  // variables of a result from which all threads work on one bucket at a time

// Bits of x under the mask, moved together (Warren, Hacker's Delight, 7-4).
__device__ __forceinline__ unsigned compress(unsigned x, const SmallIn& in) {
  x &= in.mask;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const unsigned t = x & in.mv[i];
    x = (x ^ t) | (t >> (1 << i));
  }
  return x;
}

__device__ __forceinline__ float part_max(float2 r) {  // (0 for NaN, as fmaxf against a number gives)
  return fmaxf(fmaxf(fabsf(r.x), fabsf(r.y)), 0.f);
}

// sum over u of p_u v_u as k_group takes it
__device__ __forceinline__ float2 sum_products(float2 p0, float2 p1, float2 v0, float2 v1) {
  float x = __fmul_rn(p0.x, v0.x), y = __fmul_rn(p0.x, v0.y);
  x = fmaf(-p0.y, v0.y, x);
  y = fmaf(p0.y, v0.x, y);
  x = fmaf(p1.x, v1.x, x);
  y = fmaf(p1.x, v1.y, y);
  return make_float2(fmaf(-p1.y, v1.y, x), fmaf(p1.y, v1.x, y));
}

// One bucket by all threads (t0 of step, a power of two): its inputs looked up
// once, N entries in flight per thread. Entries b + i step of one b that is
// aligned to N step differ in the bits of i alone, so their places in an input
// are the first one's plus the places of those bits. Returns the thread's
// largest part.
template <int NIN, int SPLIT>
__device__ __noinline__ float small_bucket(const SmallOp& op, const SmallIn* ins, float2* out, const float2* sh,
                                              const float2* glob, const unsigned* s_max, unsigned t0, unsigned step) {
  constexpr int N = NIN <= 3 ? 4 : (NIN <= 5 ? 2 : 1);
  const float2* base[NIN];
  float f[NIN];
#pragma unroll
  for (int j = 0; j < NIN; ++j) {
    const SmallIn& in = ins[op.in0 + j];
    base[j] = in.off & SMALL_SHARED ? sh + (in.off & ~SMALL_SHARED) : glob + in.off;
    int m;
    f[j] = in.meta < 0 ? 1.f : scale_of_max(s_max[in.meta], &m);
  }
  const unsigned n = 1u << op.bits;
  const int sh2 = op.sum;  // an input's entries are pairs over the eliminated variable, or single
  float mx = 0.f;
  auto product = [&](const float4* v) {
    float2 a0 = make_float2(v[0].x * f[0], v[0].y * f[0]), a1 = make_float2(v[0].z * f[0], v[0].w * f[0]);
    float2 p0 = make_float2(1.f, 0.f), p1 = p0;
#pragma unroll
    for (int j = 1; j < NIN; ++j) {
      const float2 w0 = make_float2(v[j].x * f[j], v[j].y * f[j]), w1 = make_float2(v[j].z * f[j], v[j].w * f[j]);
      if (!SPLIT || j < SPLIT) {
        a0 = cmul(a0, w0);
        a1 = cmul(a1, w1);
      } else {
        p0 = j == SPLIT ? w0 : cmul(p0, w0);
        p1 = j == SPLIT ? w1 : cmul(p1, w1);
      }
    }
    if (SPLIT) return sum_products(p0, p1, a0, a1);
    return op.sum ? make_float2(a0.x + a1.x, a0.y + a1.y) : a0;
  };
  auto load = [&](int j, unsigned c) {
    if (op.sum) return *reinterpret_cast<const float4*>(base[j] + c);
    const float2 w = base[j][c];
    return make_float4(w.x, w.y, 0.f, 0.f);
  };
  if (n >= N * step) {
    unsigned d1[NIN], d2[NIN];
#pragma unroll
    for (int j = 0; j < NIN; ++j) {
      d1[j] = N > 1 ? compress(step, ins[op.in0 + j]) << sh2 : 0u;
      d2[j] = N > 2 ? compress(2 * step, ins[op.in0 + j]) << sh2 : 0u;
    }
    for (unsigned b = t0; b < n; b += N * step) {
      float4 v[N][NIN];
#pragma unroll
      for (int j = 0; j < NIN; ++j) {
        const unsigned c = compress(b, ins[op.in0 + j]) << sh2;
#pragma unroll
        for (int i = 0; i < N; ++i) v[i][j] = load(j, c + ((i & 1) ? d1[j] : 0u) + ((i & 2) ? d2[j] : 0u));
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const float2 r = product(v[i]);
        out[b + i * step] = r;
        mx = fmaxf(mx, part_max(r));
      }
    }
  } else {
    for (unsigned b = t0; b < n; b += step) {
      float4 v[NIN];
#pragma unroll
      for (int j = 0; j < NIN; ++j) v[j] = load(j, compress(b, ins[op.in0 + j]) << sh2);
      const float2 r = product(v);
      out[b] = r;
      mx = fmaxf(mx, part_max(r));
    }
  }
  return mx;
}

constexpr int SMALL_IN = 4;  // inputs of a prepared entry

// One thread's entry of a level of small buckets: what does not depend on the
// level's inputs, so that it is looked up before the barrier. Absent inputs
// are the pair (1, 1); further ones (and buckets that do not sum) are looked
// up late.
struct SmallEntry {
  int op, out, grp;                  // op < 0: none
  int own;                           // inputs of the first product (SmallOp::split; all without one)
  int more;                          // first input that is not prepared (the number of inputs: none)
  int src[SMALL_IN], meta[SMALL_IN];  // tensor offset of the entry in each input, its bucket
};

__global__ void __launch_bounds__(STPB, 1) k_small(const __grid_constant__ SmallArgs A) {
  extern __shared__ float4 sm4[];
  __shared__ double2 s_scal;
  __shared__ int s_exp;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), size = (int)cluster.num_blocks();
  const int item = (int)(blockIdx.x / size), t = threadIdx.x, lane = t & 31;
  auto up = [](int bytes) { return (bytes + 15) / 16; };
  const int q_ins = up(A.n_ins * (int)sizeof(SmallIn)), q_leaf = up(A.n_small * (int)sizeof(SmallLeaf)),
            q_lev = up(A.n_levels * (int)sizeof(SmallLevel)), q_ops = up(A.n_ops * (int)sizeof(SmallOp));
  float4* tables = sm4;
  const SmallIn* ins = reinterpret_cast<const SmallIn*>(tables);
  const SmallLeaf* small = reinterpret_cast<const SmallLeaf*>(tables + q_ins);
  const SmallLevel* levels = reinterpret_cast<const SmallLevel*>(tables + q_ins + q_leaf);
  const SmallOp* ops = reinterpret_cast<const SmallOp*>(tables + q_ins + q_leaf + q_lev);
  float2* sh = reinterpret_cast<float2*>(tables + q_ins + q_leaf + q_lev + q_ops);
  unsigned* s_max0 = reinterpret_cast<unsigned*>(sh + A.smem_elems + 2);  // the first block's serve the whole cluster
  unsigned* s_max = size > 1 ? cluster.map_shared_rank(s_max0, 0) : s_max0;
  float2* glob = A.arena + (long long)item * A.arena_elems;
  auto at = [&](int off) { return off & SMALL_SHARED ? sh + (off & ~SMALL_SHARED) : glob + off; };
#pragma unroll 8
  for (int i = t; i < q_ins + q_leaf + q_lev + q_ops; i += STPB) tables[i] = __ldg(A.tables + i);
  for (int i = t; i < A.n_ops; i += STPB) s_max0[i] = 0u;
  if (t == 0) {
    s_exp = A.scale_exp;
    s_max0[A.n_ops] = 0x3f000000u;  // of an absent input: scale 1, and the pair (1, 1)
    sh[A.smem_elems] = sh[A.smem_elems + 1] = make_float2(1.f, 0.f);
  }

  // the item's fixed values
  const unsigned long long gi = A.item_base + (unsigned long long)item;
  const unsigned long long slice = A.mode == 0 ? gi : (A.p ? gi & ((1ull << A.p) - 1ull) : 0ull);
  const int brow = A.mode == 0 ? 0 : (int)((gi >> A.p) - A.bstr_base);
  auto bit = [&](int q) -> int {
    const unsigned w = A.bits ? __ldg(A.bits + (size_t)brow * A.n_words + (q >> 5)) : A.words[q >> 5];
    return (int)((w >> (q & 31)) & 1u);
  };
  auto fixed_part = [&](const LeafDev& L) -> int {
    int a = 0;
    for (int x = 0; x < L.nv; ++x) {
      if (L.vkind[x] == 2) a |= bit(L.varg[x]) << x;
      else if (L.vkind[x] == 3) a |= (int)((slice >> L.varg[x]) & 1ull) << x;
    }
    return a;
  };
  __syncthreads();
  // gate tensors restricted to the item's values (Eq. 4)
  if (rank == 0) {
    for (int i = t; i < 4 * A.n_small; i += STPB) {  // four threads each
      const SmallLeaf& L = small[i >> 2];
      float2* out = at(L.off);
      for (int e = i & 3; e < (1 << L.n_free); e += 4) {
        int a = 0;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int k = L.kind[x], g = L.arg[x];
          if (k == 0) a |= ((e >> g) & 1) << x;
          else if (k == 2) a |= bit(g) << x;
          else if (k == 3) a |= (int)((slice >> g) & 1ull) << x;
        }
        out[e] = L.val[a];
      }
    }
  }
  for (int l = t >> 5; l < A.n_leaves; l += STPB / 32) {  // a warp each, by the cluster's blocks in turn
    const LeafDev& L = A.leaves[l];
    const int off = (int)L.off, nv = L.nv, n = 1 << L.n_free;
    if ((off & SMALL_SHARED ? 0 : l % size) != rank) continue;
    float2* out = at(off);
    const int a0 = fixed_part(L);
    for (int e = lane; e < n; e += 32) {
      int a = a0;
      for (int x = 0; x < nv; ++x)
        if (L.vkind[x] == 0) a |= ((e >> L.varg[x]) & 1) << x;
      out[e] = __ldg(A.vals + L.tab + a);
    }
  }
  // product of the fully fixed gate tensors and the wires without a gate (FP64, lanes in turn, then a tree)
  if (rank == 0 && t >= STPB - 32) {
    double re = 1.0, im = 0.0;
    auto times = [&](double x, double y) {
      const double r = re * x - im * y;
      im = re * y + im * x;
      re = r;
    };
    for (int i = lane; i < A.n_scalars; i += 32) {
      const LeafDev& L = A.scalars[i];
      const float2 v = leaf_entry(L, A.vals, fixed_part(L));
      times(v.x, v.y);
    }
    for (int i = lane; i < A.n_inout; i += 32)
      if (bit(A.inout[i])) re = im = 0.0;
    for (int off = 16; off > 0; off >>= 1) {
      const double x = __shfl_down_sync(0xffffffffu, re, off), y = __shfl_down_sync(0xffffffffu, im, off);
      times(x, y);
    }
    if (lane == 0) s_scal = make_double2(re, im);
  }
  if (size > 1) cluster.sync();
  else __syncthreads();

  // the level's buckets of 2^SMALL_ALL and more entries, one after the other,
  // by threads t0 of step; returns the first bucket after them
  auto large_buckets = [&](const SmallLevel& V, unsigned* maxima, int t0, int step) {
    int o = V.op0;
    for (; o < V.op0 + V.nop && ops[o].bits >= SMALL_ALL; ++o) {
      const SmallOp op = ops[o];
      float2* out = at(op.out);
      float mx;
#define SMALL_RUN(n)                                                                       \
  mx = op.split == 0   ? small_bucket<n, 0>(op, ins, out, sh, glob, maxima, t0, step)      \
       : op.split == 1 ? small_bucket<n, 1>(op, ins, out, sh, glob, maxima, t0, step)      \
                       : small_bucket<n, n == 1 ? 1 : 2>(op, ins, out, sh, glob, maxima, t0, step); \
  break
      switch (op.nin) {
        case 1: SMALL_RUN(1);
        case 2: SMALL_RUN(2);
        case 3: SMALL_RUN(3);
        case 4: SMALL_RUN(4);
        case 5: SMALL_RUN(5);
        case 6: SMALL_RUN(6);
        case 7: SMALL_RUN(7);
        default: SMALL_RUN(8);
      }
#undef SMALL_RUN
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0 && m) atomicMax(&maxima[o], m);
    }
    return o;
  };
  auto prepare = [&](int op0, int end, int e) {
    SmallEntry E;
    E.op = -1;
    E.out = 0;
    E.grp = 1;
    E.own = KMAX;
    E.more = KMAX;
#pragma unroll
    for (int j = 0; j < SMALL_IN; ++j) {
      E.src[j] = A.smem_elems | SMALL_SHARED;
      E.meta[j] = A.n_ops;
    }
    if (op0 == end || e >= ops[end - 1].first + (1 << ops[end - 1].bits)) return E;
    int lo = op0, hi = end - 1;  // the last bucket that starts at or before e
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (ops[mid].first <= e) lo = mid;
      else hi = mid - 1;
    }
    const SmallOp op = ops[lo];
    const unsigned b = (unsigned)(e - op.first);
    E.op = lo;
    E.out = op.out + (int)b;
    E.grp = 1 << min(op.bits, 5);
    E.own = op.split ? op.split : KMAX;
    E.more = op.sum ? SMALL_IN : 0;
#pragma unroll
    for (int j = 0; j < SMALL_IN; ++j)
      if (j < op.nin && op.sum) {
        const SmallIn& in = ins[op.in0 + j];
        E.src[j] = in.off + (int)(compress(b, in) << 1);
        E.meta[j] = in.meta < 0 ? A.n_ops : in.meta;
      }
    return E;
  };
  auto finish = [&](const SmallEntry& E, unsigned* maxima) {
    if (!__any_sync(0xffffffffu, E.op >= 0)) return;  // (sixteen idle warps' instructions would be the level's time)
    float4 v[SMALL_IN];
    float f[SMALL_IN];
#pragma unroll
    for (int j = 0; j < SMALL_IN; ++j) {
      v[j] = *reinterpret_cast<const float4*>(at(E.src[j]));
      int m;
      f[j] = scale_of_max(maxima[E.meta[j]], &m);
    }
    float2 a0 = make_float2(v[0].x * f[0], v[0].y * f[0]), a1 = make_float2(v[0].z * f[0], v[0].w * f[0]);
    const bool split = __any_sync(0xffffffffu, E.own < KMAX);  // (chains' buckets are mostly larger)
    float2 p0 = make_float2(1.f, 0.f), p1 = p0;
    auto times = [&](int j, float2 w0, float2 w1) {
      if (!split || j < E.own) {
        a0 = cmul(a0, w0);
        a1 = cmul(a1, w1);
      } else {
        p0 = cmul(p0, w0);
        p1 = cmul(p1, w1);
      }
    };
#pragma unroll
    for (int j = 1; j < SMALL_IN; ++j)
      times(j, make_float2(v[j].x * f[j], v[j].y * f[j]), make_float2(v[j].z * f[j], v[j].w * f[j]));
    float mx = 0.f;
    if (E.op >= 0) {
      const SmallOp op = ops[E.op];
#pragma unroll 1
      for (int j = E.more; j < op.nin; ++j) {
        const SmallIn& in = ins[op.in0 + j];
        const float2* p = at(in.off) + (compress((unsigned)(E.out - op.out), in) << op.sum);
        int m;
        const float g = in.meta < 0 ? 1.f : scale_of_max(maxima[in.meta], &m);
        times(j, make_float2(p[0].x * g, p[0].y * g), op.sum ? make_float2(p[1].x * g, p[1].y * g) : p1);
      }
      float2 r = op.sum ? make_float2(a0.x + a1.x, a0.y + a1.y) : a0;
      if (split && op.split) r = sum_products(p0, p1, a0, a1);
      *at(E.out) = r;
      mx = part_max(r);
    }
    // buckets of a level are laid out by falling size, so their entries are aligned lane groups
    unsigned m = __float_as_uint(mx);
    if (__all_sync(0xffffffffu, E.op >= 0 && E.grp == 32)) {
      m = __reduce_max_sync(0xffffffffu, m);
    } else {
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned x = __shfl_xor_sync(0xffffffffu, m, off);
        if (off < E.grp) m = max(m, x);
      }
    }
    if (E.op >= 0 && (lane & (E.grp - 1)) == 0 && m) atomicMax(&maxima[E.op], m);
  };
  for (int l = 0; l < A.n_levels;) {
    if (levels[l].wide) {
      const SmallLevel V = levels[l];
      const int end = V.op0 + V.nop, o = large_buckets(V, s_max, rank * STPB + t, size * STPB);
      if (o < end)
        for (int e = ops[o].first + rank * STPB + t; e - lane < V.entries; e += size * STPB)
          finish(prepare(o, end, e), s_max);
      ++l;
    } else if (rank == 0) {
      // one thread's first entry of the next level is prepared before the barrier
      auto first_small = [&](const SmallLevel& V) {
        int o = V.op0;
        while (o < V.op0 + V.nop && ops[o].bits >= SMALL_ALL) ++o;
        return o;
      };
      SmallLevel V = levels[l];
      int o = first_small(V);
      SmallEntry E = prepare(o, V.op0 + V.nop, (o < V.op0 + V.nop ? ops[o].first : 0) + t);
      while (true) {
        const int end = V.op0 + V.nop;
        if (o > V.op0) large_buckets(V, s_max0, t, STPB);
        if (o < end) {
          finish(E, s_max0);
          for (int e = ops[o].first + STPB + t; e - lane < V.entries; e += STPB) finish(prepare(o, end, e), s_max0);
        }
        ++l;
        const bool more = l < A.n_levels && !levels[l].wide;
        if (more) {
          V = levels[l];
          o = first_small(V);
          E = prepare(o, V.op0 + V.nop, (o < V.op0 + V.nop ? ops[o].first : 0) + t);
        }
        __syncthreads();
        if (!more) break;
      }
    } else {
      while (l < A.n_levels && !levels[l].wide) ++l;
    }
    if (size > 1) cluster.sync();
    else __syncthreads();
  }
  if (rank != 0) return;
  // the value's exponent: every bucket is the input of one other (or final),
  // so it is the sum of all the shifts that the scales took out
  int shifts = 0;
  for (int i = t; i < A.n_ins; i += STPB) {
    int m = 0;
    if (ins[i].meta >= 0) scale_of_max(s_max0[ins[i].meta], &m);
    shifts += m;
  }
  shifts = __reduce_add_sync(0xffffffffu, shifts);
  if (lane == 0 && shifts) atomicAdd(&s_exp, shifts);
  __syncthreads();
  if (t == 0) {
    double re = s_scal.x, im = s_scal.y;
    for (int i = 0; i < A.n_finals; ++i) {
      const float2 v = *at(A.finals[i].x);
      const double r = re * v.x - im * v.y;
      im = re * v.y + im * v.x;
      re = r;
    }
    if (A.scale_half) {
      re *= 0.70710678118654752440;
      im *= 0.70710678118654752440;
    }
    A.res[item] = make_double2(ldexp(re, s_exp), ldexp(im, s_exp));
  }
}

static void small_config(const SmallArgs& a, int blocks, int cluster, cudaLaunchConfig_t* c, cudaLaunchAttribute* at) {
  *c = {};
  c->gridDim = dim3((unsigned)blocks);
  c->blockDim = dim3(STPB);
  c->dynamicSmemBytes = small_smem(a);
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)cluster;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  c->attrs = at;
  c->numAttrs = 1;
}

cudaError_t small_resident(const SmallArgs& a, int cluster, int* clusters) {
  cudaError_t e = cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM_MAX);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t c;
  cudaLaunchAttribute at;
  small_config(a, cluster, cluster, &c, &at);
  return cudaOccupancyMaxActiveClusters(clusters, k_small, &c);
}

cudaError_t small_launch(const SmallArgs& a, int n_items, int cluster, cudaStream_t s) {
  cudaLaunchConfig_t c;
  cudaLaunchAttribute at;
  small_config(a, n_items * cluster, cluster, &c, &at);
  c.stream = s;
  return cudaLaunchKernelEx(&c, k_small, a);
}

}  // namespace tnq
