// pair.cu -- k_pair: a fused chain of buckets as a register-tiled contraction
// (see pair.cuh).
#include "device_util.cuh"
#include "pair.cuh"

namespace tnq {

// Fold table entry e of one operand: the product of its small tensors at u_0 =
// 0 and 1, starting from (f, 0).
__device__ __forceinline__ float4 fold_entry(const PFold& F, int e, const float2* const* s_ptr, float f) {
  float2 p0 = make_float2(f, 0.f), p1 = p0;
  for (int j = 0; j < F.n; ++j) {
    int o = 0;
#pragma unroll
    for (int i = 0; i < PF_MAX; ++i)
      if (i < F.nf && ((e >> i) & 1)) o += F.fs[j][i];
    const float2* q = s_ptr[F.gin[j]] + o;
    p0 = cmul(p0, __ldg(q));
    p1 = cmul(p1, __ldg(q + F.ustride[j]));
  }
  return make_float4(p0.x, p0.y, p1.x, p1.y);
}

// Persistent: a block loops over tiles (item, tile variables). Per tile the
// block stages its part of A, B (and C) in shared memory once, A and B
// multiplied by the fold tables on the way, then every thread computes a 4 x 4
// register tile: per pair of summed values 4 + 4 16-byte shared loads feed 128
// FMAs.
template <int NKX, int NKY, bool HASC>
__global__ void __launch_bounds__(PTPB, 2) k_pair(const __grid_constant__ PairParams P, long long n_tiles) {
  extern __shared__ float4 sm[];
  __shared__ float4 s_fa[1 << PF_MAX], s_fb[1 << PF_MAX];
  __shared__ int4 s_it[3][1 << (PE_MAX - PTB)];  // staging iteration: global offset, slot, fold index
  __shared__ int s_hstr[PIN_MAX][PH_MAX];
  __shared__ const float2* s_ptr[PIN_MAX];
  __shared__ long long s_out;
  __shared__ float s_sc[PIN_MAX];
  __shared__ int s_e[PIN_MAX];
  __shared__ float s_red[PTPB / 32];
  constexpr int N = 1 << PR;
  const int t = threadIdx.x;
  for (int e = t; e < PIN_MAX * PH_MAX; e += PTPB) {
    const int j = e / PH_MAX, i = e - j * PH_MAX;
    s_hstr[j][i] = (i < P.n_h && j < P.n_gin) ? P.gin[j].hstride[i] : 0;
  }
  const POp* ops[3] = {&P.a, &P.b, &P.c};
  int tg[3], td[3], tf[3];  // this thread's part of the staging offsets
#pragma unroll
  for (int o = 0; o < (HASC ? 3 : 2); ++o) {
    const POp& O = *ops[o];
    tg[o] = tf[o] = 0;
    td[o] = O.base;
#pragma unroll
    for (int i = 0; i < PTB; ++i)
      if (i < O.ebits && ((t >> i) & 1)) {
        tg[o] += O.g[i];
        td[o] += O.d[i];
        tf[o] += O.f[i];
      }
    const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
    if (t < nit) {
      int4 v = make_int4(0, 0, 0, 0);
      for (int i = PTB; i < O.ebits; ++i)
        if ((t >> (i - PTB)) & 1) {
          v.x += O.g[i];
          v.y += O.d[i];
          v.z += O.f[i];
        }
      s_it[o][t] = v;
    }
  }
  int ra = P.a.base, rb = P.b.base, rc = P.c.base, ro = 0;  // this thread's register tile
#pragma unroll
  for (int i = 0; i < PTB; ++i)
    if ((t >> i) & 1) {
      ra += P.ta[i];
      rb += P.tb[i];
      rc += P.tc[i];
      ro += P.to[i];
    }
  int pa[N], pb[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    pa[i] = ra + ((i & 1) ? P.xa[0] : 0) + ((i & 2) ? P.xa[1] : 0);
    pb[i] = rb + ((i & 1) ? P.yb[0] : 0) + ((i & 2) ? P.yb[1] : 0);
  }
  const bool fold_a = P.fa.n > 0;
  const bool fold_inv = P.fa.inv && P.fb.inv;
  long long cur_item = -1;
  float tmax = 0.f;
  auto flush = [&](long long item) {
    float m = tmax;
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    __syncthreads();
    if ((t & 31) == 0) s_red[t >> 5] = m;
    __syncthreads();
    if (t == 0) {
      float b = 0.f;
      for (int w = 0; w < PTPB / 32; ++w) b = fmaxf(b, s_red[w]);
      if (b > 0.f) atomic_max_pos(&P.meta_m[(long long)P.out_meta * P.B + (P.out_dep ? item : 0ll)], b);
    }
  };
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const long long item = tile >> P.n_h;
    const long long h = tile & ((1ll << P.n_h) - 1ll);
    const bool new_item = item != cur_item;
    if (new_item) {
      if (cur_item >= 0) flush(cur_item);
      tmax = 0.f;
      cur_item = item;
    }
    __syncthreads();  // the previous tile is done with the staged operands
    for (int j = t >> 5; j <= P.n_gin; j += PTPB / 32) {
      const int lane = t & 31;
      if (j < P.n_gin) {
        const int v = __reduce_add_sync(0xffffffffu, ((h >> lane) & 1ll) ? s_hstr[j][lane] : 0);
        if (lane == 0) s_ptr[j] = P.gin[j].ptr + (P.gin[j].dep ? item * P.gin[j].istride : 0ll) + v;
      } else if (lane == 0) {
        long long v = P.out_dep ? item * P.out_istride : 0ll;
        for (int i = 0; i < P.n_h; ++i)
          if ((h >> i) & 1ll) v += P.out_hstride[i];
        s_out = v;
      }
    }
    if (new_item && t < P.n_gin) {
      const PIn& g = P.gin[t];
      int m = 0, e = 0;
      float f = 1.f;
      if (g.meta >= 0) {
        const long long row = (long long)g.meta * P.B + (g.dep ? item : 0ll);
        f = scale_of_max(P.meta_m[row], &m);
        e = P.meta_e[row] + m;
      }
      s_sc[t] = f;
      s_e[t] = e;
    }
    __syncthreads();
    if (new_item || !fold_inv) {  // small tensors and every input's power-of-two scale
      float f = 1.f;
      for (int j = 0; j < P.n_gin; ++j) f *= s_sc[j];
      if (t < (1 << P.fb.nf)) s_fb[t] = fold_entry(P.fb, t, s_ptr, f);
      if (fold_a && t < (1 << P.fa.nf)) s_fa[t] = fold_entry(P.fa, t, s_ptr, 1.f);
      __syncthreads();
    }
#pragma unroll
    for (int o = 0; o < (HASC ? 3 : 2); ++o) {
      const POp& O = *ops[o];
      const float2* src = s_ptr[O.gin] + tg[o];
      const float4* ft = (o == 0 ? s_fa : s_fb) + tf[o];
      const bool fold = o == 1 || (o == 0 && fold_a);
      const int nit = O.ebits > PTB ? 1 << (O.ebits - PTB) : 1;
      if (O.ebits < PTB && t >= (1 << O.ebits)) continue;
#pragma unroll 4
      for (int it = 0; it < nit; ++it) {
        const int4 k = s_it[o][it];
        float4 v = __ldg(reinterpret_cast<const float4*>(src + k.x));
        if (fold) {
          const float4 f = ft[k.z];
          const float2 v0 = cmul(make_float2(v.x, v.y), make_float2(f.x, f.y));
          const float2 v1 = cmul(make_float2(v.z, v.w), make_float2(f.z, f.w));
          v = make_float4(v0.x, v0.y, v1.x, v1.y);
        }
        sm[td[o] + k.y] = v;
      }
    }
    __syncthreads();
    constexpr int XO = N >> NKX, YO = N >> NKY;
    float2 acc[XO][YO];
#pragma unroll
    for (int i = 0; i < XO; ++i)
#pragma unroll
      for (int j = 0; j < YO; ++j) acc[i][j] = make_float2(0.f, 0.f);
    const int n1 = 1 << P.n1, n2 = HASC ? 1 << P.n2 : 1;
    for (int q2 = 0; q2 < n2; ++q2) {
      int oa = 0, ob = 0, oc = 0;
      if (HASC)
        for (int i = 0; i < P.n2; ++i)
          if ((q2 >> i) & 1) {
            oa += P.k2a[i];
            ob += P.k2b[i];
            oc += P.k2c[i];
          }
      float2 x[N][N];
#pragma unroll
      for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < N; ++j) x[i][j] = make_float2(0.f, 0.f);
      for (int q = 0; q < n1; ++q) {
        int ka = oa, kb = ob;
        for (int i = 0; i < P.n1; ++i)
          if ((q >> i) & 1) {
            ka += P.k1a[i];
            kb += P.k1b[i];
          }
        float4 va[N], vb[N];
#pragma unroll
        for (int i = 0; i < N; ++i) va[i] = sm[pa[i] + ka];
#pragma unroll
        for (int j = 0; j < N; ++j) vb[j] = sm[pb[j] + kb];
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
          for (int j = 0; j < N; ++j) {
            float2 r = x[i][j];
            r.x = fmaf(va[i].x, vb[j].x, r.x);
            r.y = fmaf(va[i].x, vb[j].y, r.y);
            r.x = fmaf(-va[i].y, vb[j].y, r.x);
            r.y = fmaf(va[i].y, vb[j].x, r.y);
            r.x = fmaf(va[i].z, vb[j].z, r.x);
            r.y = fmaf(va[i].z, vb[j].w, r.y);
            r.x = fmaf(-va[i].w, vb[j].w, r.x);
            r.y = fmaf(va[i].w, vb[j].z, r.y);
            x[i][j] = r;
          }
      }
      if constexpr (HASC) {  // times C, summed over the K2 register bits (C's bit 0 is B's register bit 0)
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
          for (int j = 0; j < N; j += 2) {
            const float4 c = sm[rc + oc + ((i & 1) ? P.xc[0] : 0) + ((i & 2) ? P.xc[1] : 0) + ((j & 2) ? P.yc[1] : 0)];
            float2 r = acc[i >> NKX][j >> NKY];
            const float2 u = x[i][j], w = x[i][j + 1];
            r.x = fmaf(u.x, c.x, r.x);
            r.y = fmaf(u.x, c.y, r.y);
            r.x = fmaf(-u.y, c.y, r.x);
            r.y = fmaf(u.y, c.x, r.y);
            r.x = fmaf(w.x, c.z, r.x);
            r.y = fmaf(w.x, c.w, r.y);
            r.x = fmaf(-w.y, c.w, r.x);
            r.y = fmaf(w.y, c.z, r.y);
            acc[i >> NKX][j >> NKY] = r;
          }
      } else {
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
          for (int j = 0; j < N; ++j) acc[i][j] = x[i][j];
      }
    }
    float2* dst = P.out + s_out + ro;
#pragma unroll
    for (int i = 0; i < XO; ++i)
#pragma unroll
      for (int j = 0; j < YO; ++j) {
        const int ri = i << NKX, rj = j << NKY;
        const int o = ((ri & 1) ? P.xo[0] : 0) + ((ri & 2) ? P.xo[1] : 0) + ((rj & 1) ? P.yo[0] : 0) +
                      ((rj & 2) ? P.yo[1] : 0);
        dst[o] = acc[i][j];
        tmax = fmaxf(tmax, fmaxf(fabsf(acc[i][j].x), fabsf(acc[i][j].y)));
      }
    if (h == 0 && t == 0) {
      int e = 0;
      for (int j = 0; j < P.n_gin; ++j) e += s_e[j];
      P.meta_e[(long long)P.out_meta * P.B + (P.out_dep ? item : 0ll)] = e;
    }
  }
  if (cur_item >= 0) flush(cur_item);
}

using PairKernel = void (*)(PairParams, long long);
static PairKernel pair_kernel(const PairParams& p) {
  if (p.c.gin < 0) return k_pair<0, 0, false>;
  switch (p.nkx * 4 + p.nky) {
    case 1: return k_pair<0, 1, true>;
    case 2: return k_pair<0, 2, true>;
    case 5: return k_pair<1, 1, true>;
    case 6: return k_pair<1, 2, true>;
    case 9: return k_pair<2, 1, true>;
    default: return k_pair<2, 2, true>;
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
