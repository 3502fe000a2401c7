// Applies of the elastic trace operator from symmetric packed copies of S_K, one warp per element.
//
// The blocks (m_e up to 180) are too large for the registers of one lane, and their bytes bound every
// apply. So only the blocks on and above the diagonal are stored: S_K is cut into 16 x 16 units, unit
// (I, J >= I) at I nb - I (I - 1) / 2 + J - I of the element's nb (nb + 1) / 2, the diagonal ones whole
// and zero beyond m_e. Lane l of a unit holds column 16 J + (l & 15), rows 16 I + 8 (l >> 4) + 0..7: a
// 16-byte load brings eight FP16 entries (two bring eight FP32 entries) and a warp reads 512 contiguous
// bytes. An entry above the diagonal blocks is used twice: for its column (accumulators of the lane) and
// for its row (eight partial sums, added over the 16 lanes once per row of units).
#pragma once

#include "dflocal.cuh"
#include "elastic.cuh"

namespace hdg {

__host__ __device__ constexpr int sym_blocks(int m) { return (m + 15) / 16; }
__host__ __device__ constexpr int sym_units(int m) { return sym_blocks(m) * (sym_blocks(m) + 1) / 2; }

// Element sizes and the trace entry of a local one (-1: a boundary entry): per-element degrees
struct SymIdxVd {
  static constexpr int NB = 12;          // m_e <= 180
  const int64_t *p_off, *s_off;          // first unit, first FP64 entry of an element
  const int32_t *m_off, *gint;
  __device__ __forceinline__ int64_t m0(int64_t e) const { return m_off[e]; }
  __device__ __forceinline__ int m(int64_t e) const { return m_off[e + 1] - m_off[e]; }
  __device__ __forceinline__ int64_t unit0(int64_t e) const { return p_off[e]; }
  __device__ __forceinline__ int64_t s0(int64_t e) const { return s_off[e]; }
  __device__ __forceinline__ int64_t entry(int64_t, int64_t m0, int c) const { return gint[m0 + c]; }
};

// Uniform degree. The copies are used where their units hold fewer entries than the full block
// (degrees 2 and 3 on tetrahedra and 4 on triangles; the padding of smaller blocks outweighs the half saved).
__host__ __device__ constexpr bool sym_pays(int m) { return sym_units(m) * 256 < m * m; }
template <class L>
struct SymIdxUni {
  static constexpr int M = L::M, NB = sym_blocks(L::M);
  const int32_t *elem_face, *face_bnd;
  __device__ __forceinline__ int64_t m0(int64_t e) const { return e * M; }
  __device__ __forceinline__ int m(int64_t) const { return M; }
  __device__ __forceinline__ int64_t unit0(int64_t e) const { return e * sym_units(M); }
  __device__ __forceinline__ int64_t s0(int64_t e) const { return e * M * M; }
  __device__ __forceinline__ int64_t entry(int64_t e, int64_t, int c) const {
    const int f = elem_face[e * L::NFC + c / L::NF];
    return face_bnd[f] < 0 ? (int64_t)f * L::NF + c % L::NF : -1;
  }
};

// Sums of v[0..7] over the 16 lanes of a half-warp; lane l receives index l & 7
template <class T, class ADD>
__device__ __forceinline__ T sym_reduce8(T (&v)[8], ADD&& exch_add) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const bool b = (lane >> s) & 1;
#pragma unroll
    for (int j = 0; j < (4 >> s); ++j) {
      const T a = v[2 * j], c = v[2 * j + 1];
      v[j] = exch_add(b ? c : a, b ? a : c, 1 << s);
    }
  }
  return exch_add(v[0], v[0], 8);
}

// Kernel A of the two-kernel FP32 iteration (Cg2State): slot = S_K p_K with p_K formed in the gather.
// ST: float, or __half with one scale per element. What bounds it: the bytes of S_K. The units are one
// stream, and the next D of them are loaded before the products of the current D; the columns' sums stay in
// shared memory, so that the registers hold the loads in flight and 20 warps fit an SM.
// 24,576 tets of degrees 1..4, FP16: 0.21 ms (0.26 ms with the whole blocks, a row at a time).
template <class IX, class ST>
__global__ void __launch_bounds__(128, 5) sym_apply_two_kernel(int64_t ne, IX ix, const ST* __restrict__ S,
                                                               const float* __restrict__ sc, const float* __restrict__ z,
                                                               const float* __restrict__ p, float* __restrict__ slot,
                                                               Cg2Args o2) {
  constexpr int NB = IX::NB, VQ = sizeof(ST) / 2, D = 4 / VQ, NG = (NB + 1) / 2;
  __shared__ __align__(16) float lx[4][16 * NB];
  __shared__ float ys[4][16 * NB];   // row sums
  __shared__ float as[4][32 * NB];   // column sums of each lane
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cl = lane & 15, hl = lane >> 4;
  int64_t e = (int64_t)blockIdx.x * 4 + w, m0 = 0;
  int me = 0;
  float zr[NG], pr[NG];
  auto gather = [&] {
    if (e >= ne) return;
    m0 = ix.m0(e);
    me = ix.m(e);
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int c = 32 * q + lane;
      const int64_t t = c < me ? ix.entry(e, m0, c) : -1;
      zr[q] = t >= 0 ? z[t] : 0.f;
      pr[q] = t >= 0 ? p[t] : 0.f;
    }
  };
  gather();
  float beta;
  bool first;
  if (!cg2_begin_a<4>(o2, beta, first)) return;   // while the gather is in flight
  Acc2 pq;
  while (e < ne) {
    const int nb = sym_blocks(me), nu = nb * (nb + 1) / 2;
    const uint4* Se = reinterpret_cast<const uint4*>(S) + ix.unit0(e) * (32 * VQ) + lane;
    uint4 v[D][VQ];
    auto load = [&](int u0, uint4 (&d)[D][VQ]) {
#pragma unroll
      for (int j = 0; j < D; ++j)
#pragma unroll
        for (int h = 0; h < VQ; ++h)
          if (u0 + j < nu) d[j][h] = __ldg(Se + ((u0 + j) * VQ + h) * 32);
    };
    load(0, v);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NG; ++q)
      if (32 * q + lane < 16 * NB) lx[w][32 * q + lane] = cg2_dir(first, beta, pr[q], zr[q]);
    for (int J = 0; J < nb; ++J) as[w][32 * J + lane] = 0.f;
    __syncwarp();
    int I = 0, J = 0;
    float xr[8], ra[8];
    for (int u0 = 0; u0 < nu; u0 += D) {
      uint4 n[D][VQ];
      load(u0 + D, n);
#pragma unroll
      for (int j = 0; j < D; ++j) {
        if (u0 + j >= nu) break;
        if (J == I) {
          const float4 a = *reinterpret_cast<const float4*>(&lx[w][16 * I + 8 * hl]);
          const float4 b = *reinterpret_cast<const float4*>(&lx[w][16 * I + 8 * hl + 4]);
          xr[0] = a.x; xr[1] = a.y; xr[2] = a.z; xr[3] = a.w;
          xr[4] = b.x; xr[5] = b.y; xr[6] = b.z; xr[7] = b.w;
#pragma unroll
          for (int k = 0; k < 8; ++k) ra[k] = 0.f;
        }
        const float xc = J > I ? lx[w][16 * J + cl] : 0.f;
        float acc = as[w][32 * J + lane];
#pragma unroll
        for (int h = 0; h < VQ; ++h) {
          const unsigned q[4] = {v[j][h].x, v[j][h].y, v[j][h].z, v[j][h].w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if constexpr (VQ == 1) {
              const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&q[i]));
              acc = fmaf(f.x, xr[2 * i], acc);
              acc = fmaf(f.y, xr[2 * i + 1], acc);
              ra[2 * i] = fmaf(f.x, xc, ra[2 * i]);
              ra[2 * i + 1] = fmaf(f.y, xc, ra[2 * i + 1]);
            } else {
              const float f = __uint_as_float(q[i]);
              acc = fmaf(f, xr[4 * h + i], acc);
              ra[4 * h + i] = fmaf(f, xc, ra[4 * h + i]);
            }
          }
        }
        as[w][32 * J + lane] = acc;
        if (++J == nb) {
          const float yr = sym_reduce8(ra, [](float keep, float send, int o) { return keep + __shfl_xor_sync(0xffffffffu, send, o); });
          if ((lane & 8) == 0) ys[w][16 * I + 8 * hl + (lane & 7)] = yr;
          J = ++I;
        }
      }
#pragma unroll
      for (int j = 0; j < D; ++j)
#pragma unroll
        for (int h = 0; h < VQ; ++h) v[j][h] = n[j][h];
    }
    __syncwarp();
    const float scl = sc ? sc[e] : 1.f;
    for (int r = lane; r < me; r += 32) {
      const float* a = &as[w][32 * (r >> 4) + (r & 15)];
      const float y = scl * ((a[0] + a[16]) + ys[w][r]);
      slot[m0 + r] = y;
      pq.dot(lx[w][r], y);
    }
    e += (int64_t)gridDim.x * 4;
    gather();
  }
  cg2_end_a<4>(o2, pq);
}

// Refinement apply of the per-element degrees on the FP32 pipe: S_K = hi + lo (hi = fl32(S_K), lo =
// fl32(S_K - hi)), x in double-floats, compensated sums. Bounded by the bytes of the two copies; pipelined
// as above. 24,576 tets of degrees 1..4: 0.47 ms (0.72 to 1.47 ms, by the tile chosen, with the whole blocks).
// With one degree the residual comes from the FP64 blocks: this kernel was faster there (7,986 tets, k = 2: 57
// instead of 95 us), but a solve stalled at a residual of 1e-13 to 2e-13 |b| at alpha = 0.2 (48 to 384 tets, k = 2
// and 3; 4e-12 at alpha = 0.01), above the default tolerance, where FP64 reaches 1e-14 (1.6e-13).
template <class IX>
__global__ void __launch_bounds__(128, 4) sym_apply_df_kernel(int64_t ne, IX ix, const float* __restrict__ Shi,
                                                              const float* __restrict__ Slo, const double* __restrict__ x,
                                                              double* __restrict__ slot) {
  constexpr int NB = IX::NB, D = 2;
  __shared__ __align__(16) df2 lx[4][16 * NB];
  __shared__ df2 ys[4][16 * NB];
  __shared__ df2 as[4][32 * NB];   // column accumulators (sum, compensation)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cl = lane & 15, hl = lane >> 4;
  const int64_t e = (int64_t)blockIdx.x * 4 + w;
  if (e >= ne) return;
  const int64_t m0 = ix.m0(e), base = ix.unit0(e) * 64 + lane;
  const int me = ix.m(e), nb = sym_blocks(me), nu = nb * (nb + 1) / 2;
  const float4 *H = reinterpret_cast<const float4*>(Shi) + base, *L = reinterpret_cast<const float4*>(Slo) + base;
  float4 v[D][4];
  auto load = [&](int u0, float4 (&d)[D][4]) {
#pragma unroll
    for (int j = 0; j < D; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (u0 + j < nu) {
          d[j][h] = __ldg(H + ((u0 + j) * 2 + h) * 32);
          d[j][2 + h] = __ldg(L + ((u0 + j) * 2 + h) * 32);
        }
  };
  load(0, v);
  for (int c = lane; c < 16 * nb; c += 32) {   // zero from m_e to the end of the last block
    const int64_t t = c < me ? ix.entry(e, m0, c) : -1;
    lx[w][c] = t >= 0 ? dfl_from(x[t]) : df2{0.f, 0.f};
  }
  for (int J = 0; J < nb; ++J) as[w][32 * J + lane] = df2{0.f, 0.f};
  __syncwarp();
  auto exch = [](df2 keep, df2 send, int o) {
    return df_add(keep, df2{__shfl_xor_sync(0xffffffffu, send.h, o), __shfl_xor_sync(0xffffffffu, send.l, o)});
  };
  int I = 0, J = 0;
  DfAcc ra[8];
  for (int u0 = 0; u0 < nu; u0 += D) {
    float4 n[D][4];
    load(u0 + D, n);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      if (u0 + j >= nu) break;
      if (J == I)
#pragma unroll
        for (int k = 0; k < 8; ++k) ra[k] = DfAcc();
      const df2 xc = J > I ? lx[w][16 * J + cl] : df2{0.f, 0.f};
      const df2 a0 = as[w][32 * J + lane];
      DfAcc acc;
      acc.s = a0.h;
      acc.c = a0.l;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float sh[4] = {v[j][h].x, v[j][h].y, v[j][h].z, v[j][h].w};
        const float sl[4] = {v[j][2 + h].x, v[j][2 + h].y, v[j][2 + h].z, v[j][2 + h].w};
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
          const float4 xr = *reinterpret_cast<const float4*>(&lx[w][16 * I + 8 * hl + 4 * h + k]);
          acc.fma(df2{sh[k], sl[k]}, df2{xr.x, xr.y});
          acc.fma(df2{sh[k + 1], sl[k + 1]}, df2{xr.z, xr.w});
          ra[4 * h + k].fma(df2{sh[k], sl[k]}, xc);
          ra[4 * h + k + 1].fma(df2{sh[k + 1], sl[k + 1]}, xc);
        }
      }
      as[w][32 * J + lane] = df2{acc.s, acc.c};
      if (++J == nb) {
        df2 rv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) rv[k] = df_of(ra[k]);
        const df2 yr = sym_reduce8(rv, exch);
        if ((lane & 8) == 0) ys[w][16 * I + 8 * hl + (lane & 7)] = yr;
        J = ++I;
      }
    }
#pragma unroll
    for (int j = 0; j < D; ++j)
#pragma unroll
      for (int h = 0; h < 4; ++h) v[j][h] = n[j][h];
  }
  __syncwarp();
  for (int r = lane; r < me; r += 32) {
    const df2 *a = &as[w][32 * (r >> 4) + (r & 15)], b = df_two_sum(a[0].h, a[0].l), c = df_two_sum(a[16].h, a[16].l);
    slot[m0 + r] = dfl_to(df_add(df_add(b, c), ys[w][r]));
  }
}

// The packed copies of every S_K (row-major FP64): hi; the remainder, where lo is given; and with S16 the FP16
// copy with one scale per element (max |S_K| rounded up, so that every stored value lies in [-1, 1]). An FP16 entry
// is the FP32 quotient of hi and the scale, rounded: at most 2^-23 of it beside the 2^-11 of the rounding. CTA
// per element.
template <class IX>
__global__ void __launch_bounds__(256) sym_pack_kernel(int64_t ne, IX ix, const double* __restrict__ S, float4* __restrict__ hi,
                                                       float4* __restrict__ lo, uint4* __restrict__ S16,
                                                       float* __restrict__ sc16) {
  __shared__ long long red[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cl = lane & 15, hl = lane >> 4;
  for (int64_t e = blockIdx.x; e < ne; e += gridDim.x) {
    const int me = ix.m(e), nb = sym_blocks(me), nu = nb * (nb + 1) / 2;
    const double* Se = S + ix.s0(e);
    float scale = 1.f;
    if (S16) {
      long long m = 0;   // |S| ordered as integers
      for (int t = threadIdx.x; t < me * me; t += 256) m = max(m, __double_as_longlong(Se[t]) & 0x7fffffffffffffffll);
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) red[w] = m;
      __syncthreads();
      for (int i = 0; i < 8; ++i) m = max(m, red[i]);
      __syncthreads();
      if (m > 0) scale = __double2float_ru(__longlong_as_double(m));
      if (threadIdx.x == 0) sc16[e] = scale;
    }
    for (int u = w; u < nu; u += 8) {
      int I = 0, J = u;
      while (J >= nb - I) { J -= nb - I; ++I; }
      J += I;
      const int c = 16 * J + cl;
      float h[8], l[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = 16 * I + 8 * hl + k;
        split_f64(r < me && c < me ? Se[(int64_t)r * me + c] : 0.0, h[k], l[k]);
      }
      const int64_t o = (ix.unit0(e) + u) * 64 + lane;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        hi[o + 32 * q] = make_float4(h[4 * q], h[4 * q + 1], h[4 * q + 2], h[4 * q + 3]);
        if (lo) lo[o + 32 * q] = make_float4(l[4 * q], l[4 * q + 1], l[4 * q + 2], l[4 * q + 3]);
      }
      if (S16) {
        unsigned p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __half2 v = __floats2half2_rn(h[2 * i] / scale, h[2 * i + 1] / scale);
          p[i] = *reinterpret_cast<const unsigned*>(&v);
        }
        S16[(ix.unit0(e) + u) * 32 + lane] = make_uint4(p[0], p[1], p[2], p[3]);
      }
    }
  }
}

}  // namespace hdg
