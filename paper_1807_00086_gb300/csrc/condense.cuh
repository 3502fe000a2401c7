// Condensation of the acoustic element blocks (the formulas of kernels.cuh): H, its Cholesky
// factor, W = L^{-1} Bt, S = W^T W + the trace terms, H^{-1}, and the copies of S_K that the
// mixed-precision solves read.
//
// What bounds it: FP64 issue (a warp's FP64 instruction holds its SM partition for about 64
// cycles, whatever lanes are live), so lanes must not idle and no operation be done twice.
// EPW elements share a warp, LPE = 32 / EPW lanes each. The factorisation is left-looking with
// the rows of Bt^T and of the identity carried below those of H: at every column exactly
// NP + M rows are in play (an H row leaves as an identity row enters), a whole number of
// passes of the lanes but for a few, every partial sum is in a register, and one reciprocal
// square root per column replaces the divisions, shared by the EPW elements. H (lower) and
// L^{-1} (upper, by rows of its transpose) share one square: their common diagonal holds
// 1 / L_jj. S is accumulated in TS x TS register tiles of its upper triangle only.
// 82,944 tets, k = 3: 6.76 ms (15.7 ms with a 128-thread CTA per element, all of S and a division
// per row and column); its 35 k FP64 multiply-adds per element without an idle lane: 4.6 ms.
#pragma once

#include "kernels.cuh"

namespace hdg {

template <int DIM, int K>
struct CondCfg {
  static constexpr int NP = Dims<DIM, K>::NP, M = Dims<DIM, K>::M, NFC = DIM + 1;
  static constexpr int NS = DIM * (DIM + 1) / 2;
  static constexpr int NTRI = NP * (NP + 1) / 2;
  // odd row stride: the eight lanes of an element, one row each, fall into distinct banks
  static constexpr int LD = NP % 2 ? NP : NP + 1;
  static constexpr int CW = NFC * (DIM + 1);           // coefficients of Bt per face
  static constexpr int NCO = NFC + NS + CW + NFC * NFC;
  static constexpr int SM0 = (NP + M) * LD + NCO;
  // = 8 mod 16: the elements' equal offsets lie in two bank groups
  static constexpr int SM_E = SM0 + (24 - SM0 % 16) % 16;
  // elements per warp: four while five warps fit an SM, else two
  static constexpr int EPW = SM_E * 8 * 4 * 5 <= 224 * 1024 ? 4 : 2;
  static constexpr int LPE = 32 / EPW;
  static constexpr int RT = (NP + M + LPE - 1) / LPE;  // rows per lane in a column
  static constexpr int TS = M % 4 == 0 ? 4 : 3;        // S tile side
  static_assert(M % TS == 0, "whole tiles");
  static constexpr size_t SMEM = sizeof(double) * EPW * SM_E;
};

// reference tables of the assembly: HP [NFC + NS][NTRI] rows of the lower triangles of E^_f and of
// the symmetric combinations Dr_r Dr_r^T, then Dr_r Dr_s^T + Dr_s Dr_r^T (r < s)
struct CondTabs {
  const double* HP;
  const double *Ff, *DFrf, *Pfg;
};

template <int DIM, int K>
__global__ void __launch_bounds__(32) condense_kernel(DevMesh mesh, CondTabs T, double alpha, double tau,
                                                      double* __restrict__ S, double* __restrict__ Hinv,
                                                      int* __restrict__ err) {
  using D = Dims<DIM, K>;
  using C = CondCfg<DIM, K>;
  constexpr int NP = C::NP, NF = D::NF, M = C::M, NFC = C::NFC, NS = C::NS, LD = C::LD, LPE = C::LPE, RT = C::RT, TS = C::TS;
  extern __shared__ __align__(16) double csm[];
  const int lane = threadIdx.x % LPE, sub = threadIdx.x / LPE;
  double* H = csm + sub * C::SM_E;       // [NP][LD]: L (lower), L^{-T} (upper), 1 / L_jj
  double* W = H + NP * LD;               // [M][LD]: Bt^T, then (L^{-1} Bt)^T
  double* cH = W + M * LD;               // [NFC + NS]
  double* cW = cH + NFC + NS;            // [NFC][DIM + 1]
  double* cP = cW + C::CW;               // [NFC][NFC]
  const int64_t e0 = (int64_t)blockIdx.x * C::EPW;
  const bool live = e0 + sub < mesh.ne;
  const int64_t e = live ? e0 + sub : e0;   // a group past the end repeats the first one's work
  const double* g = mesh.geo + e * GEO_STRIDE;
  const double dJ = g[0], rho = mesh.rho[e], cc = mesh.c[e];
  const double b = alpha * rho, ib = 1.0 / b, ibd = 1.0 / (b * dJ);
  const double adJ = alpha / (rho * cc * cc) * dJ;
  for (int t = lane; t < C::NCO; t += LPE) {
    double v = 0.0;
    if (t < NFC) {
      v = tau * g[D::OJF + t];
    } else if (t < NFC + NS) {
      int r = t - NFC, s = r;   // (0,0) .. (d-1,d-1), then (0,1), (0,2), (1,2)
      if (r >= DIM) { r = t - NFC - DIM == 2 ? 1 : 0; s = t - NFC - DIM == 0 ? 1 : 2; }
      for (int j = 0; j < DIM; ++j) v += g[1 + r * DIM + j] * g[1 + s * DIM + j];
      v *= dJ * ib;
    } else if (t < NFC + NS + C::CW) {
      const int f = (t - NFC - NS) / (DIM + 1), r = (t - NFC - NS) % (DIM + 1) - 1;
      if (r < 0) {
        v = -g[D::OJF + f] * tau;
      } else {
        for (int j = 0; j < DIM; ++j) v += g[D::ON + f * DIM + j] * g[1 + r * DIM + j];
        v *= -g[D::OJF + f] * ib;
      }
    } else {
      const int f = (t - NFC - NS - C::CW) / NFC, h = (t - NFC - NS - C::CW) % NFC;
      for (int j = 0; j < DIM; ++j) v += g[D::ON + f * DIM + j] * g[D::ON + h * DIM + j];
      v *= ibd * g[D::OJF + f] * g[D::OJF + h];
    }
    cH[t] = v;
  }
  __syncwarp();
  {
    double ch[NFC + NS];
#pragma unroll
    for (int t = 0; t < NFC + NS; ++t) ch[t] = cH[t];
    int i = 0, i0 = 0;   // row of idx and its first packed index
    for (int idx = lane; idx < C::NTRI; idx += LPE) {
      while (idx > i0 + i) { i0 += i + 1; ++i; }
      const int l = idx - i0;
      double v = i == l ? adJ : 0.0;
#pragma unroll
      for (int t = 0; t < NFC + NS; ++t) v += ch[t] * T.HP[t * C::NTRI + idx];
      H[i * LD + l] = v;
    }
  }
#pragma unroll 2
  for (int idx = lane; idx < NP * M; idx += LPE) {
    const int i = idx / M, col = idx % M, f = col / NF, mm = col % NF;
    double v = cW[f * (DIM + 1)] * T.Ff[(f * NP + i) * NF + mm];
#pragma unroll
    for (int r = 0; r < DIM; ++r) v += cW[f * (DIM + 1) + 1 + r] * T.DFrf[((r * NFC + f) * NP + i) * NF + mm];
    W[col * LD + i] = v;
  }
  __syncwarp();
  for (int j = 0; j < NP; ++j) {
    // rows of this column: q = 0 the pivot, then the H rows below it, Bt^T, the identity rows c < j
    int off[RT], l0[RT];   // offset of the row (W follows H), first column its sum takes
    double acc[RT];
#pragma unroll
    for (int t = 0; t < RT; ++t) {
      const int q = lane + LPE * t, c = q - (NP - j) - M;   // c: identity row
      off[t] = c < 0 ? (j + q) * LD : (c < j ? c * LD : 0);
      l0[t] = c < 0 ? 0 : (c < j ? c : NP);
      acc[t] = c < 0 ? H[off[t] + j] : 0.0;
    }
    const double* Lj = H + j * LD;
    for (int l = 0; l < j; ++l) {
      const double v = Lj[l];
#pragma unroll
      for (int t = 0; t < RT; ++t)
        if (l >= l0[t]) acc[t] -= H[off[t] + l] * v;
    }
    double d = __shfl_sync(0xffffffffu, acc[0], 0, LPE);
    if (!(d > 0.0)) {
      if (live && lane == 0) atomicExch(err, 1);
      d = 1.0;
    }
    const double r = rsqrt(d);
    __syncwarp();   // every lane has read row j and the entries it overwrites
#pragma unroll
    for (int t = 0; t < RT; ++t) {
      const int q = lane + LPE * t;
      if (q < NP + M) H[off[t] + j] = q == 0 ? r : acc[t] * r;
    }
    __syncwarp();
  }
  double* Se = S + e * (int64_t)(M * M);
  {
    constexpr int NTS = M / TS, NTILE = NTS * (NTS + 1) / 2;
    int ti = 0, t0 = 0;   // tile row and the index of its diagonal tile (row-wise upper triangle)
    for (int t = lane; t < NTILE; t += LPE) {
      while (t >= t0 + NTS - ti) { t0 += NTS - ti; ++ti; }
      const int tj = ti + t - t0;
      const double *z1 = W + ti * TS * LD, *z2 = W + tj * TS * LD;
      double acc[TS][TS];
#pragma unroll
      for (int x = 0; x < TS; ++x)
#pragma unroll
        for (int y = 0; y < TS; ++y) acc[x][y] = 0.0;
#pragma unroll 2
      for (int i = 0; i < NP; ++i) {
        double a1[TS], a2[TS];
#pragma unroll
        for (int x = 0; x < TS; ++x) { a1[x] = z1[x * LD + i]; a2[x] = z2[x * LD + i]; }
#pragma unroll
        for (int x = 0; x < TS; ++x)
#pragma unroll
          for (int y = 0; y < TS; ++y) acc[x][y] += a1[x] * a2[y];
      }
      if (!live) continue;
#pragma unroll
      for (int x = 0; x < TS; ++x) {
        const int ra = ti * TS + x, f = ra / NF, aa = ra % NF;
#pragma unroll
        for (int y = 0; y < TS; ++y) {
          const int cb = tj * TS + y, h = cb / NF, bb = cb % NF;
          double v = acc[x][y];
          if (ra == cb) v -= cH[f];
          v -= cP[f * NFC + h] * T.Pfg[((f * NFC + h) * NF + aa) * NF + bb];
          acc[x][y] = v;
          Se[ra * M + cb] = v;
        }
      }
      if (ti != tj) {
#pragma unroll
        for (int y = 0; y < TS; ++y)
#pragma unroll
          for (int x = 0; x < TS; ++x) Se[(tj * TS + y) * M + ti * TS + x] = acc[x][y];
      }
    }
  }
  if (!live) return;
  double* He = Hinv + e * (int64_t)(NP * NP);
  int i = 0, i0 = 0;
  for (int idx = lane; idx < C::NTRI; idx += LPE) {
    while (idx > i0 + i) { i0 += i + 1; ++i; }
    const int l = idx - i0;
    double s = 0.0;
#pragma unroll 4
    for (int q = i; q < NP; ++q) s += H[i * LD + q] * H[l * LD + q];
    He[i * NP + l] = s;
    He[l * NP + i] = s;
  }
}

// The same for small meshes: one CTA of four warps per element, which also writes the coefficients of the
// local solves (local_co_kernel). A warp of condense_kernel that is alone on its SM partition takes 64 cycles
// per FP64 instruction, for EPW elements, while other partitions are idle. hdg_condense in mixed precision, this
// kernel / condense_kernel, us: triangles, k = 2: 128: 53 / 59, 578: 61 / 63, 1,152: 72 / 63; k = 3: 128: 65 / 76,
// 578: 75 / 76, 1,152: 91 / 76; k = 4: 128: 86 / 105, 578: 99 / 105, 1,152: 128 / 107. Tetrahedra, k = 1: 384:
// 54 / 63, 750: 61 / 61, 1,296: 74 / 64; k = 2: 384: 85 / 105, 750: 95 / 107, 1,296: 128 / 113; k = 3: 384:
// 162 / 286, 750: 209 / 287, 1,296: 321 / 298; k = 4: 384: 382 / 500, 750: 536 / 508. The lines lie where this
// kernel still gains: at most so many elements per SM.
template <int DIM, int K>
__host__ __device__ constexpr int cond_cta_per_sm() {
  return DIM == 3 && (K == 2 || K == 3) ? 6 : 4;
}
template <int DIM, int K>
__global__ void __launch_bounds__(128) condense_cta_kernel(DevMesh mesh, Tabs T, double alpha, double tau,
                                                          double* __restrict__ S, double* __restrict__ Hinv,
                                                          int* __restrict__ err, double* __restrict__ co64,
                                                          df2* __restrict__ codf) {
  constexpr int NT = 128;
  using D = Dims<DIM, K>;
  constexpr int NP = D::NP, NF = D::NF, M = D::M, NFC = D::NFC;
  __shared__ double H[NP * NP];
  __shared__ double W[NP * M];
  __shared__ double Li[NP * NP];
  __shared__ double g[GEO_STRIDE];
  __shared__ double Grs[DIM * DIM], Bfr[NFC * DIM], nn[NFC * NFC];
  const int64_t e = blockIdx.x;
  const int tid = threadIdx.x;
  if (tid < GEO_STRIDE) g[tid] = mesh.geo[e * GEO_STRIDE + tid];
  __syncthreads();
  const double dJ = g[0];
  const double rho = mesh.rho[e], cc = mesh.c[e];
  const double a = alpha / (rho * cc * cc), b = alpha * rho;
  if (tid == NT - 1) {
    const double v[4] = {1.0 / b, a * dJ, b * dJ, 1.0 / (b * dJ)};
    for (int i = 0; i < 4; ++i)
      if (co64) co64[4 * e + i] = v[i];
      else if (codf) codf[4 * e + i] = df_from(v[i]);
  }
  if (tid < DIM * DIM) {
    int r = tid / DIM, s = tid % DIM;
    double v = 0.0;
    for (int j = 0; j < DIM; ++j) v += g[1 + r * DIM + j] * g[1 + s * DIM + j];
    Grs[tid] = v;
  } else if (tid < DIM * DIM + NFC * DIM) {
    int t = tid - DIM * DIM, f = t / DIM, r = t % DIM;
    double v = 0.0;
    for (int j = 0; j < DIM; ++j) v += g[D::ON + f * DIM + j] * g[1 + r * DIM + j];
    Bfr[t] = v;
  } else if (tid < DIM * DIM + NFC * DIM + NFC * NFC) {
    int t = tid - DIM * DIM - NFC * DIM, f = t / NFC, h = t % NFC;
    double v = 0.0;
    for (int j = 0; j < DIM; ++j) v += g[D::ON + f * DIM + j] * g[D::ON + h * DIM + j];
    nn[t] = v;
  }
  __syncthreads();
  for (int idx = tid; idx < NP * NP; idx += NT) {
    const int i = idx / NP, l = idx % NP;
    double v = (i == l) ? a * dJ : 0.0;
    double fe = 0.0;
    for (int f = 0; f < NFC; ++f) fe += g[D::OJF + f] * T.Ef[(f * NP + i) * NP + l];
    double dd = 0.0;
    for (int rs = 0; rs < DIM * DIM; ++rs) dd += Grs[rs] * T.Trs[(rs * NP + i) * NP + l];
    H[idx] = v + tau * fe + (dJ / b) * dd;
    Li[idx] = (i == l) ? 1.0 : 0.0;
  }
  for (int idx = tid; idx < NP * M; idx += NT) {
    const int i = idx / M, col = idx % M, f = col / NF, mm = col % NF;
    double v = tau * T.Ff[(f * NP + i) * NF + mm];
    double d2 = 0.0;
    for (int r = 0; r < DIM; ++r) d2 += Bfr[f * DIM + r] * T.DFrf[((r * NFC + f) * NP + i) * NF + mm];
    W[idx] = -g[D::OJF + f] * (v + d2 / b);
  }
  __syncthreads();
  // Cholesky, right-looking, lower triangle in place
  for (int j = 0; j < NP; ++j) {
    if (tid == 0) {
      double d = H[j * NP + j];
      if (!(d > 0.0)) { atomicExch(err, 1); d = 1.0; }
      H[j * NP + j] = sqrt(d);
    }
    __syncthreads();
    for (int i = j + 1 + tid; i < NP; i += NT) H[i * NP + j] /= H[j * NP + j];
    __syncthreads();
    const int w = NP - j - 1;
    for (int idx = tid; idx < w * w; idx += NT) {
      const int i = j + 1 + idx / w, l = j + 1 + idx % w;
      if (l <= i) H[i * NP + l] -= H[i * NP + j] * H[l * NP + j];
    }
    __syncthreads();
  }
  // forward substitution, one column per thread: W <- L^{-1} Bt, Li <- L^{-1}
  for (int col = tid; col < M + NP; col += NT) {
    if (col < M) {
      for (int i = 0; i < NP; ++i) {
        double s = W[i * M + col];
        for (int l = 0; l < i; ++l) s -= H[i * NP + l] * W[l * M + col];
        W[i * M + col] = s / H[i * NP + i];
      }
    } else {
      const int c2 = col - M;
      for (int i = c2; i < NP; ++i) {
        double s = (i == c2) ? 1.0 : 0.0;
        for (int l = c2; l < i; ++l) s -= H[i * NP + l] * Li[l * NP + c2];
        Li[i * NP + c2] = s / H[i * NP + i];
      }
    }
  }
  __syncthreads();
  double* Se = S + e * (int64_t)(M * M);
  const double ib = 1.0 / (b * dJ);
  for (int idx = tid; idx < M * M; idx += NT) {
    const int ra = idx / M, cb = idx % M;
    const int f = ra / NF, aa = ra % NF, h = cb / NF, bb = cb % NF;
    double s = 0.0;
    for (int i = 0; i < NP; ++i) s += W[i * M + ra] * W[i * M + cb];
    if (ra == cb) s -= tau * g[D::OJF + f];
    s -= ib * g[D::OJF + f] * g[D::OJF + h] * nn[f * NFC + h] * T.Pfg[((f * NFC + h) * NF + aa) * NF + bb];
    Se[idx] = s;
  }
  double* He = Hinv + e * (int64_t)(NP * NP);
  for (int idx = tid; idx < NP * NP; idx += NT) {
    const int i = idx / NP, l = idx % NP;
    const int q0 = i > l ? i : l;
    double s = 0.0;
    for (int q = q0; q < NP; ++q) s += Li[q * NP + i] * Li[q * NP + l];
    He[idx] = s;
  }
}

// Double-float copy of an FP64 array (H^{-1} after each condensation, the element geometry).
static __global__ void to_df_kernel(int64_t n, const double* __restrict__ a, df2* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    df2 v;
    split_f64(a[t], v.h, v.l);
    out[t] = v;
  }
}

// Every copy of S_K that a mixed-precision context reads, from one pass over the FP64 blocks
// (null: not wanted). One kernel per copy read S_K up to four times and searched the row of every
// packed entry: 2.61 ms for the FP32, FP16 and double-float copies of 82,944 blocks of 40 x 40,
// against 0.57 ms here; what remains is the shared-memory transposition and the 2.0 GB moved.
// An FP16 entry is the FP32 quotient of hi and the scale, rounded: at most 2^-23 of it beside the 2^-11 of the
// rounding.
struct PackOut {
  float* Sdf;      // [e][hi | lo] diagonal-major upper triangles (refinement apply)
  float* S32;      // [group][P4][32][4] packed rows of the upper triangle
  __half* S16;     // [group][P8][32][8] of S / sc16
  float* sc16;     // [e] max |S_K|, rounded up
  float* S32m;     // [e][P4 * 4] packed rows
  float *Shi, *Slo;   // [e][M][M]
};

template <int DIM, int K>
struct PackCfg {
  static constexpr int M = Packed<DIM, K>::M, P = Packed<DIM, K>::P, P4 = Packed<DIM, K>::P4, PD = P4 * 4;
  static constexpr int P8 = Packed16<DIM, K>::P8;
  static constexpr int EPB = 8;   // elements per CTA, one per warp: 128-byte runs of the group layouts
  static constexpr size_t SMEM = sizeof(float) * EPB * 2 * PD;
};

// position of packed entry p (rows of the upper triangle) in the diagonal-major order
template <int M>
__device__ __forceinline__ int pack_diag_pos(int p) {
  int r = (int)((2 * M + 1 - sqrtf((float)((2 * M + 1) * (2 * M + 1) - 8 * p))) * 0.5f);
  if (r > 0 && packed_index(M, r, r) > p) --r;
  if (r + 1 < M && packed_index(M, r + 1, r + 1) <= p) ++r;
  return diag_off(M, p - packed_index(M, r, r)) + r;
}

template <int DIM, int K>
__global__ void __launch_bounds__(256) pack_kernel(int64_t ne, const double* __restrict__ S, PackOut o) {
  using C = PackCfg<DIM, K>;
  constexpr int M = C::M, P = C::P, P4 = C::P4, P8 = C::P8, PD = C::PD, EPB = C::EPB;
  extern __shared__ __align__(16) float pksm[];   // [EPB][hi PD | lo PD]
  __shared__ float scs[EPB];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t e0 = (int64_t)blockIdx.x * EPB, e = e0 + w;
  float* hi = pksm + w * 2 * PD;
  float* lo = hi + PD;
  if (e < ne) {
    const double* Se = S + e * (int64_t)(M * M);
    float mx = 0.f;
    // RB rows at a time, so that several loads are in flight per lane (one load per row and pass
    // left the kernel waiting on latency: 1.06 ms instead of 0.57 ms for 82,944 blocks of 40 x 40)
    constexpr int RB = 6, CP = (M + 31) / 32;
    for (int r0 = 0; r0 < M; r0 += RB) {
      double v[RB][CP];
#pragma unroll
      for (int y = 0; y < RB; ++y)
#pragma unroll
        for (int q = 0; q < CP; ++q) {
          const int r = r0 + y, c = r + lane + 32 * q;
          v[y][q] = r < M && c < M ? __ldcs(Se + r * M + c) : 0.0;
        }
#pragma unroll
      for (int y = 0; y < RB; ++y)
#pragma unroll
        for (int q = 0; q < CP; ++q) {
          const int r = r0 + y, c = r + lane + 32 * q;
          if (r >= M || c >= M) continue;
          float h, l;
          split_f64(v[y][q], h, l);
          const int pos = diag_off(M, c - r) + r;
          hi[pos] = h;
          lo[pos] = l;
          // |S| rounded up to FP32: hi, or the next float where lo points outwards
          const float ah = fabsf(h), al = h < 0.f ? -l : l;
          mx = fmaxf(mx, al > 0.f ? __uint_as_float(__float_as_uint(ah) + 1u) : ah);
        }
    }
    for (int t = P + lane; t < PD; t += 32) hi[t] = lo[t] = 0.f;
    for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    if (lane == 0) {
      scs[w] = mx > 0.f ? mx : 1.f;
      if (o.sc16) o.sc16[e] = scs[w];
    }
    __syncwarp();
    if (o.Sdf) {
      float4* d = reinterpret_cast<float4*>(o.Sdf + e * 2 * PD);
      for (int t = lane; t < 2 * PD / 4; t += 32) d[t] = reinterpret_cast<const float4*>(hi)[t];
    }
    if (o.S32m)
      for (int p = lane; p < PD; p += 32) o.S32m[e * PD + p] = p < P ? hi[pack_diag_pos<M>(p)] : 0.f;
    if (o.Shi)
      for (int t = lane; t < M * M; t += 32) {
        const int r = t / M, c = t % M, a = r < c ? r : c, pos = diag_off(M, r < c ? c - r : r - c) + a;
        o.Shi[e * (int64_t)(M * M) + t] = hi[pos];
        o.Slo[e * (int64_t)(M * M) + t] = lo[pos];
      }
  } else {
    for (int t = lane; t < 2 * PD; t += 32) hi[t] = 0.f;   // the last group's missing elements
    if (lane == 0) scs[w] = 1.f;
  }
  if (!o.S32 && !o.S16) return;
  __syncthreads();
  // group layouts: 16 bytes per (vector, element), the CTA's eight elements side by side
  const int el = threadIdx.x % EPB;
  const float* he = pksm + el * 2 * PD;
  const int64_t g = (e0 + el) >> 5;
  const int ln = (int)((e0 + el) & 31);
  if (o.S32)
    for (int q = threadIdx.x / EPB; q < P4; q += 256 / EPB) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = 4 * q + j < P ? he[pack_diag_pos<M>(4 * q + j)] : 0.f;
      reinterpret_cast<float4*>(o.S32)[(g * P4 + q) * 32 + ln] = make_float4(v[0], v[1], v[2], v[3]);
    }
  if (o.S16) {
    const float sc = scs[el];
    for (int q = threadIdx.x / EPB; q < P8; q += 256 / EPB) {
      __half2 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float a = 8 * q + 2 * j < P ? __fdiv_rn(he[pack_diag_pos<M>(8 * q + 2 * j)], sc) : 0.f;
        const float b = 8 * q + 2 * j + 1 < P ? __fdiv_rn(he[pack_diag_pos<M>(8 * q + 2 * j + 1)], sc) : 0.f;
        v[j] = __floats2half2_rn(a, b);
      }
      reinterpret_cast<uint4*>(o.S16)[(g * P8 + q) * 32 + ln] = *reinterpret_cast<const uint4*>(v);
    }
  }
}

}  // namespace hdg
