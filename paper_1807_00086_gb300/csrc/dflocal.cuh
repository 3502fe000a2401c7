// Element-local solves of the acoustic scheme in double-float arithmetic on the FP32 pipe.
//
// The same two maps as local_kernel (Sec. 2.4, Eq. LS, the element blocks of the condensed
// system): MODE 0 forms gslot = C_K A_K^{-1} (F_K - B_K lamD_K), MODE 1 recovers
// u_K = A_K^{-1} (F_K - B_K lam_K). Every product and sum is carried as an unevaluated pair
// hi + lo of floats (about 48 significant bits): products by fmaf-based exact splitting
// (Dekker's two-product), sums by Knuth's two-sum, so the results agree with the FP64 kernel
// to a few units of 1e-14 relative while the work runs on the FP32 units (FP64 issues at a
// small fraction of the FP32 rate on this GPU). Only the conversions from and to FP64 and
// the per-element coefficients use FP64 instructions.
#pragma once

#include "kernels.cuh"

namespace hdg {

// Reference tables as rows of their nonzero entries (sparse_rows): the derivative of a mode has a lower
// degree, and the collapsed-coordinate basis is orthonormal, so Dr holds 202 of 1200 entries and Ff 320 of
// 800 for k = 3 tetrahedra; the others are quadrature round-off (below 1e-13). Row groups, in this order:
//   A  [NP]        idx r NP + l, Dr[r][i][l]   (derivative matrices, volume-row sums)
//   B  [DIM][NP]   idx l,        Dr[r][l][i]   (transposed products)
//   C  [NFC][NP]   idx m,        Ff[f][i][m]   (face mass, volume-row sums)
//   D  [NFC][NF]   idx q,        Ff[f][q][m]   (face mass, face-row sums)
// perm: the volume rows by falling length of A (rising length of B), so that the rows of a warp are
// about equally long.
struct alignas(16) SpDf {
  float h, l;
  int idx, pad;
};
struct TabsDf {
  const SpDf* ent;
  const int32_t *ptr, *perm;
};

struct df2x2 {
  df2 a, b;
};
__device__ __forceinline__ df2x2 df_ld2(const df2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ void df_st2(df2* p, df2 a, df2 b) { *reinterpret_cast<float4*>(p) = make_float4(a.h, a.l, b.h, b.l); }

// s0, s1 += table row times two neighbouring columns of x (rows WS apart)
template <int WS>
__device__ __forceinline__ void sp_row2(const TabsDf& T, int row, const df2* x, DfAcc& s0, DfAcc& s1) {
  const int b = __ldg(T.ptr + row + 1);
#pragma unroll 4
  for (int q = __ldg(T.ptr + row); q < b; ++q) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(T.ent + q));
    const df2x2 v = df_ld2(x + __float_as_int(t.z) * WS);
    s0.fma(df2{t.x, t.y}, v.a);
    s1.fma(df2{t.x, t.y}, v.b);
  }
}

// Element coefficients of the local solves at the mass shift alpha: 1/b, a' dJ, b dJ, 1/(b dJ) with
// b = alpha rho, a' = alpha/(rho c^2); formed once per condensation, because an FP64 division by one
// thread of a CTA holds its SM partition as long as a full warp's
static __global__ void local_co_kernel(DevMesh mesh, double alpha, df2* __restrict__ co) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < mesh.ne; e += (int64_t)gridDim.x * blockDim.x) {
    const double rho = mesh.rho[e], cc = mesh.c[e], dJ = mesh.geo[e * GEO_STRIDE];
    const double b = alpha * rho, ap = alpha / (rho * cc * cc);
    co[4 * e] = df_from(1.0 / b);
    co[4 * e + 1] = df_from(ap * dJ);
    co[4 * e + 2] = df_from(b * dJ);
    co[4 * e + 3] = df_from(1.0 / (b * dJ));
  }
}

// One kernel for one column (CW = 0) and for column blocks (the multi-source and serving batches, CW =
// min(R, 16) columns of EPB elements per CTA). Every array is [row][W] with the W columns of the CTA:
// its elements, or (element, right-hand side) pairs. A thread holds row i of two neighbouring columns, so
// that one table entry serves two products and one 16-byte read both of their factors; lanes run over the
// columns first, so that the rows of a warp are few and of like length. H^{-1}, which differs by element,
// is read along its rows instead. One column: F, the history and the results pass through shared memory,
// so that the global accesses are contiguous.
// What bounds it: the instructions of the double-float products (11 each) and of the
// pointwise steps. k = 3 tetrahedra, modes 0 / 1: 196,608 elements, one column 0.68 / 0.68 ms (0.75 / 0.72
// with dense tables), 24,576 x 64 columns 3.3 / 4.1 ms (5.1 / 4.9), 16,464 x 4 columns 0.16 / 0.20 ms (0.24).
template <int DIM, int K, int CW>
struct LocalDfCfg {
  static constexpr int NP = Dims<DIM, K>::NP;
  static constexpr bool ONE = CW == 0;
  static constexpr int PE = NP * (ONE ? 1 : CW) / 2;          // threads per element of a column block
  static constexpr int EPB = ONE ? (NP <= 10 ? 32 : NP <= 20 ? 16 : 8) : PE >= 160 ? 1 : 160 / PE;
  static constexpr int W = ONE ? EPB : EPB * CW;
  static constexpr int WS = ONE ? W + 2 : W;                  // padded where rows are filled column by column
  static constexpr int HW = W / 2;                            // threads per row
  static constexpr int NT = NP * HW;
};

template <int DIM, int K, int MODE, int CW>
__global__ void __launch_bounds__(LocalDfCfg<DIM, K, CW>::NT)
    local_df_kernel(DevMesh mesh, TabsDf T, const df2* __restrict__ geo, const df2* __restrict__ coef,
                    const df2* __restrict__ Hinv, df2 tau, int R, const double* __restrict__ F,
                    const double* __restrict__ hist, SrcArgs src, const double* __restrict__ lam, double* __restrict__ out) {
  using D = Dims<DIM, K>;
  using L = LocalDfCfg<DIM, K, CW>;
  constexpr int NP = D::NP, NF = D::NF, M = D::M, NFC = D::NFC, N = D::N, EPB = L::EPB, NT = L::NT, WS = L::WS, HW = L::HW;
  constexpr int RB = NP, RC = RB + DIM * NP, RD = RC + NFC * NP;
  constexpr bool ONE = L::ONE;
  __shared__ df2 g[EPB][GEO_STRIDE], co[EPB][4], nj[EPB][NFC * DIM];   // nj: J_F n_f
  __shared__ __align__(16) df2 Fs[ONE ? N : 1][WS];     // one column: F or history, then u
  __shared__ __align__(16) df2 Tr[DIM * NP][WS];        // the face weights w_f (f < DIM) in MODE 0
  __shared__ __align__(16) df2 rp[NP][WS];              // the last face's weights in MODE 0
  __shared__ __align__(16) df2 pp[NP][WS];
  __shared__ __align__(16) df2 ll[M][WS];               // traces; one column, MODE 0: then the result
  __shared__ int anyf[EPB];                             // faces with a (nonzero) trace, as bits
  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int cb = ONE ? 0 : blockIdx.y * CW;
  for (int t = tid; t < EPB * GEO_STRIDE; t += NT) {
    const int64_t e = e0 + t / GEO_STRIDE;
    g[t / GEO_STRIDE][t % GEO_STRIDE] = e < mesh.ne ? geo[e * GEO_STRIDE + t % GEO_STRIDE] : df2{0.f, 0.f};
  }
  for (int t = tid; t < EPB * NFC * DIM; t += NT) {
    const int q = t / (NFC * DIM), x = t % (NFC * DIM);
    const df2* ge = geo + (e0 + q) * GEO_STRIDE;
    nj[q][x] = e0 + q < mesh.ne ? df_mul(ge[D::ON + x], ge[D::OJF + x / DIM]) : df2{0.f, 0.f};
  }
  for (int t = tid; t < EPB * 4; t += NT) co[t / 4][t % 4] = e0 + t / 4 < mesh.ne ? coef[4 * e0 + t] : df2{0.f, 0.f};
  for (int q = tid; q < EPB; q += NT) {
    int use = 0;
    if (e0 + q < mesh.ne && lam)
      for (int f = 0; f < NFC; ++f)
        if (MODE == 1 || mesh.face_bnd[mesh.elem_face[(e0 + q) * NFC + f]] >= 0) use |= 1 << f;
    anyf[q] = use;
  }
  if (lam)
    for (int t = tid; t < M * L::W; t += NT) {
      const int q = ONE ? t / M : t / (M * CW), r = ONE ? t % M : (t / (ONE ? 1 : CW)) % M, jc = ONE ? 0 : t % (ONE ? 1 : CW);
      const int64_t e = e0 + q;
      double v = 0.0;
      if (e < mesh.ne) {
        const int f = mesh.elem_face[e * NFC + r / NF];
        if ((MODE == 1) || (mesh.face_bnd[f] >= 0)) v = lam[((int64_t)f * NF + r % NF) * R + cb + jc];
      }
      ll[r][ONE ? q : q * CW + jc] = dfl_from(v);
    }
  if constexpr (ONE) {
    const double* X = hist ? hist : F;
    for (int t = tid; t < EPB * N; t += NT) Fs[t % N][t / N] = dfl_from(e0 + t / N < mesh.ne ? X[e0 * N + t] : 0.0);
  }
  __syncthreads();
  const int i = __ldg(T.perm + tid / HW), j0 = 2 * (tid % HW);
  const int el[2] = {ONE ? j0 : j0 / (ONE ? 1 : CW), ONE ? j0 + 1 : j0 / (ONE ? 1 : CW)};
  // row i of F~ for all components (+ the F^ lam face products it needs)
  df2 Fu[DIM + 1][2];
  {
    const int use = anyf[el[0]] | anyf[el[1]];
    df2 Fl[NFC][2];
    if (use)
#pragma unroll
      for (int f = 0; f < NFC; ++f) {
        DfAcc s0, s1;
        if ((use >> f) & 1) sp_row2<WS>(T, RC + f * NP + i, &ll[f * NF][j0], s0, s1);
        Fl[f][0] = df_of(s0);
        Fl[f][1] = df_of(s1);
      }
#pragma unroll
    for (int comp = 0; comp <= DIM; ++comp) {
      df2 x[2];
      if constexpr (ONE) {
        const df2x2 y = df_ld2(&Fs[comp * NP + i][j0]);
        x[0] = y.a;
        x[1] = y.b;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t e = e0 + el[h];
        const df2* ge = g[el[h]];
        df2 v{0.f, 0.f};
        if (e < mesh.ne) {
          const int j = ONE ? 0 : cb + (j0 + h) % (ONE ? 1 : CW);
          if constexpr (!ONE) x[h] = dfl_from((hist ? hist : F)[(e * N + comp * NP + i) * R + j]);
          v = x[h];
          if (hist) {
            v = df_mul(co[el[h]][comp == 0 ? 1 : 2], v);
            if (comp == 0 && src.ptr && src.ptr[e] < src.ptr[e + 1]) {
              double sv = 0.0;
              for (int q = src.ptr[e]; q < src.ptr[e + 1]; ++q)
                if (ONE || src.col[q] == j) sv += ricker_at(src, q) * src.phi[(int64_t)q * NP + i];
              v = df_add(v, df_from(sv));
            }
          }
        }
        if (use) {
          DfAcc bl;
          if (comp == 0) {
#pragma unroll
            for (int f = 0; f < NFC; ++f) bl.fma(ge[D::OJF + f], Fl[f][h]);
            v = df_add(v, df_mul(tau, df_of(bl)));
          } else {
#pragma unroll
            for (int f = 0; f < NFC; ++f) bl.fma(nj[el[h]][f * DIM + comp - 1], Fl[f][h]);
            v = df_add(v, df_neg(df_of(bl)));
          }
        }
        Fu[comp][h] = v;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < DIM; ++r) {
    df2 t[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      DfAcc s;
#pragma unroll
      for (int jj = 0; jj < DIM; ++jj) s.fma(g[el[h]][1 + r * DIM + jj], Fu[jj + 1][h]);
      t[h] = df_of(s);
    }
    df_st2(&Tr[r * NP + i][j0], t[0], t[1]);
  }
  __syncthreads();
  {
    DfAcc s0, s1;
    sp_row2<WS>(T, i, &Tr[0][j0], s0, s1);
    df_st2(&rp[i][j0], df_add(Fu[0][0], df_neg(df_mul(df_of(s0), co[el[0]][0]))),
           df_add(Fu[0][1], df_neg(df_mul(df_of(s1), co[el[1]][0]))));
  }
  __syncthreads();
  {
    // p = H^{-1} rp; H^{-1} is symmetric, so row i is read as column i
    constexpr int HC = ONE ? 1 : CW / 2;
    const int q = tid / (NP * HC), i2 = (tid / HC) % NP, j2 = ONE ? 2 * q : q * CW + 2 * (tid % HC);
    const int64_t ea = e0 + (ONE ? 2 * q : q);
    const df2* Ha = Hinv + (ea < mesh.ne ? ea : 0) * (int64_t)(NP * NP) + i2;
    DfAcc s0, s1;
    if constexpr (ONE) {
      const df2* Hb = Hinv + (ea + 1 < mesh.ne ? ea + 1 : 0) * (int64_t)(NP * NP) + i2;
#pragma unroll 5
      for (int l = 0; l < NP; ++l) {
        const df2x2 x = df_ld2(&rp[l][j2]);
        s0.fma(Ha[l * NP], x.a);
        s1.fma(Hb[l * NP], x.b);
      }
    } else {
#pragma unroll 5
      for (int l = 0; l < NP; ++l) {
        const df2 tv = Ha[l * NP];
        const df2x2 x = df_ld2(&rp[l][j2]);
        s0.fma(tv, x.a);
        s1.fma(tv, x.b);
      }
    }
    df_st2(&pp[i2][j2], df_of(s0), df_of(s1));
  }
  __syncthreads();
  const df2x2 pw = df_ld2(&pp[i][j0]);
  const df2 pv[2] = {pw.a, pw.b};
  df2 vv[DIM][2];
  {
    df2 qd[DIM][2];
#pragma unroll
    for (int r = 0; r < DIM; ++r) {
      DfAcc s0, s1;
      sp_row2<WS>(T, RB + r * NP + i, &pp[0][j0], s0, s1);
      qd[r][0] = df_of(s0);
      qd[r][1] = df_of(s1);
    }
#pragma unroll
    for (int jj = 0; jj < DIM; ++jj)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        DfAcc s;
#pragma unroll
        for (int r = 0; r < DIM; ++r) s.fma(g[el[h]][1 + r * DIM + jj], qd[r][h]);
        vv[jj][h] = df_add(df_mul(Fu[jj + 1][h], co[el[h]][3]), df_mul(df_of(s), co[el[h]][0]));
      }
  }
  if (MODE == 1) {
    if constexpr (ONE) {
      // a thread read exactly these entries of Fs
      df_st2(&Fs[i][j0], pv[0], pv[1]);
#pragma unroll
      for (int jj = 0; jj < DIM; ++jj) df_st2(&Fs[(jj + 1) * NP + i][j0], vv[jj][0], vv[jj][1]);
      __syncthreads();
      for (int t = tid; t < EPB * N; t += NT)
        if (e0 + t / N < mesh.ne) out[e0 * N + t] = dfl_to(Fs[t % N][t / N]);
    } else if (e0 + el[0] < mesh.ne) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t o = ((e0 + el[0]) * N + i) * R + cb + (j0 + h) % (ONE ? 1 : CW);
        out[o] = dfl_to(pv[h]);
#pragma unroll
        for (int jj = 0; jj < DIM; ++jj) out[o + (int64_t)(jj + 1) * NP * R] = dfl_to(vv[jj][h]);
      }
    }
    return;
  }
  // all reads of Tr and rp are past the barrier after the H^{-1} product: reuse them for the face weights
#pragma unroll
  for (int f = 0; f < NFC; ++f) {
    df2 w[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      DfAcc s;
#pragma unroll
      for (int jj = 0; jj < DIM; ++jj) s.fma(g[el[h]][D::ON + f * DIM + jj], vv[jj][h]);
      w[h] = df_add(df_mul(tau, pv[h]), df_of(s));
    }
    df_st2(f < DIM ? &Tr[f * NP + i][j0] : &rp[i][j0], w[0], w[1]);
  }
  __syncthreads();
  for (int t = tid; t < M * HW; t += NT) {
    const int r = t / HW, f = r / NF, j = 2 * (t % HW);
    DfAcc s0, s1;
    sp_row2<WS>(T, RD + r, f < DIM ? &Tr[f * NP][j] : &rp[0][j], s0, s1);
    if constexpr (ONE) {
      df_st2(&ll[r][j], df_mul(g[j][D::OJF + f], df_of(s0)), df_mul(g[j + 1][D::OJF + f], df_of(s1)));
    } else {
      const int q = j / (ONE ? 1 : CW);
      if (e0 + q >= mesh.ne) continue;
      double* o = out + ((e0 + q) * M + r) * R + cb + j % (ONE ? 1 : CW);
      o[0] = dfl_to(df_mul(g[q][D::OJF + f], df_of(s0)));
      o[1] = dfl_to(df_mul(g[q][D::OJF + f], df_of(s1)));
    }
  }
  if constexpr (ONE) {
    __syncthreads();
    for (int t = tid; t < EPB * M; t += NT)
      if (e0 + t / M < mesh.ne) out[e0 * M + t] = dfl_to(ll[t % M][t / M]);
  }
}

}  // namespace hdg
