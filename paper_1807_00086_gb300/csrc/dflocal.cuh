// Element-local solves of the acoustic scheme (Sec. 2.4, Eq. LS, the element blocks of the condensed
// system): MODE 0 forms gslot = C_K A_K^{-1} (F_K - B_K lamD_K), MODE 1 recovers
// u_K = A_K^{-1} (F_K - B_K lam_K). Arithmetic AR: FP64 (ArF64), or double-float on the FP32 pipe (ArDf, the
// mixed modes): every product and sum is carried as an unevaluated pair hi + lo of floats (about 48
// significant bits), products by fmaf-based exact splitting (Dekker's two-product), sums by Knuth's two-sum,
// so the results agree with FP64 to a few units of 1e-14 relative while the work runs on the FP32 units
// (FP64 issues at a small fraction of the FP32 rate on this GPU).
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
template <class T>
struct alignas(16) SpEnt {
  T v;
  int idx, pad;
};
template <class T>
struct TabsRows {
  const SpEnt<T>* ent;
  const int32_t *ptr, *perm;
};

// Packed FP32 pairs (one instruction for two columns): half of the issue slots of the scalar forms, the
// same bits. sub: b * -1 + a, one rounding.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float a, float b) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ float2 unpk(f32x2 v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ f32x2 pk_mul(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 pk_add(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 pk_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ f32x2 pk_neg(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 pk_sub(f32x2 a, f32x2 b) { return pk_fma(b, 0xbf800000bf800000ull, a); }

// Arithmetic of two neighbouring columns: T one value (8 bytes), P a pair, Acc a pair of running sums. A
// pair lies at &X[row][even column]: for ArDf as (h, h', l, l').
struct ArDf {
  using T = df2;
  struct P {
    f32x2 h, l;
  };
  // the operations of DfAcc, df_mul, df_add, df_two_sum
  struct Acc {
    f32x2 s = 0, c = 0;
    __device__ __forceinline__ void fma(P a, P b) {
      const f32x2 p = pk_mul(a.h, b.h);
      const f32x2 e = pk_fma(a.h, b.l, pk_fma(a.l, b.h, pk_fma(a.h, b.h, pk_neg(p))));
      const f32x2 t = pk_add(s, p), bb = pk_sub(t, s);
      c = pk_add(c, pk_add(pk_add(pk_sub(s, pk_sub(t, bb)), pk_sub(p, bb)), e));
      s = t;
    }
  };
  static __device__ __forceinline__ T from(double x) { return dfl_from(x); }
  static __device__ __forceinline__ double to(T x) { return dfl_to(x); }
  static __device__ __forceinline__ T round(double x) { return df_from(x); }
  static __device__ __forceinline__ T mul1(T a, T b) { return df_mul(a, b); }
  static __device__ __forceinline__ P pair(T a, T b) { return {pk(a.h, b.h), pk(a.l, b.l)}; }
  static __device__ __forceinline__ T first(P x) { return {unpk(x.h).x, unpk(x.l).x}; }
  static __device__ __forceinline__ T second(P x) { return {unpk(x.h).y, unpk(x.l).y}; }
  static __device__ __forceinline__ P ld(const T* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
  }
  static __device__ __forceinline__ void st(T* p, P x) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(x.h, x.l); }
  static __device__ __forceinline__ void set(T* row, int col, T x) {
    float* f = reinterpret_cast<float*>(row + (col & ~1)) + (col & 1);
    f[0] = x.h;
    f[2] = x.l;
  }
  static __device__ __forceinline__ T get(const T* row, int col) {
    const float* f = reinterpret_cast<const float*>(row + (col & ~1)) + (col & 1);
    return {f[0], f[2]};
  }
  static __device__ __forceinline__ P two_sum(f32x2 a, f32x2 b) {
    const f32x2 s = pk_add(a, b), bb = pk_sub(s, a);
    return {s, pk_add(pk_sub(a, pk_sub(s, bb)), pk_sub(b, bb))};
  }
  static __device__ __forceinline__ P of(const Acc& a) { return two_sum(a.s, a.c); }
  static __device__ __forceinline__ P mul(P a, P b) {
    const f32x2 p = pk_mul(a.h, b.h);
    const f32x2 e = pk_fma(a.h, b.l, pk_fma(a.l, b.h, pk_fma(a.h, b.h, pk_neg(p))));
    const f32x2 s = pk_add(p, e);
    return {s, pk_sub(e, pk_sub(s, p))};
  }
  static __device__ __forceinline__ P add(P a, P b) {
    const P s = two_sum(a.h, b.h);
    const f32x2 err = pk_add(s.l, pk_add(a.l, b.l)), h = pk_add(s.h, err);
    return {h, pk_sub(err, pk_sub(h, s.h))};
  }
  static __device__ __forceinline__ P sub(P a, P b) { return add(a, {pk_neg(b.h), pk_neg(b.l)}); }
};
struct ArF64 {
  using T = double;
  struct P {
    double a, b;
  };
  struct Acc {
    double a = 0.0, b = 0.0;
    __device__ __forceinline__ void fma(P x, P y) {
      a += x.a * y.a;
      b += x.b * y.b;
    }
  };
  static __device__ __forceinline__ T from(double x) { return x; }
  static __device__ __forceinline__ double to(T x) { return x; }
  static __device__ __forceinline__ T round(double x) { return x; }
  static __device__ __forceinline__ T mul1(T a, T b) { return a * b; }
  static __device__ __forceinline__ P pair(T a, T b) { return {a, b}; }
  static __device__ __forceinline__ T first(P x) { return x.a; }
  static __device__ __forceinline__ T second(P x) { return x.b; }
  static __device__ __forceinline__ P ld(const T* p) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return {v.x, v.y};
  }
  static __device__ __forceinline__ void st(T* p, P x) { *reinterpret_cast<double2*>(p) = make_double2(x.a, x.b); }
  static __device__ __forceinline__ void set(T* row, int col, T x) { row[col] = x; }
  static __device__ __forceinline__ T get(const T* row, int col) { return row[col]; }
  static __device__ __forceinline__ P of(const Acc& a) { return {a.a, a.b}; }
  static __device__ __forceinline__ P mul(P x, P y) { return {x.a * y.a, x.b * y.b}; }
  static __device__ __forceinline__ P add(P x, P y) { return {x.a + y.a, x.b + y.b}; }
  static __device__ __forceinline__ P sub(P x, P y) { return {x.a - y.a, x.b - y.b}; }
};

// table row times two neighbouring columns of x (rows WS apart)
template <class AR, int WS>
__device__ __forceinline__ typename AR::P sp_row2(const TabsRows<typename AR::T>& T, int row, const typename AR::T* x) {
  typename AR::Acc s;
  const int b = __ldg(T.ptr + row + 1);
#pragma unroll 4
  for (int q = __ldg(T.ptr + row); q < b; ++q) {
    const int4 u = __ldg(reinterpret_cast<const int4*>(T.ent + q));
    const SpEnt<typename AR::T> t = *reinterpret_cast<const SpEnt<typename AR::T>*>(&u);
    s.fma(AR::pair(t.v, t.v), AR::ld(x + t.idx * WS));
  }
  return AR::of(s);
}

// Element coefficients of the local solves at the mass shift alpha: 1/b, a' dJ, b dJ, 1/(b dJ) with
// b = alpha rho, a' = alpha/(rho c^2); formed once per condensation, because an FP64 division by one
// thread of a CTA holds its SM partition as long as a full warp's
template <class AR>
__global__ void local_co_kernel(DevMesh mesh, double alpha, typename AR::T* __restrict__ co) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < mesh.ne; e += (int64_t)gridDim.x * blockDim.x) {
    const double rho = mesh.rho[e], cc = mesh.c[e], dJ = mesh.geo[e * GEO_STRIDE];
    const double b = alpha * rho, ap = alpha / (rho * cc * cc);
    co[4 * e] = AR::round(1.0 / b);
    co[4 * e + 1] = AR::round(ap * dJ);
    co[4 * e + 2] = AR::round(b * dJ);
    co[4 * e + 3] = AR::round(1.0 / (b * dJ));
  }
}

// One kernel for one column (CW = 0) and for column blocks (the multi-source and serving batches, CW =
// min(R, 16) columns of EPB elements per CTA). Every array is [row][W] with the W columns of the CTA:
// its elements, or (element, right-hand side) pairs. A thread holds row i of two neighbouring columns, so
// that one table entry serves two products and one 16-byte read both of their factors; lanes run over the
// columns first, so that the rows of a warp are few and of like length. H^{-1}, which differs by element,
// is read along its rows instead. One column: F, the history and the results pass through shared memory,
// so that the global accesses are contiguous.
// What bounds it: FP64 issue (ArF64), or the issue of the double-float products (11 packed instructions for
// two columns) and of the pointwise steps. Modes 0 / 1: ArF64, 41,154 tets, k = 2: 0.094 / 0.088 ms (0.20 /
// 0.18 with dense tables and divisions in every thread); ArDf, k = 3: 24,576 tets x 64 columns 2.8 / 3.7 ms
// (5.1 / 4.9 with dense tables, 3.3 / 4.1 with scalar instructions), 16,464 x 4 columns 0.16 / 0.17 ms (0.24).
template <int DIM, int K, int CW>
struct LocalCfg {
  static constexpr int NP = Dims<DIM, K>::NP;
  static constexpr bool ONE = CW == 0;
  static constexpr int PE = NP * (ONE ? 1 : CW) / 2;          // threads per element of a column block
  static constexpr int EPB = ONE ? (NP <= 10 ? 32 : NP <= 20 ? 16 : 8) : PE >= 160 ? 1 : 160 / PE;
  static constexpr int W = ONE ? EPB : EPB * CW;
  static constexpr int WS = ONE ? W + 2 : W;                  // padded where rows are filled column by column
  static constexpr int HW = W / 2;                            // threads per row
  static constexpr int NT = NP * HW;
};

template <class AR, int DIM, int K, int MODE, int CW>
__global__ void __launch_bounds__(LocalCfg<DIM, K, CW>::NT)
    local_kernel(DevMesh mesh, TabsRows<typename AR::T> T, const typename AR::T* __restrict__ geo,
                 const typename AR::T* __restrict__ coef, const typename AR::T* __restrict__ Hinv, typename AR::T tau, int R,
                 const double* __restrict__ F,
                    const double* __restrict__ hist, SrcArgs src, const double* __restrict__ lam, double* __restrict__ out) {
  using D = Dims<DIM, K>;
  using L = LocalCfg<DIM, K, CW>;
  using V = typename AR::T;
  using P = typename AR::P;
  using Acc = typename AR::Acc;
  constexpr int NP = D::NP, NF = D::NF, M = D::M, NFC = D::NFC, N = D::N, EPB = L::EPB, NT = L::NT, WS = L::WS, HW = L::HW;
  constexpr int RB = NP, RC = RB + DIM * NP, RD = RC + NFC * NP;
  constexpr bool ONE = L::ONE;
  // columns of the geometry (each element twice in a block), padded as the rows that are filled column by column
  constexpr int CD = ONE ? 1 : CW, GW = ONE ? EPB : 2 * EPB, GS = ONE ? GW + 2 : GW;
  __shared__ __align__(16) V g[GEO_STRIDE][GS], co[4][GS], nj[NFC * DIM][GS];   // nj: J_F n_f
  __shared__ __align__(16) V Fs[ONE ? N : 1][WS];     // one column: F or history, then u
  __shared__ __align__(16) V Tr[DIM * NP][WS];        // the face weights w_f (f < DIM) in MODE 0
  __shared__ __align__(16) V rp[NP][WS];              // the last face's weights in MODE 0
  __shared__ __align__(16) V pp[NP][WS];
  __shared__ __align__(16) V ll[M][WS];               // traces; one column, MODE 0: then the result
  __shared__ int anyf[EPB];                           // faces with a (nonzero) trace, as bits
  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int cb = ONE ? 0 : blockIdx.y * CW;
  for (int t = tid; t < GEO_STRIDE * GW; t += NT) {
    const int x = ONE ? t % GEO_STRIDE : (t / 2) % GEO_STRIDE, q = ONE ? t / GEO_STRIDE : t / (2 * GEO_STRIDE);
    AR::set(g[x], ONE ? q : 2 * q + (t & 1), e0 + q < mesh.ne ? geo[(e0 + q) * GEO_STRIDE + x] : V{});
  }
  for (int t = tid; t < NFC * DIM * GW; t += NT) {
    const int x = t / GW, cc = t % GW;
    const int64_t e = e0 + (ONE ? cc : cc / 2);
    const V* ge = geo + e * GEO_STRIDE;
    AR::set(nj[x], cc, e < mesh.ne ? AR::mul1(ge[D::ON + x], ge[D::OJF + x / DIM]) : V{});
  }
  for (int t = tid; t < 4 * GW; t += NT) {
    const int64_t e = e0 + (ONE ? t / 4 : t / 8);
    AR::set(co[t % 4], t / 4, e < mesh.ne ? coef[4 * e + t % 4] : V{});
  }
  for (int q = tid; q < EPB; q += NT) {
    int use = 0;
    if (e0 + q < mesh.ne && lam)
      for (int f = 0; f < NFC; ++f)
        if (MODE == 1 || mesh.face_bnd[mesh.elem_face[(e0 + q) * NFC + f]] >= 0) use |= 1 << f;
    anyf[q] = use;
  }
  if (lam)
    for (int t = tid; t < M * L::W; t += NT) {
      const int q = ONE ? t / M : t / (M * CD), r = ONE ? t % M : (t / CD) % M, jc = ONE ? 0 : t % CD;
      const int64_t e = e0 + q;
      double v = 0.0;
      if (e < mesh.ne) {
        const int f = mesh.elem_face[e * NFC + r / NF];
        if ((MODE == 1) || (mesh.face_bnd[f] >= 0)) v = lam[((int64_t)f * NF + r % NF) * R + cb + jc];
      }
      AR::set(ll[r], ONE ? q : q * CD + jc, AR::from(v));
    }
  if constexpr (ONE) {
    const double* X = hist ? hist : F;
    for (int t = tid; t < EPB * N; t += NT) AR::set(Fs[t % N], t / N, AR::from(e0 + t / N < mesh.ne ? X[e0 * N + t] : 0.0));
  }
  __syncthreads();
  const int i = __ldg(T.perm + tid / HW), j0 = 2 * (tid % HW);
  const int el[2] = {ONE ? j0 : j0 / CD, ONE ? j0 + 1 : j0 / CD};
  const int gc = ONE ? j0 : 2 * el[0];   // the pair's geometry column
  const P tau2 = AR::pair(tau, tau);
  // row i of F~ for all components (+ the F^ lam face products it needs)
  P Fu[DIM + 1];
  {
    const int use = anyf[el[0]] | anyf[el[1]];
    P Fl[NFC];
    if (use)
#pragma unroll
      for (int f = 0; f < NFC; ++f)
        Fl[f] = (use >> f) & 1 ? sp_row2<AR, WS>(T, RC + f * NP + i, &ll[f * NF][j0]) : AR::pair(V{}, V{});
#pragma unroll
    for (int comp = 0; comp <= DIM; ++comp) {
      P v;
      if constexpr (ONE) {
        v = AR::ld(&Fs[comp * NP + i][j0]);
      } else {
        V x[2] = {V{}, V{}};
        if (e0 + el[0] < mesh.ne) {
          const double* X = (hist ? hist : F) + ((e0 + el[0]) * N + comp * NP + i) * R + cb + j0 % CD;
          x[0] = AR::from(X[0]);
          x[1] = AR::from(X[1]);
        }
        v = AR::pair(x[0], x[1]);
      }
      if (hist) {
        v = AR::mul(AR::ld(&co[comp == 0 ? 1 : 2][gc]), v);
        if (comp == 0 && src.ptr) {
          double sv[2] = {0.0, 0.0};
          bool any = false;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int64_t e = e0 + el[h];
            if (e < mesh.ne)
              for (int q = src.ptr[e]; q < src.ptr[e + 1]; ++q)
                if (ONE || src.col[q] == cb + j0 % CD + h) {
                  sv[h] += ricker_at(src, q) * src.phi[(int64_t)q * NP + i];
                  any = true;
                }
          }
          if (any) v = AR::add(v, AR::pair(AR::round(sv[0]), AR::round(sv[1])));
        }
      }
      if (use) {
        Acc bl;
#pragma unroll
        for (int f = 0; f < NFC; ++f)
          bl.fma(comp == 0 ? AR::ld(&g[D::OJF + f][gc]) : AR::ld(&nj[f * DIM + (comp == 0 ? 0 : comp - 1)][gc]), Fl[f]);
        v = comp == 0 ? AR::add(v, AR::mul(tau2, AR::of(bl))) : AR::sub(v, AR::of(bl));
      }
      Fu[comp] = v;
    }
  }
#pragma unroll
  for (int r = 0; r < DIM; ++r) {
    Acc s;
#pragma unroll
    for (int jj = 0; jj < DIM; ++jj) s.fma(AR::ld(&g[1 + r * DIM + jj][gc]), Fu[jj + 1]);
    AR::st(&Tr[r * NP + i][j0], AR::of(s));
  }
  __syncthreads();
  const P ib = AR::ld(&co[0][gc]);
  AR::st(&rp[i][j0], AR::sub(Fu[0], AR::mul(sp_row2<AR, WS>(T, i, &Tr[0][j0]), ib)));
  __syncthreads();
  {
    // p = H^{-1} rp; H^{-1} is symmetric, so row i is read as column i
    constexpr int HC = ONE ? 1 : CW / 2;
    const int q = tid / (NP * HC), i2 = (tid / HC) % NP, j2 = ONE ? 2 * q : q * CW + 2 * (tid % HC);
    const int64_t ea = e0 + (ONE ? 2 * q : q);
    const V* Ha = Hinv + (ea < mesh.ne ? ea : 0) * (int64_t)(NP * NP) + i2;
    const V* Hb = ONE ? Hinv + (ea + 1 < mesh.ne ? ea + 1 : 0) * (int64_t)(NP * NP) + i2 : Ha;
    Acc s;
#pragma unroll 5
    for (int l = 0; l < NP; ++l) {
      const V ha = Ha[l * NP];
      s.fma(AR::pair(ha, ONE ? Hb[l * NP] : ha), AR::ld(&rp[l][j2]));
    }
    AR::st(&pp[i2][j2], AR::of(s));
  }
  __syncthreads();
  const P pv = AR::ld(&pp[i][j0]);
  P vv[DIM];
  {
    P qd[DIM];
#pragma unroll
    for (int r = 0; r < DIM; ++r) qd[r] = sp_row2<AR, WS>(T, RB + r * NP + i, &pp[0][j0]);
    const P ibd = AR::ld(&co[3][gc]);
#pragma unroll
    for (int jj = 0; jj < DIM; ++jj) {
      Acc s;
#pragma unroll
      for (int r = 0; r < DIM; ++r) s.fma(AR::ld(&g[1 + r * DIM + jj][gc]), qd[r]);
      vv[jj] = AR::add(AR::mul(Fu[jj + 1], ibd), AR::mul(AR::of(s), ib));
    }
  }
  if (MODE == 1) {
    if constexpr (ONE) {
      // a thread read exactly these entries of Fs
      AR::st(&Fs[i][j0], pv);
#pragma unroll
      for (int jj = 0; jj < DIM; ++jj) AR::st(&Fs[(jj + 1) * NP + i][j0], vv[jj]);
      __syncthreads();
      for (int t = tid; t < EPB * N; t += NT)
        if (e0 + t / N < mesh.ne) out[e0 * N + t] = AR::to(AR::get(Fs[t % N], t / N));
    } else if (e0 + el[0] < mesh.ne) {
      double* o = out + ((e0 + el[0]) * N + i) * R + cb + j0 % CD;
      o[0] = AR::to(AR::first(pv));
      o[1] = AR::to(AR::second(pv));
#pragma unroll
      for (int jj = 0; jj < DIM; ++jj) {
        o += (int64_t)NP * R;
        o[0] = AR::to(AR::first(vv[jj]));
        o[1] = AR::to(AR::second(vv[jj]));
      }
    }
    return;
  }
  // all reads of Tr and rp are past the barrier after the H^{-1} product: reuse them for the face weights
  const P tp = AR::mul(tau2, pv);
#pragma unroll
  for (int f = 0; f < NFC; ++f) {
    Acc s;
#pragma unroll
    for (int jj = 0; jj < DIM; ++jj) s.fma(AR::ld(&g[D::ON + f * DIM + jj][gc]), vv[jj]);
    AR::st(f < DIM ? &Tr[f * NP + i][j0] : &rp[i][j0], AR::add(tp, AR::of(s)));
  }
  __syncthreads();
  for (int t = tid; t < M * HW; t += NT) {
    const int r = t / HW, f = r / NF, j = 2 * (t % HW);
    const P y = AR::mul(AR::ld(&g[D::OJF + f][ONE ? j : 2 * (j / CD)]),
                        sp_row2<AR, WS>(T, RD + r, f < DIM ? &Tr[f * NP][j] : &rp[0][j]));
    if constexpr (ONE) {
      AR::st(&ll[r][j], y);
    } else {
      const int q = j / CD;
      if (e0 + q >= mesh.ne) continue;
      double* o = out + ((e0 + q) * M + r) * R + cb + j % CD;
      o[0] = AR::to(AR::first(y));
      o[1] = AR::to(AR::second(y));
    }
  }
  if constexpr (ONE) {
    __syncthreads();
    for (int t = tid; t < EPB * M; t += NT)
      if (e0 + t / M < mesh.ne) out[e0 * M + t] = AR::to(AR::get(ll[t % M], t / M));
  }
}

}  // namespace hdg
