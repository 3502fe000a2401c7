// Element-local solves of the elastic scheme (uniform and per-element degrees), FP64.
//
// MODE 0: out = C_K A_K^{-1} (F_K - B_K lamD_K) at the element's trace entries; MODE 1: out = u_K =
// A_K^{-1} (F_K - B_K lam_K). F_K = F or alpha Mw_K hist (no sources in the elastic path). With
// Y = C (r_sigma) and Jinv applied on both sides of the derivative matrices,
//   rhs_v = r_v + (1/alpha) sum_r Dr[r] (Jinv[r] Y),   v = H^{-1} rhs_v,
//   sigma = Y / (alpha dJ) - (1/alpha) C sym(Jinv^T Dr^T v).
// What bounds it: FP64 issue (a warp's FP64 instruction holds its SM partition for about 64 cycles). So the
// products with the reference tables run over their nonzero entries (sparse_rows; a row's lanes carry the
// DIM components, rows of like length share a warp), every pointwise step of a mode (compliance, stiffness,
// geometry) is done by one thread in registers from the isotropic form, and no division is left: the
// element coefficients are formed at the condensation. 24,576 tets
// of degrees 1..4: 0.66 ms (1.27 ms with dense tables and a thread per entry); 7,986 tets, k = 2: 0.12 ms
// (0.20 ms).
#pragma once

#include "dflocal.cuh"
#include "elastic.cuh"

namespace hdg {

// volume degree K, face tables of degree KT >= K
template <int DIM, int K, int KT>
struct VdDims {
  static constexpr int NP = Dims<DIM, K>::NP;
  static constexpr int NFP = Dims<DIM, KT>::NF;   // scalar face modes of the padded layout
  static constexpr int NF = DIM * NFP;
  static constexpr int NFC = DIM + 1;
  static constexpr int NT = DIM * (DIM + 1) / 2;
  static constexpr int NV = DIM * NP;
  static constexpr int N = (DIM + NT) * NP;
  static constexpr int M = NFC * NF;
  static constexpr int OJF = 1 + DIM * DIM;
  static constexpr int ON = 1 + DIM * DIM + DIM + 1;
};

// nonzero rows of the reference tables and the order of the rows of group B (see SparseRows)
struct TabsSp : TabsRows<double> {
  const int32_t* permb;
};
__device__ __forceinline__ double sp_row(const TabsSp& T, int row, const double* x) {
  double s = 0.0;
  const int b = __ldg(T.ptr + row + 1);
#pragma unroll 4
  for (int q = __ldg(T.ptr + row); q < b; ++q) {
    const double2 t = __ldg(reinterpret_cast<const double2*>(T.ent + q));
    s += t.x * x[__double2loint(t.y)];
  }
  return s;
}

// Element coefficients: stabilisation s = 2 sqrt(rho mu), alpha rho dJ; the mass matrix of the stress
// alpha dJ times 1/(2 mu) (normal), 1/mu (shear), lam/((DIM lam + 2 mu) 2 mu) (trace); 1/(alpha dJ); lam; mu
constexpr int EL_CO = 8;
static __global__ void local_el_co_kernel(DevMesh mesh, int dim, const double* __restrict__ lamv,
                                          const double* __restrict__ muv, double alpha, double* __restrict__ co) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < mesh.ne; e += (int64_t)gridDim.x * blockDim.x) {
    const double rho = mesh.rho[e], lam = lamv[e], mu = muv[e], ad = alpha * mesh.geo[e * GEO_STRIDE];
    double* o = co + e * EL_CO;
    o[0] = 2.0 * sqrt(rho * mu);
    o[1] = ad * rho;
    o[2] = ad * (1.0 / (2.0 * mu));
    o[3] = ad * (1.0 / mu);
    o[4] = ad * (lam / ((dim * lam + 2.0 * mu) * 2.0 * mu));
    o[5] = 1.0 / ad;
    o[6] = lam;
    o[7] = mu;
  }
}

template <int DIM, int K, int KT>
struct LocalElSmem {
  using D = VdDims<DIM, K, KT>;
  static constexpr int G = 0, NJ = G + GEO_STRIDE, CO = NJ + D::NFC * DIM, LL = CO + EL_CO, FL = LL + D::M,
                       RV = FL + D::NFC * DIM * D::NP, TT = RV + D::NV, RHS = TT + DIM * DIM * D::NP, V = RHS + D::NV,
                       FUSE = V + D::NV, TOTAL = FUSE + 1;
};

// Where an element's fields, H^{-1} and trace entries lie; compact entry a has the padded local index pad(a)
template <int DIM, int K>
struct ElIdxUni {
  using D = VdDims<DIM, K, K>;
  const int32_t* elem_face;
  __device__ __forceinline__ int64_t u0(int64_t e) const { return e * D::N; }
  __device__ __forceinline__ int64_t h0(int64_t e) const { return e * D::NV * D::NV; }
  __device__ __forceinline__ int64_t m0(int64_t e) const { return e * D::M; }
  __device__ __forceinline__ int m(int64_t) const { return D::M; }
  __device__ __forceinline__ int pad(int64_t, int a) const { return a; }
  __device__ __forceinline__ int64_t trace(int64_t e, int64_t, int a) const {
    return (int64_t)elem_face[e * D::NFC + a / D::NF] * D::NF + a % D::NF;
  }
};

// One element by NTH >= NP threads; sm: LocalElSmem::TOTAL doubles.
template <int DIM, int K, int KT, int MODE, int NTH, class IX>
__device__ __forceinline__ void local_el_body(const DevMesh& mesh, const TabsSp& T, const double* __restrict__ coef,
                                              const double* __restrict__ Hinv, double ia, const IX& X, int64_t e,
                                              const double* __restrict__ F, const double* __restrict__ hist,
                                              const double* __restrict__ lamt, double* __restrict__ out, double* sm) {
  using D = VdDims<DIM, K, KT>;
  using SM = LocalElSmem<DIM, K, KT>;
  constexpr int NP = D::NP, NFP = D::NFP, NF = D::NF, NFC = D::NFC, NT = D::NT, NV = D::NV, M = D::M;
  constexpr int RB = NP, RC = RB + DIM * NP, RD = RC + NFC * NP;
  static_assert(NTH >= NP, "one thread per mode");
  double *g = sm + SM::G, *nj = sm + SM::NJ, *co = sm + SM::CO, *ll = sm + SM::LL, *Fl = sm + SM::FL, *rv = sm + SM::RV,
         *tt = sm + SM::TT, *rhs = sm + SM::RHS, *v = sm + SM::V, *z = tt;
  int* fuse = reinterpret_cast<int*>(sm + SM::FUSE);   // faces with a (nonzero) trace, as bits
  const int tid = threadIdx.x;
  const int64_t u0 = X.u0(e), m0 = X.m0(e);
  const int me = X.m(e);
  for (int t = tid; t < GEO_STRIDE; t += NTH) g[t] = mesh.geo[e * GEO_STRIDE + t];
  for (int t = tid; t < NFC * DIM; t += NTH) {
    const double* ge = mesh.geo + e * GEO_STRIDE;
    nj[t] = ge[D::ON + t] * ge[D::OJF + t / DIM];
  }
  for (int t = tid; t < EL_CO; t += NTH) co[t] = coef[e * EL_CO + t];
  for (int t = tid; t < M; t += NTH) ll[t] = 0.0;
  if (tid == 0) {
    int use = 0;
    if (lamt)
      for (int f = 0; f < NFC; ++f)
        if (MODE == 1 || mesh.face_bnd[mesh.elem_face[e * NFC + f]] >= 0) use |= 1 << f;
    *fuse = use;
  }
  __syncthreads();
  const int use = *fuse;
  if (use) {
    for (int a = tid; a < me; a += NTH) {
      const int pc = X.pad(m0, a);
      if ((use >> (pc / NF)) & 1) ll[pc] = lamt[X.trace(e, m0, a)];
    }
    __syncthreads();
    for (int t = tid; t < NFC * NP * DIM; t += NTH) {
      const int p = t % DIM, row = t / DIM, f = row / NP, l = row % NP;
      Fl[(f * DIM + p) * NP + l] = (use >> f) & 1 ? sp_row(T, RC + row, ll + f * NF + p * NFP) : 0.0;
    }
    __syncthreads();
  }
  const double s = co[0];
  const bool mode = tid < NP;   // pointwise steps: thread l holds mode l
  const int l = tid;
  double y[NT];                 // C r_sigma
  if (mode) {
    const double* X0 = (hist ? hist : F) + u0 + l;
    double x[NT], b[DIM][DIM];
#pragma unroll
    for (int a = 0; a < NT; ++a) x[a] = X0[(DIM + a) * NP];
    if (hist) {
      double tr = 0.0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) tr += x[a];
      tr *= co[4];
#pragma unroll
      for (int a = 0; a < NT; ++a) x[a] = a < DIM ? co[2] * x[a] - tr : co[3] * x[a];
    }
    double fv[DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      fv[i] = X0[i * NP];
      if (hist) fv[i] *= co[1];
    }
    if (use) {
      // b[i][j] = sum_f J_F n_fj (F^ lam)_fi
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
        double fl[NFC], bl = 0.0;
#pragma unroll
        for (int f = 0; f < NFC; ++f) {
          fl[f] = Fl[(f * DIM + i) * NP + l];
          bl += g[D::OJF + f] * fl[f];
        }
        fv[i] += s * bl;
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          b[i][j] = 0.0;
#pragma unroll
          for (int f = 0; f < NFC; ++f) b[i][j] += nj[f * DIM + j] * fl[f];
        }
      }
#pragma unroll
      for (int a = 0; a < NT; ++a) {
        int i, j;
        sym_ij<DIM>(a, i, j);
        x[a] += i == j ? b[i][i] : b[i][j] + b[j][i];
      }
    }
    double tr = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) tr += x[a];
    tr *= co[6];
    const double mu = co[7], mu2 = 2.0 * mu;
#pragma unroll
    for (int a = 0; a < NT; ++a) y[a] = a < DIM ? mu2 * x[a] + tr : mu * x[a];
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
      rv[i * NP + l] = fv[i];
#pragma unroll
      for (int r = 0; r < DIM; ++r) {
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < DIM; ++q) acc += g[1 + r * DIM + q] * y[sym_index<DIM>(i, q)];
        tt[(i * DIM + r) * NP + l] = acc;
      }
    }
  }
  __syncthreads();
  for (int t = tid; t < NV; t += NTH) {
    const int i = t % DIM, m = __ldg(T.perm + t / DIM);
    rhs[i * NP + m] = rv[i * NP + m] + ia * sp_row(T, m, tt + i * DIM * NP);
  }
  __syncthreads();
  const double* He = Hinv + X.h0(e);
  for (int t = tid; t < NV; t += NTH) {
    double acc = 0.0;
#pragma unroll 5
    for (int q = 0; q < NV; ++q) acc += He[q * NV + t] * rhs[q];   // H^{-1} symmetric: column read
    v[t] = acc;
  }
  __syncthreads();
  for (int t = tid; t < DIM * NP * DIM; t += NTH) {
    const int p = t % DIM, rl = __ldg(T.permb + t / DIM), r = rl / NP, m = rl % NP;
    z[(r * DIM + p) * NP + m] = sp_row(T, RB + rl, v + p * NP);
  }
  __syncthreads();
  if (mode) {
    double G[DIM][DIM], x[NT];
#pragma unroll
    for (int p = 0; p < DIM; ++p)
#pragma unroll
      for (int q = 0; q < DIM; ++q) {
        G[p][q] = 0.0;
#pragma unroll
        for (int r = 0; r < DIM; ++r) G[p][q] += g[1 + r * DIM + q] * z[(r * DIM + p) * NP + l];
      }
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      int i, j;
      sym_ij<DIM>(a, i, j);
      x[a] = i == j ? G[i][i] : G[i][j] + G[j][i];
    }
    double tr = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) tr += x[a];
    tr *= co[6];
    const double iad = co[5], mu = co[7], mu2 = 2.0 * mu;
#pragma unroll
    for (int a = 0; a < NT; ++a) x[a] = y[a] * iad - ia * (a < DIM ? mu2 * x[a] + tr : mu * x[a]);   // sigma
    double vl[DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i) vl[i] = v[i * NP + l];
    if (MODE == 1) {
#pragma unroll
      for (int i = 0; i < DIM; ++i) out[u0 + i * NP + l] = vl[i];
#pragma unroll
      for (int a = 0; a < NT; ++a) out[u0 + (DIM + a) * NP + l] = x[a];
    } else {
      // weights -s v_i + sum_j n_fj sigma_ij
#pragma unroll
      for (int f = 0; f < NFC; ++f)
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
          double acc = -s * vl[i];
#pragma unroll
          for (int j = 0; j < DIM; ++j) acc += g[D::ON + f * DIM + j] * x[sym_index<DIM>(i, j)];
          Fl[(f * DIM + i) * NP + l] = acc;
        }
    }
  }
  if (MODE == 1) return;
  __syncthreads();
  for (int a = tid; a < me; a += NTH) {
    const int t = X.pad(m0, a);
    const int f = t / NF, i = (t % NF) / NFP, mm = t % NFP;
    out[m0 + a] = g[D::OJF + f] * sp_row(T, RD + f * NFP + mm, Fl + (f * DIM + i) * NP);
  }
}

template <int DIM, int K>
struct LocalElCfg {
  static constexpr int NTH = Dims<DIM, K>::NP <= 10 ? 64 : 128;
};
template <int DIM, int K, int MODE>
__global__ void __launch_bounds__(LocalElCfg<DIM, K>::NTH)
    local_el_kernel(DevMesh mesh, TabsSp T, const double* __restrict__ coef, const double* __restrict__ Hinv, double ia,
                    const double* __restrict__ F, const double* __restrict__ hist, const double* __restrict__ lamt,
                    double* __restrict__ out) {
  __shared__ __align__(16) double sm[LocalElSmem<DIM, K, K>::TOTAL];
  local_el_body<DIM, K, K, MODE, LocalElCfg<DIM, K>::NTH>(mesh, T, coef, Hinv, ia, ElIdxUni<DIM, K>{mesh.elem_face},
                                                          blockIdx.x, F, hist, lamt, out, sm);
}

}  // namespace hdg
