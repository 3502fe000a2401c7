// Element-local post-processing of the acoustic pressure into P_{k+1} (the local, superconvergent
// post-processing step of HDG methods named in Sec. 1; acoustic reading of the standard one).
//
// Per element K with fields p (degree k, orthonormal phi) and traces lam_f on its faces:
//   q_h in [P_k(K)]^d is the discrete gradient of the local momentum equation,
//     (q_h, r)_K = -(p, div r)_K + <lam, r.n>_dK, mass |det J| I, so
//     q^j = -sum_r Jinv[r][j] Dr[r]^T p + (1/|det J|) sum_f n_f,j J_F,f Ff[f] lam_f;
//   p* in P_{k+1}(K) (orthonormal psi) solves (grad p*, grad psi_i)_K = (q_h, grad psi_i)_K for
//   i >= 1, both sides divided by |det J|:
//     A_il = sum_{r,s} (Jinv Jinv^T)[r][s] K1[r][s][i][l],  b_i = sum_{j,r} Jinv[r][j] (E1[r] q^j)_i;
//   the mean condition (p*, 1)_K = (p, 1)_K fixes the constant mode: p*_0 = p_0 (psi_0 = phi_0),
//   and psi_0 has no gradient, so A' c' = b' on the modes 1..Np1-1 (SPD) gives the rest.
// FP64 throughout: the step runs once per output time.
//
// What bounds it: FP64 issue. A warp's FP64 instruction occupies its SM partition for about 64
// cycles however many lanes are active, so the split is chosen by how many lanes the triangular
// loops keep busy: EPW = 4 elements per warp, LPE = 8 lanes each, which also shares the
// reciprocal square root of a Cholesky column among four elements. A' (lower triangle, packed
// by rows, so that as many warps as possible are resident) carries b' as one more row: the
// left-looking column loop then does the forward substitution too, with every partial sum in a
// register. The gradient q_h is never formed: with G = Jinv Jinv^T,
//   sum_j Jinv[r][j] q^j = sum_f nf[f][r] s_f - sum_s G[r][s] t_s,   t_s = Dr[s]^T p, s_f = Ff[f] lam_f,
//   nf[f][r] = J_F,f / |det J| sum_j Jinv[r][j] n_f,j,
// so each table product is formed once instead of once per component, and G symmetric halves
// the off-diagonal K1 terms. 118,098 tets, k = 3: 4.23 ms (23.4 ms with one warp per element,
// the component-wise products and a right-looking update of the square A'); the FP64 multiply-adds
// alone, with no idle lane, would take 2.9 ms.
#pragma once

#include "kernels.cuh"

namespace hdg {

struct PostTabs {
  const double* K1;   // [NS][NA (NA + 1) / 2] rows of the lower triangle, modes 1..Np1-1; the
                      // NS = dim (dim + 1) / 2 blocks are K1[r][r], then K1[r][s] + K1[s][r], r < s
  const double* E1;   // [dim][Np][NA] E1[r] transposed, modes 1..Np1-1 (constant mode left out)
};

template <int DIM, int K>
struct PostCfg {
  static constexpr int NP = Dims<DIM, K>::NP;
  static constexpr int NP1 = Dims<DIM, K + 1>::NP;
  static constexpr int NA = NP1 - 1;
  static constexpr int NS = DIM * (DIM + 1) / 2;
  static constexpr int NR = NA + 1;                    // rows of A' and b'
  static constexpr int LPE = 8, EPW = 32 / LPE;
  static constexpr int TM = (NR + LPE - 1) / LPE;      // rows per lane, at most
  static constexpr int AP = NR * (NR + 1) / 2;
  // doubles per element: A' | b' (first p, lam, s), t, metric; = 8 mod 16, so that the four
  // elements' equal offsets lie in two bank groups, the least for 32 eight-byte accesses
  static constexpr int SM0 = AP + DIM * NP + 32;
  static constexpr int SM_E = SM0 + (24 - SM0 % 16) % 16;
  static constexpr size_t SMEM = sizeof(double) * EPW * SM_E;
  static_assert(NP + (DIM + 1) * (Dims<DIM, K>::NF + NP) <= AP, "p, lam and s fit the A' area");
  static_assert(SM_E % 16 == 8 && SM_E >= SM0, "element stride");
};

// Column j of the packed left-looking Cholesky: rows j + lane + 8 t, t < TN (rows past the last
// one read the last row's entries and store nothing).
template <int TN, int LPE>
__device__ __forceinline__ void post_column(double* A, int j, int nr, int lane) {
  int off[TN];
  double acc[TN];
#pragma unroll
  for (int t = 0; t < TN; ++t) {
    const int i = min(j + lane + LPE * t, nr - 1);
    off[t] = i * (i + 1) / 2;
    acc[t] = A[off[t] + j];
  }
  const double* Aj = A + j * (j + 1) / 2;
#pragma unroll 4
  for (int l = 0; l < j; ++l) {
    const double v = Aj[l];
#pragma unroll
    for (int t = 0; t < TN; ++t) acc[t] -= A[off[t] + l] * v;
  }
  const double r = rsqrt(__shfl_sync(0xffffffffu, acc[0], 0, LPE));   // 1 / L[j][j], kept in place of it
#pragma unroll
  for (int t = 0; t < TN; ++t) {
    const int i = j + lane + LPE * t;
    if (i < nr) A[off[t] + j] = i == j ? r : acc[t] * r;
  }
}

// One warp per CTA (all synchronisation by __syncwarp), four elements at a time.
template <int DIM, int K>
__global__ void __launch_bounds__(32) post_kernel(DevMesh mesh, Tabs T, PostTabs P, const double* __restrict__ u,
                                                  const double* __restrict__ lam, double* __restrict__ pstar) {
  using D = Dims<DIM, K>;
  using C = PostCfg<DIM, K>;
  constexpr int NP = C::NP, NF = D::NF, NFC = D::NFC, N = D::N, NP1 = C::NP1, NA = C::NA, NS = C::NS, LPE = C::LPE;
  extern __shared__ __align__(16) double psm[];
  const int lane = threadIdx.x % LPE, sub = threadIdx.x / LPE;
  double* A = psm + sub * C::SM_E;       // packed rows of A', then b'
  double* t = A + C::AP;                 // t_r [DIM][NP], then sum_j Jinv[r][j] q^j
  double* gm = t + DIM * NP;             // G [DIM][DIM] | nf [NFC][DIM]
  double* p = A;                         // [NP], and behind it
  double* lf = p + NP;                   // [NFC][NF]
  double* sf = lf + NFC * NF;            // [NFC][NP]
  for (int64_t e0 = (int64_t)blockIdx.x * C::EPW; e0 < mesh.ne; e0 += (int64_t)gridDim.x * C::EPW) {
    const bool live = e0 + sub < mesh.ne;
    const int64_t e = live ? e0 + sub : e0;   // a group past the end repeats the first one's work
    const double* ge = mesh.geo + e * GEO_STRIDE;
    for (int i = lane; i < NP; i += LPE) p[i] = u[e * N + i];
    for (int i = lane; i < NFC * NF; i += LPE) lf[i] = lam[(int64_t)mesh.elem_face[e * NFC + i / NF] * NF + i % NF];
    for (int i = lane; i < DIM * DIM; i += LPE) {
      double v = 0.0;
      for (int j = 0; j < DIM; ++j) v += ge[1 + (i / DIM) * DIM + j] * ge[1 + (i % DIM) * DIM + j];
      gm[i] = v;
    }
    const double idj = 1.0 / ge[0];
    for (int i = lane; i < NFC * DIM; i += LPE) {
      const int f = i / DIM, r = i % DIM;
      double v = 0.0;
      for (int j = 0; j < DIM; ++j) v += ge[1 + r * DIM + j] * ge[D::ON + f * DIM + j];
      gm[DIM * DIM + i] = v * ge[D::OJF + f] * idj;
    }
    __syncwarp();
    const double p0 = p[0];
    for (int o = lane; o < DIM * NP; o += LPE) {
      const int r = o / NP, i = o % NP;
      double s = 0.0;
#pragma unroll 4
      for (int l = 0; l < NP; ++l) s += T.Dr[(r * NP + l) * NP + i] * p[l];
      t[o] = s;
    }
    for (int o = lane; o < NFC * NP; o += LPE) {
      const int f = o / NP;
      double s = 0.0;
#pragma unroll
      for (int m = 0; m < NF; ++m) s += T.Ff[o * NF + m] * lf[f * NF + m];
      sf[o] = s;
    }
    __syncwarp();
    for (int i = lane; i < NP; i += LPE) {
      double tv[DIM], sv[NFC];
#pragma unroll
      for (int s = 0; s < DIM; ++s) tv[s] = t[s * NP + i];
#pragma unroll
      for (int f = 0; f < NFC; ++f) sv[f] = sf[f * NP + i];
#pragma unroll
      for (int r = 0; r < DIM; ++r) {
        double v = 0.0;
#pragma unroll
        for (int f = 0; f < NFC; ++f) v += gm[DIM * DIM + f * DIM + r] * sv[f];
#pragma unroll
        for (int s = 0; s < DIM; ++s) v -= gm[r * DIM + s] * tv[s];
        t[r * NP + i] = v;
      }
    }
    __syncwarp();
    // b' into the last row, A' into the rows above it
    double* bv = A + NA * (NA + 1) / 2;
    for (int i = lane; i < NA; i += LPE) {
      double s = 0.0;
#pragma unroll 4
      for (int rl = 0; rl < DIM * NP; ++rl) s += P.E1[rl * NA + i] * t[rl];
      bv[i] = s;
    }
    double gs[NS];
    {
      int c = DIM;
#pragma unroll
      for (int r = 0; r < DIM; ++r) {
        gs[r] = gm[r * DIM + r];
#pragma unroll
        for (int s = r + 1; s < DIM; ++s) gs[c++] = gm[r * DIM + s];
      }
    }
    constexpr int NL = NA * (NA + 1) / 2;
    for (int o = lane; o < NL; o += LPE) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < NS; ++c) s += gs[c] * P.K1[c * NL + o];
      A[o] = s;
    }
    __syncwarp();
    // Cholesky A' = L L^T with the row b': y = L^{-1} b' appears in its place
    for (int j = 0; j < NA; ++j) {
      switch ((C::NR - j + LPE - 1) / LPE) {   // rows per lane still in play
        case 1: post_column<1, LPE>(A, j, C::NR, lane); break;
        case 2: post_column<C::TM < 2 ? C::TM : 2, LPE>(A, j, C::NR, lane); break;
        case 3: post_column<C::TM < 3 ? C::TM : 3, LPE>(A, j, C::NR, lane); break;
        case 4: post_column<C::TM < 4 ? C::TM : 4, LPE>(A, j, C::NR, lane); break;
        case 5: post_column<C::TM < 5 ? C::TM : 5, LPE>(A, j, C::NR, lane); break;
        case 6: post_column<C::TM < 6 ? C::TM : 6, LPE>(A, j, C::NR, lane); break;
        default: post_column<C::TM, LPE>(A, j, C::NR, lane); break;
      }
      __syncwarp();
    }
    // L^T c' = y, column by column
    for (int i = NA - 1; i >= 0; --i) {
      const double* Li = A + i * (i + 1) / 2;
      const double ci = bv[i] * Li[i];
      __syncwarp();
      if (lane == 0) bv[i] = ci;
      for (int l = lane; l < i; l += LPE) bv[l] -= Li[l] * ci;
      __syncwarp();
    }
    if (live)
      for (int i = lane; i < NP1; i += LPE) pstar[e * NP1 + i] = i == 0 ? p0 : bv[i - 1];
    __syncwarp();
  }
}

}  // namespace hdg
