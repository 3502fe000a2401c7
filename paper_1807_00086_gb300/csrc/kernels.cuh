// Device kernels of the FP64 HDG hot path (sm_103a).
//
// Per element K with affine map x = X0 + J xi, |det J| = dJ, the acoustic local blocks
// are (Sec. 2.4, Eq. LS, acoustic specialisation of Eqs. eq:HDG_linelas1-5):
//   A_K = [ a dJ I + tau sum_f E_f    Dx_1 .. Dx_d ]      a = alpha/(rho c^2)
//         [ -Dx_j^T                   b dJ I       ]      b = alpha rho
//   B_K: p rows -tau F_f, v_j rows n_fj F_f;   C_K = [tau F_f^T, n_fj F_f^T];
//   D_K = -tau J_f I per face,
// with Dx_j = dJ sum_r Jinv[r][j] Dr_r, F_f = J_f Ff_f, E_f = J_f Ff_f Ff_f^T from the
// reference tables. The diagonal velocity block is eliminated analytically, leaving the
// SPD pressure block
//   H = a dJ I + tau sum_f J_f E^_f + (dJ/b) sum_{r,s} (Jinv Jinv^T)_{rs} Dr_r Dr_s^T,
// so A_K^{-1} costs one H^{-1} mat-vec plus derivative-table products, and
//   S_K = Bt^T H^{-1} Bt + D_K - (1/(b dJ)) [J_f J_g (n_f . n_g) Ff_f^T Ff_g]_{fg},
//   Bt_f = -J_f (tau Ff_f + (1/b) sum_r (n_f . Jinv[r]) Dr_r Ff_f).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <type_traits>

#include <cstdint>

#include "mesh.h"

namespace hdg {

struct Tabs {
  const double *Dr, *Ff, *Ef, *Trs, *DFrf, *Pfg;
};

struct DevMesh {
  int64_t ne, nf;
  const double* geo;
  const double* rho;
  const double* c;
  const int32_t* elem_face;
  const int32_t* face_slot;
  const int32_t* face_bnd;
};

// Point sources: CSR by element (ptr[e]..ptr[e+1]), per source the basis values at the
// point times its amplitude (phi), its right-hand-side column and its time delay; the
// Ricker wavelet r(t - delay) = (1 - 2a) exp(-a), a = (pi f0 (t - delay - t0))^2.
struct SrcArgs {
  const int32_t* ptr;
  const double* phi;
  const int32_t* col;
  const double* delay;
  double f0, t0, t;
};

__device__ __forceinline__ double ricker_at(const SrcArgs& s, int q) {
  const double x = 3.14159265358979323846 * s.f0 * (s.t - s.delay[q] - s.t0);
  const double a = x * x;
  return (1.0 - 2.0 * a) * exp(-a);
}

template <int DIM, int K>
struct Dims {
  static constexpr int NP = (DIM == 2) ? (K + 1) * (K + 2) / 2 : (K + 1) * (K + 2) * (K + 3) / 6;
  static constexpr int NF = (DIM == 2) ? (K + 1) : (K + 1) * (K + 2) / 2;
  static constexpr int NFC = DIM + 1;
  static constexpr int N = NFC * NP;
  static constexpr int M = NFC * NF;
  static constexpr int OJF = 1 + DIM * DIM;
  static constexpr int ON = 1 + DIM * DIM + DIM + 1;
};

// Jacobi preconditioner: dinv = sgn / (sum over the face's slots of diag S_K), sgn = -1 for the
// acoustic convention (K negative definite), +1 for the elastic one (K positive definite).
template <class D>
__global__ void diag_kernel(DevMesh mesh, const double* __restrict__ S, double sgn, double* __restrict__ dinv) {
  constexpr int NF = D::NF, M = D::M;
  const int64_t n = mesh.nf * NF;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = t / NF;
    const int mm = (int)(t % NF);
    double d = 0.0;
    if (mesh.face_bnd[f] < 0) {
      for (int s = 0; s < 2; ++s) {
        const int64_t slot = mesh.face_slot[2 * f + s];
        const int64_t e = slot / D::NFC;
        const int r = (int)(slot % D::NFC) * NF + mm;
        d += S[e * (int64_t)(M * M) + (int64_t)r * M + r];
      }
      dinv[t] = sgn / d;
    } else {
      dinv[t] = 0.0;
    }
  }
}

// ---------------------------------------------------------------- matrix-free trace apply (d)
// zslot[e][r] = sum_c S_K[r][c] x_K[c], x gathered from faces (boundary faces read as 0).
// S_K is symmetric, so thread r reads column r (coalesced across the element's threads).
template <class L>
struct ApplyCfg {
  static constexpr int M = L::M;
  static constexpr int EPB = (128 / M) > 0 ? (128 / M) : 1;
  static constexpr int NT = EPB * M;
};

template <class D>
__global__ void __launch_bounds__(ApplyCfg<D>::NT) apply_kernel(DevMesh mesh, const double* __restrict__ S,
                                                                const double* __restrict__ x,
                                                                double* __restrict__ zslot,
                                                                const int* __restrict__ done) {
  using C = ApplyCfg<D>;
  constexpr int NF = D::NF, M = D::M, NFC = D::NFC;
  if (done && *done) return;
  __shared__ double lx[C::EPB][M];
  const int el = threadIdx.x / M, r = threadIdx.x % M;
  const int64_t e = (int64_t)blockIdx.x * C::EPB + el;
  if (e < mesh.ne) {
    const int f = mesh.elem_face[e * NFC + r / NF];
    lx[el][r] = mesh.face_bnd[f] < 0 ? x[(int64_t)f * NF + r % NF] : 0.0;
  }
  __syncthreads();
  if (e < mesh.ne) {
    const double* Se = S + e * (int64_t)(M * M);
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < M; ++c) s += Se[c * M + r] * lx[el][c];
    zslot[e * M + r] = s;
  }
}

// ---------------------------------------------------------------- face passes and PCG
// done: the stop code, for the kernels that follow and the host. halt[parity]: the same for the kernel of
// the iteration with this parity that records the stop code. Its CTA 0 writes the other slot, so no CTA
// reads what its own launch writes: read from `done`, the warps of a late CTA could disagree and part
// at a barrier.
struct CgScal {
  double rho[2];
  double bb, rr, tol2;
  int done, iters;
  int halt[2];
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic block sum of one value per thread (blockDim = 256); result in thread 0.
__device__ __forceinline__ double block_sum256(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < 8; ++i) s += red[i];
  return s;
}

// Inner products of FP32 vectors, accurate to FP64 level but evaluated on the FP32 pipe
// (GB300's FP64 rate is 1/58 of FP32): each product is split exactly into p + e with an
// FMA, and the terms are accumulated in a compensated (s, c) float pair (TwoSum). Only
// the per-thread result is widened to FP64 for the block/grid reduction.
struct Acc2 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x;
    const float bb = t - s;
    c += (s - (t - bb)) + (x - bb);
    s = t;
  }
  __device__ __forceinline__ void dot(float a, float b) {
    const float p = a * b;
    c += fmaf(a, b, -p);
    add(p);
  }
  __device__ __forceinline__ void dot4(float4 a, float4 b) { dot(a.x, b.x); dot(a.y, b.y); dot(a.z, b.z); dot(a.w, b.w); }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
  // both pairs' sum: the heads by TwoSum, as in add; symmetric in its operands
  __device__ __forceinline__ void merge(float s2, float c2) {
    const float t = s + s2;
    const float bb = t - s;
    c = (c + c2) + ((s - (t - bb)) + (s2 - bb));
    s = t;
  }
  // sum over the lanes that differ in the bits lo, 2 lo, .. 16 of their index (every lane: the same)
  __device__ __forceinline__ void warp_merge(int lo = 1) {
    for (int o = 16; o >= lo; o >>= 1) merge(__shfl_xor_sync(0xffffffffu, s, o), __shfl_xor_sync(0xffffffffu, c, o));
  }
};

// a / b of two compensated pairs, rounded to FP32 once (one Newton correction of the heads' quotient)
__device__ __forceinline__ float pair_ratio(float2 a, float2 b) {
  const float q = a.x / b.x;
  const float r = (fmaf(-q, b.x, a.x) + a.y) - q * b.y;
  return q + r / b.x;
}

// Sums of NQ pairs per thread over the CTA (NW warps), to every thread. On the FP32 pipe: an FP64
// instruction holds an SM partition for about 64 cycles, so widening each thread's pairs and adding
// doubles in the tree made the reductions the longest part of the small vector kernels.
template <int NQ, int NW>
__device__ __forceinline__ void block_pairs(Acc2 (&a)[NQ]) {
  __shared__ float2 red[NQ][NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();   // an earlier sum's readers are done
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    a[q].warp_merge();
    if (lane == 0) red[q][w] = make_float2(a[q].s, a[q].c);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    a[q] = Acc2();
#pragma unroll
    for (int i = 0; i < NW; ++i) a[q].merge(red[q][i].x, red[q][i].y);
  }
}
// sums of the partials part[q n + i], i < n, to every thread
template <int NQ, int NW>
__device__ __forceinline__ void sum_pairs(const float2* __restrict__ part, int n, Acc2 (&a)[NQ]) {
  constexpr int U = 4;
#pragma unroll
  for (int q = 0; q < NQ; ++q) a[q] = Acc2();
  for (int i = threadIdx.x; i < n; i += U * 32 * NW) {
    float2 v[NQ][U];   // all loads of a trip before its sums
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int u = 0; u < U; ++u) v[q][u] = i + u * 32 * NW < n ? part[q * n + i + u * 32 * NW] : make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < NQ; ++q) a[q].merge(v[q][u].x, v[q][u].y);
  }
  block_pairs<NQ, NW>(a);
}

// Deterministic sum of a partials array (same order in every block); result in all threads.
__device__ __forceinline__ double reduce_partials(const double* __restrict__ part, int n, int stride, double* red) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += part[(int64_t)i * stride];
  v = block_sum256(v, red);
  __shared__ double bc;
  if (threadIdx.x == 0) bc = v;
  __syncthreads();
  return bc;
}

// a / b by one thread for the CTA (once per kernel): by every thread of a full SM an FP64 division takes
// about 4 us of its FP64 pipe
__device__ __forceinline__ double cta_ratio(double a, double b) {
  __shared__ double r;
  if (threadIdx.x == 0) r = a / b;
  __syncthreads();
  return r;
}

// Scalars of an FP32 inner solve whose iteration is two kernels: A multiplies every element block by
// its direction p_K = z_K + beta p_K, formed in the gather, and leaves block partials of (p, S p);
// B forms alpha from them, advances p, x, r, z and leaves partials of (r, z) and (r, r), from which
// the next A takes beta and the convergence test. Every CTA of a kernel sums the partials it needs
// itself, in the same order, as compensated FP32 pairs; CTA 0 alone records the state, in the slot
// of the other iteration parity, so that no CTA reads what it writes. A small system's iteration is
// bounded by the latency of its dependent kernels and of their sums: 16,562 triangles, k = 3: 9.2 us
// (21.0 us as apply, update and direction with FP64 sums). The pairs of a thread were summed in FP64 there: an error of
// 1e-16 to 3e-15 of sum |terms| (300 to 4 million entries, lognormal factors), as pairs 1e-15 to 1.4e-14. alpha and
// beta are FP32 either way, and the rounded sums were the same.
struct Cg2State {
  float2 rho[2];     // (r, z) of the iteration with this parity
  float2 tol2;
  float beta;        // of the running iteration
  int it[2];         // updates completed before the iteration with this parity
};

// sum of the two slot contributions of each face entry (interior faces), 0 on boundary.
__device__ __forceinline__ double face_sum(const int32_t* __restrict__ face_slot, const double* __restrict__ zslot,
                                           int64_t f, int mm, int NF) {
  const int64_t s0 = face_slot[2 * f], s1 = face_slot[2 * f + 1];
  return zslot[s0 * NF + mm] + zslot[s1 * NF + mm];
}

// b = sum of slots (interior), 0 on boundary; optional scale.
static __global__ void face_gather_kernel(int64_t nf, int NF, const int32_t* __restrict__ face_slot,
                                   const int32_t* __restrict__ face_bnd, const double* __restrict__ zslot,
                                   double scale, double* __restrict__ out) {
  const int64_t n = nf * NF;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = t / NF;
    const int mm = (int)(t % NF);
    out[t] = face_bnd[f] < 0 ? scale * face_sum(face_slot, zslot, f, mm, NF) : 0.0;
  }
}

// r = b - (sgn K) x0, z = Dinv r, p = z; partials (rz, rr, bb) per block.
static __global__ void cg_init_kernel(int64_t nf, int NF, double sgn, const int32_t* __restrict__ face_slot,
                               const int32_t* __restrict__ face_bnd, const double* __restrict__ zslot,
                               const double* __restrict__ bvec, const double* __restrict__ dinv, double* __restrict__ r,
                               double* __restrict__ z, double* __restrict__ p, double* __restrict__ part) {
  __shared__ double red[8];
  const int64_t n = nf * NF;
  double rz = 0, rr = 0, bb = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = t / NF;
    const int mm = (int)(t % NF);
    double rv = 0, zv = 0;
    if (face_bnd[f] < 0) {
      const double q = sgn * face_sum(face_slot, zslot, f, mm, NF);
      const double bv = bvec[t];
      rv = bv - q;
      zv = dinv[t] * rv;
      bb += bv * bv;
    }
    r[t] = rv; z[t] = zv; p[t] = zv;
    rz += rv * zv; rr += rv * rv;
  }
  double s;
  s = block_sum256(rz, red); if (threadIdx.x == 0) part[blockIdx.x * 3 + 0] = s;
  s = block_sum256(rr, red); if (threadIdx.x == 0) part[blockIdx.x * 3 + 1] = s;
  s = block_sum256(bb, red); if (threadIdx.x == 0) part[blockIdx.x * 3 + 2] = s;
}

// State of the two-kernel FP64 iteration beside CgScal (the scheme of Cg2State)
struct Cg64State {
  double beta;   // of the running iteration
  int it[2];     // updates completed before the iteration with this parity
};

static __global__ void cg_init_scalars(int nb, const double* __restrict__ part, double rtol, CgScal* sc,
                                       Cg64State* st = nullptr) {
  __shared__ double red[8];
  const double rz = reduce_partials(part + 0, nb, 3, red);
  const double rr = reduce_partials(part + 1, nb, 3, red);
  const double bb = reduce_partials(part + 2, nb, 3, red);
  if (threadIdx.x == 0) {
    sc->rho[0] = rz; sc->rho[1] = 0; sc->bb = bb; sc->rr = rr;
    sc->tol2 = rtol * rtol * bb;
    sc->iters = 0;
    // a zero right-hand side ends the solve here (its solution is zero on interior faces)
    sc->done = sc->halt[0] = sc->halt[1] = (bb == 0.0 || rr <= sc->tol2) ? 1 : 0;
    if (st) st->it[0] = st->it[1] = 0;
  }
}

// q = (-K) p on faces (sgn = -1; +K for sgn = +1); partial p.q (NF compile-time)
template <class LD>
__global__ void __launch_bounds__(256) cg_face_q_kernel(int nf, double sgn, const int32_t* __restrict__ face_slot,
                                                        const int32_t* __restrict__ face_bnd,
                                                        const double* __restrict__ zslot, const double* __restrict__ p,
                                                        double* __restrict__ q, double* __restrict__ part,
                                                        const CgScal* __restrict__ sc) {
  constexpr int NF = LD::NF;
  if (sc->done) return;
  __shared__ double red[8];
  double pq = 0;
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    double qv[NF];
    if (face_bnd[f] < 0) {
      const double* s0 = zslot + (int64_t)face_slot[2 * f] * NF;
      const double* s1 = zslot + (int64_t)face_slot[2 * f + 1] * NF;
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) qv[mm] = sgn * (s0[mm] + s1[mm]);
    } else {
#pragma unroll
      for (int mm = 0; mm < NF; ++mm) qv[mm] = 0.0;
    }
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      q[(int64_t)f * NF + mm] = qv[mm];
      pq += p[(int64_t)f * NF + mm] * qv[mm];
    }
  }
  const double s = block_sum256(pq, red);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// alpha = rho/pq; x += alpha p; r -= alpha q; z = Dinv r; partials (rz, rr)
static __global__ void cg_update_kernel(int64_t n, int nb, int parity, const double* __restrict__ part_pq,
                                 const double* __restrict__ p, const double* __restrict__ q,
                                 const double* __restrict__ dinv, double* __restrict__ x, double* __restrict__ r,
                                 double* __restrict__ z, double* __restrict__ part, const CgScal* __restrict__ sc) {
  if (sc->done) return;
  __shared__ double red[8];
  const double pq = reduce_partials(part_pq, nb, 1, red);
  const double al = cta_ratio(sc->rho[parity], pq);
  double rz = 0, rr = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; t + 3 * stride < n; t += 4 * stride) {
    double pv[4], qv[4], xv[4], rv[4], dv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      pv[u] = p[t + u * stride]; qv[u] = q[t + u * stride]; xv[u] = x[t + u * stride];
      rv[u] = r[t + u * stride]; dv[u] = dinv[t + u * stride];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[t + u * stride] = xv[u] + al * pv[u];
      const double rn = rv[u] - al * qv[u];
      const double zn = dv[u] * rn;
      r[t + u * stride] = rn; z[t + u * stride] = zn;
      rz += rn * zn; rr += rn * rn;
    }
  }
  for (; t < n; t += stride) {
    const double pv = p[t];
    x[t] += al * pv;
    const double rv = r[t] - al * q[t];
    const double zv = dinv[t] * rv;
    r[t] = rv; z[t] = zv;
    rz += rv * zv; rr += rv * rv;
  }
  double s;
  s = block_sum256(rz, red); if (threadIdx.x == 0) part[blockIdx.x * 2 + 0] = s;
  s = block_sum256(rr, red); if (threadIdx.x == 0) part[blockIdx.x * 2 + 1] = s;
}

// beta = rz_new / rho; p = z + beta p; convergence test. iter >= 0: the iteration index from the
// host, h unused. iter < 0 (device-driven loop): block 0 counts the iterations in sc->iters and
// sets the loop condition h (continue while not done), also when the solve had already finished.
static __global__ void cg_direction_kernel(int64_t n, int nb, int parity, int iter, const double* __restrict__ part,
                                    const double* __restrict__ z, double* __restrict__ p, CgScal* sc, int maxit,
                                    cudaGraphConditionalHandle h) {
  if (sc->halt[parity]) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      sc->halt[parity ^ 1] = 1;
      if (iter < 0) cudaGraphSetConditional(h, 0u);
    }
    return;
  }
  __shared__ double red[8];
  const double rz = reduce_partials(part + 0, nb, 2, red);
  const double rr = reduce_partials(part + 1, nb, 2, red);
  const bool conv = rr <= sc->tol2;
  // with a host index no block reads what block 0 writes; on the device only block 0 uses it
  const int it = iter >= 0 ? iter + 1 : sc->iters + 1;
  if (!conv && (iter < 0 || it < maxit)) {
    const double be = cta_ratio(rz, sc->rho[parity]);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; t + 3 * stride < n; t += 4 * stride) {
      double pv[4], zv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) { pv[u] = p[t + u * stride]; zv[u] = z[t + u * stride]; }
#pragma unroll
      for (int u = 0; u < 4; ++u) p[t + u * stride] = zv[u] + be * pv[u];
    }
    for (; t < n; t += stride) p[t] = z[t] + be * p[t];
  }
  // every block has read sc->rho[parity] above; block 0 alone writes the other slot
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sc->rho[parity ^ 1] = rz;
    sc->rr = rr;
    sc->iters = it;
    const int done = conv ? 1 : (it >= maxit ? 2 : 0);
    if (done) sc->done = sc->halt[parity ^ 1] = done;
    if (iter < 0) cudaGraphSetConditional(h, done ? 0u : 1u);
  }
}

// ---- FP64 iteration in two kernels (one column, discontinuous traces): A = operator with the direction
// p_K = z_K + beta p_K formed in the gather, B = update of p, x, r, z; the scheme of Cg2State with FP64
// partials. For small systems, bounded by the latency of an iteration's dependent launches; each sum
// is formed by the warps side by side, and one thread of a CTA divides. 512 triangles, k = 2: 10 us an
// iteration (14.8 us in four kernels).
struct Cg64Args {
  CgScal* sc;
  Cg64State* st;
  double *partA, *partB;   // [na], [2][nb]
  int na, nb;
  int parity, maxit, dev;
  double sgn;
  cudaGraphConditionalHandle h;
};

// sums over the CTA (NW warps), to lane 0 of warp 0
template <int NQ, int NW>
__device__ __forceinline__ void block_sums(double (&a)[NQ]) {
  __shared__ double red[NQ][NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) a[q] = warp_sum(a[q]);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NQ; ++q) red[q][w] = a[q];
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      a[q] = lane < NW ? red[q][lane] : 0.0;
#pragma unroll
      for (int o = NW > 4 ? 4 : NW > 2 ? 2 : 1; o > 0; o >>= 1) a[q] += __shfl_down_sync(0xffffffffu, a[q], o);
    }
  }
}
// this thread's share of the sums of part[q n + i], i < n
template <int NQ, int NT>
__device__ __forceinline__ void partial_sums(const double* __restrict__ part, int n, double (&a)[NQ]) {
  constexpr int U = 4;
#pragma unroll
  for (int q = 0; q < NQ; ++q) a[q] = 0.0;
  for (int i = threadIdx.x; i < n; i += U * NT) {
    double v[NQ][U];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int u = 0; u < U; ++u) v[q][u] = i + u * NT < n ? part[q * n + i + u * NT] : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i + u * NT < n)
#pragma unroll
        for (int q = 0; q < NQ; ++q) a[q] += v[q][u];
  }
}

template <class D>
struct ApplyTwoCfg {
  static constexpr int EPB = ApplyCfg<D>::EPB;
  static constexpr int NW = (ApplyCfg<D>::NT + 31) / 32, NT = 32 * NW;
};

template <class D>
__global__ void __launch_bounds__(ApplyTwoCfg<D>::NT) apply_two64_kernel(DevMesh mesh, const double* __restrict__ S,
                                                                        const double* __restrict__ z,
                                                                        const double* __restrict__ p,
                                                                        double* __restrict__ zslot, Cg64Args o) {
  using C = ApplyTwoCfg<D>;
  constexpr int NF = D::NF, M = D::M, NFC = D::NFC;
  __shared__ double lx[C::EPB][M];
  __shared__ double bcast[2];
  const int el = threadIdx.x / M, r = threadIdx.x % M;
  const int64_t e = (int64_t)blockIdx.x * C::EPB + el;
  const bool live = el < C::EPB && e < mesh.ne;
  double zv = 0.0, pv = 0.0;
  if (live) {
    const int f = mesh.elem_face[e * NFC + r / NF];
    const int64_t t = (int64_t)f * NF + r % NF;
    if (mesh.face_bnd[f] < 0) {
      zv = z[t];
      pv = p[t];
    }
  }
  const int over = o.sc->halt[o.parity], k = o.st->it[o.parity];
  const double rho = o.sc->rho[o.parity], tol2 = o.sc->tol2;
  double a[2];
  partial_sums<2, C::NT>(o.partB, o.nb, a);   // at k = 0 for nothing
  if (over) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      o.sc->halt[o.parity ^ 1] = 1;
      if (o.dev) cudaGraphSetConditional(o.h, 0u);
    }
    return;
  }
  block_sums<2, C::NW>(a);
  if (threadIdx.x == 0) {
    double beta = 0.0, rz = rho;
    int done = 0;
    if (k > 0) {
      rz = a[0];
      beta = rz / rho;
      done = a[1] <= tol2 ? 1 : (k >= o.maxit ? 2 : 0);
    }
    bcast[0] = beta;
    bcast[1] = (double)done;
    if (blockIdx.x == 0) {
      if (k > 0) o.sc->rr = a[1];
      o.sc->rho[o.parity ^ 1] = rz;
      o.st->it[o.parity ^ 1] = k + 1;
      o.st->beta = beta;
      o.sc->iters = k;
      if (done) o.sc->done = o.sc->halt[o.parity ^ 1] = done;
      if (o.dev) cudaGraphSetConditional(o.h, done ? 0u : 1u);
    }
  }
  __syncthreads();
  if (bcast[1] != 0.0) return;
  const double beta = bcast[0];
  const double pn = k == 0 ? zv : fma(beta, pv, zv);
  if (live) lx[el][r] = pn;
  __syncthreads();
  double pq[1] = {0.0};
  if (live) {
    const double* Se = S + e * (int64_t)(M * M);
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < M; ++c) s += Se[c * M + r] * lx[el][c];
    zslot[e * M + r] = s;
    pq[0] = pn * s;
  }
  block_sums<1, C::NW>(pq);
  if (threadIdx.x == 0) o.partA[blockIdx.x] = pq[0];
}

template <class LD>
__global__ void __launch_bounds__(256) cg_update_two64_kernel(int64_t n, const int2* __restrict__ face_slot2,
                                                              const int32_t* __restrict__ face_bnd,
                                                              const double* __restrict__ zslot, double* __restrict__ p,
                                                              const double* __restrict__ dinv, double* __restrict__ x,
                                                              double* __restrict__ r, double* __restrict__ z, Cg64Args o) {
  constexpr int NF = LD::NF, U = 2;
  __shared__ double bcast;
  const int64_t S = (int64_t)gridDim.x * 256;
  int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x;
  double pv[U], zv[U], xv[U], rv[U], dv[U], q0[U], q1[U];
  auto load = [&] {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t tu = t + u * S;
      q0[u] = q1[u] = 0.0;
      if (tu < n) {
        const uint32_t f = (uint32_t)(tu / NF);
        const int mm = (int)(tu - (int64_t)f * NF);
        const int fb = face_bnd[f];
        const int2 fs = face_slot2[f];
        pv[u] = p[tu]; zv[u] = z[tu]; xv[u] = x[tu]; rv[u] = r[tu]; dv[u] = dinv[tu];
        if (fb < 0) {
          q0[u] = zslot[(int64_t)fs.x * NF + mm];
          q1[u] = zslot[(int64_t)fs.y * NF + mm];
        }
      }
    }
  };
  load();   // the first trip's, while alpha is formed
  const int over = o.sc->done, k = o.st->it[o.parity];
  const double rho = o.sc->rho[o.parity ^ 1], beta = o.st->beta;
  double pq[1];
  partial_sums<1, 256>(o.partA, o.na, pq);
  if (over) return;
  block_sums<1, 8>(pq);
  if (threadIdx.x == 0) bcast = rho / pq[0];   // sgn alpha: q = sgn (slot + slot) and sgn = +-1
  __syncthreads();
  const double sal = bcast, al = o.sgn * sal;
  double a[2] = {0.0, 0.0};   // (r, z), (r, r)
  while (t < n) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t tu = t + u * S;
      if (tu >= n) break;
      const double pn = k == 0 ? zv[u] : fma(beta, pv[u], zv[u]);
      p[tu] = pn;
      x[tu] = fma(al, pn, xv[u]);
      const double rn = fma(-sal, q0[u] + q1[u], rv[u]);
      const double zn = dv[u] * rn;
      r[tu] = rn;
      z[tu] = zn;
      a[0] += rn * zn;
      a[1] += rn * rn;
    }
    t += U * S;
    load();
  }
  block_sums<2, 8>(a);
  if (threadIdx.x == 0) {
    o.partB[blockIdx.x] = a[0];
    o.partB[gridDim.x + blockIdx.x] = a[1];
  }
}

// Least-squares initial guess over stored stage solutions. ring: [Q][n] contiguous.
// dots_ring_kernel: block partials of (v_i, w) for i < q and of (w, w), part[blk][q + 1].
static __global__ void dots_ring_kernel(int64_t n, int q, int64_t stride, const double* __restrict__ ring,
                                        const double* __restrict__ w, double* __restrict__ part) {
  __shared__ double red[8];
  double acc[9];
  for (int i = 0; i <= q; ++i) acc[i] = 0.0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const double wv = w[t];
    for (int i = 0; i < q; ++i) acc[i] += ring[i * stride + t] * wv;
    acc[q] += wv * wv;
  }
  for (int i = 0; i <= q; ++i) {
    const double s = block_sum256(acc[i], red);
    if (threadIdx.x == 0) part[blockIdx.x * (q + 1) + i] = s;
  }
}

static __global__ void dots_final_kernel(int nb, int q, const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double red[8];
  for (int i = 0; i <= q; ++i) {
    const double s = reduce_partials(part + i, nb, q + 1, red);
    if (threadIdx.x == 0) out[i] = s;
  }
}

struct Coef8 {
  double c[8];
};

// out[t] = sum_i c_i ring[i][t] on interior trace entries (mask != 0); boundary entries untouched
static __global__ void lincomb_ring_kernel(int64_t n, int q, int64_t stride, const double* __restrict__ ring, Coef8 c,
                                           const uint8_t* __restrict__ mask, double* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    if (!mask[t]) continue;
    double s = 0.0;
    for (int i = 0; i < q; ++i) s += c.c[i] * ring[i * stride + t];
    out[t] = s;
  }
}

// out = sum_q c_q in_q (up to four inputs), elementwise.
static __global__ void combine_kernel(int64_t n, double c0, const double* __restrict__ i0, double c1,
                               const double* __restrict__ i1, double c2, const double* __restrict__ i2, double c3,
                               const double* __restrict__ i3, double* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    double v = c0 * i0[t];
    if (i1) v += c1 * i1[t];
    if (i2) v += c2 * i2[t];
    if (i3) v += c3 * i3[t];
    out[t] = v;
  }
}

// boundary entries of lam <- coef[b] * fac (Dirichlet trace at the current time).
static __global__ void dirichlet_kernel(int64_t nb, int NF, const int64_t* __restrict__ bnd_faces,
                                 const double* __restrict__ coef, double fac, double* __restrict__ lam) {
  const int64_t n = nb * NF;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = t / NF;
    lam[bnd_faces[b] * NF + t % NF] = coef ? coef[t] * fac : 0.0;
  }
}

// interior entries of x <- 0
static __global__ void zero_interior_kernel(int64_t nf, int NF, const int32_t* __restrict__ face_bnd, double* __restrict__ x) {
  const int64_t n = nf * NF;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    if (face_bnd[t / NF] < 0) x[t] = 0.0;
}

// volume projection: u[e][c*NP+i] = sum_q w_q vals[e][q][c] phi_i(xi_q)  (mass = dJ I cancels dJ)
static __global__ void project_volume_kernel(int64_t ne, int NP, int nq, int ncomp, const double* __restrict__ w,
                                      const double* __restrict__ phi, const double* __restrict__ vals,
                                      double* __restrict__ u) {
  const int64_t n = ne * ncomp * NP;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = t / (ncomp * NP);
    const int c = (int)((t / NP) % ncomp), i = (int)(t % NP);
    double s = 0.0;
    for (int q = 0; q < nq; ++q) s += w[q] * vals[(e * nq + q) * ncomp + c] * phi[q * NP + i];
    u[t] = s;
  }
}

}  // namespace hdg

namespace hdg {

// ================================================================ mixed precision (FP32 inner solve)
// S32: the upper triangle (row-major, c >= r) of every S_K rounded to FP32, stored for groups
// of 32 elements as [group][P4][32][4] floats, P4 = ceil(M(M+1)/2 / 4): one warp handles a
// group, lane = element, each lane reads float4s and the warp's loads are contiguous.
template <int DIM, int K>
struct Packed {
  static constexpr int M = Dims<DIM, K>::M;
  static constexpr int P = M * (M + 1) / 2;
  static constexpr int P4 = (P + 3) / 4;
};

__host__ __device__ constexpr int packed_index(int M, int r, int c) { return r * M - r * (r - 1) / 2 + (c - r); }

// p.q of the Krylov iteration, formed inside the element apply: with q = sgn K p and K the
// sum of the element blocks, p.q = sgn sum_K p_K . (S_K p_K) (boundary entries of p are zero
// on both sides). Each 4-warp block writes its partial; the last block to finish (ticket
// counter, no waiting) sums the partials in index order and resets the counter.
// Launch timing on the device (also inside CUDA graphs): the first CTA to start lowers
// start_ns, the last CTA to finish (the one that sums the partials) adds the elapsed
// %globaltimer time to ms and counts the launch. Launches that return early (solve converged)
// are not counted.
struct DevTiming {
  unsigned long long start_ns;   // ULLONG_MAX between launches
  unsigned long long count;
  double ms;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct PqOut {
  double* part;       // [gridDim.x] block partials
  unsigned* ticket;   // zero between launches
  double* pq;         // result
  float sgn;
  DevTiming* timing;  // may be null
};

// t: global_ns() at the start of the CTA, in thread 0. A launch that may still turn out to have nothing to
// do stamps once it is known to be a live one.
__device__ __forceinline__ void timing_start(const PqOut& o, unsigned long long t) {
  if (o.timing && o.part && threadIdx.x == 0) atomicMin(&o.timing->start_ns, t);
}

// A kernel that leaves its partials to the next one still counts its CTAs for the launch timing.
__device__ __forceinline__ void timing_end(const PqOut& o) {
  if (!o.timing || threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(o.ticket, 1u) != gridDim.x - 1) return;
  const unsigned long long t1 = global_ns(), t0 = *(volatile unsigned long long*)&o.timing->start_ns;
  if (t1 > t0) {
    o.timing->ms += 1e-6 * (double)(t1 - t0);
    o.timing->count += 1;
  }
  o.timing->start_ns = ~0ull;
  *o.ticket = 0u;
}

__device__ __forceinline__ void pq_epilogue(const PqOut& o, double v) {
  __shared__ double wsum[4];
  __shared__ bool last;
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wsum[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    o.part[blockIdx.x] = ((wsum[0] + wsum[1]) + (wsum[2] + wsum[3]));
    __threadfence();
    last = atomicAdd(o.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) s += __ldcg(o.part + i);
  s = warp_sum(s);
  if (lane == 0) wsum[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    *o.pq = (double)o.sgn * ((wsum[0] + wsum[1]) + (wsum[2] + wsum[3]));
    *o.ticket = 0u;
    if (o.timing) {
      const unsigned long long t1 = global_ns();
      const unsigned long long t0 = *(volatile unsigned long long*)&o.timing->start_ns;
      if (t1 > t0) {
        o.timing->ms += 1e-6 * (double)(t1 - t0);
        o.timing->count += 1;
      }
      o.timing->start_ns = ~0ull;
    }
  }
}

// What kernels A and B of a two-kernel iteration share (see Cg2State)
struct Cg2Args {
  CgScal* sc;
  Cg2State* st;
  float2 *partA, *partB;   // partials of A [na], of B [2][nb]
  int na, nb;
  int parity, maxit, dev;
  float sgn;
  cudaGraphConditionalHandle h;
};

// Start of A: beta, or false when the solve is finished (recorded by CTA 0). first: p is still z.
template <int NW>
__device__ __forceinline__ bool cg2_begin_a(const Cg2Args& o, float& beta, bool& first) {
  // everything is loaded before any of it is tested: at k = 0 the partials are loaded for nothing
  const int over = o.sc->halt[o.parity], k = o.st->it[o.parity];
  const float2 rho = o.st->rho[o.parity], t2 = o.st->tol2;
  Acc2 a[2];
  sum_pairs<2, NW>(o.partB, o.nb, a);
  if (over) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      o.sc->halt[o.parity ^ 1] = 1;
      if (o.dev) cudaGraphSetConditional(o.h, 0u);
    }
    return false;
  }
  first = k == 0;
  beta = 0.f;
  float2 rz = rho;
  int done = 0;
  if (!first) {
    rz = make_float2(a[0].s, a[0].c);
    beta = pair_ratio(rz, rho);
    done = (a[1].s - t2.x) + (a[1].c - t2.y) <= 0.f ? 1 : (k >= o.maxit ? 2 : 0);
    if (blockIdx.x == 0 && threadIdx.x == 0) o.sc->rr = a[1].value();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    o.st->rho[o.parity ^ 1] = rz;
    o.st->it[o.parity ^ 1] = k + 1;
    o.st->beta = beta;
    o.sc->iters = k;
    if (done) o.sc->done = o.sc->halt[o.parity ^ 1] = done;
    if (o.dev) cudaGraphSetConditional(o.h, done ? 0u : 1u);
  }
  return done == 0;
}

// End of A: this CTA's partial of (p, S p)
template <int NW>
__device__ __forceinline__ void cg2_end_a(const Cg2Args& o, Acc2 pq) {
  Acc2 a[1] = {pq};
  block_pairs<1, NW>(a);
  if (threadIdx.x == 0) o.partA[blockIdx.x] = make_float2(a[0].s, a[0].c);
}

// direction entry of a two-kernel iteration: one multiply-add wherever it is formed, so both
// elements of a face and the owner of the entry hold the same bits
__device__ __forceinline__ float cg2_dir(bool first, float beta, float p, float z) { return first ? z : fmaf(beta, p, z); }

// slot32 layout: [e][M] floats (element-major, like the FP64 slots); the warp transposes
// its 32 x M products through shared memory so that the stores are contiguous float4s.
// TWO: kernel A of a two-kernel iteration (x = z, the direction from z and p, partials left in o2);
// else x is the direction and the epilogue completes (p, q).
template <int DIM, int K, bool TWO>
__global__ void __launch_bounds__(128, 4) apply32_kernel(int64_t ne, const int32_t* __restrict__ elem_face,
                                                      const int32_t* __restrict__ face_bnd,
                                                      const float* __restrict__ S32, const float* __restrict__ x,
                                                      const float* __restrict__ p, float* __restrict__ slot,
                                                      const int* __restrict__ done, PqOut pqo, Cg2Args o2) {
  using D = Dims<DIM, K>;
  using PK = Packed<DIM, K>;
  constexpr int NF = D::NF, M = D::M, NFC = D::NFC, P4 = PK::P4;
  constexpr int MP = M + 1;   // padded row: conflict-free transposed writes
  __shared__ float tr[4][32 * MP];
  if constexpr (!TWO) {
    if (done && *done) return;
    timing_start(pqo, global_ns());
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t g0 = (int64_t)blockIdx.x * 4 + wid;
  const bool wact = g0 * 32 < ne;                 // the last block may hold idle warps
  const int64_t g = wact ? g0 : 0;
  const int64_t e = g0 * 32 + lane;
  float xl[M], y[M];   // TWO: y holds p until the direction is formed
#pragma unroll
  for (int f = 0; f < NFC; ++f) {
    int fid = -1;
    if (e < ne) fid = elem_face[e * NFC + f];
    const bool use = fid >= 0 && face_bnd[fid] < 0;
#pragma unroll
    for (int mm = 0; mm < NF; ++mm) {
      const int64_t t = (int64_t)fid * NF + mm;
      xl[f * NF + mm] = use ? x[t] : 0.f;
      if constexpr (TWO) y[f * NF + mm] = use ? p[t] : 0.f;
    }
  }
  if constexpr (TWO) {
    float beta;
    bool first;
    const unsigned long long t0 = threadIdx.x == 0 ? global_ns() : 0ull;
    if (!cg2_begin_a<4>(o2, beta, first)) return;   // while the gather is in flight
    timing_start(pqo, t0);
#pragma unroll
    for (int r = 0; r < M; ++r) xl[r] = cg2_dir(first, beta, y[r], xl[r]);
  }
#pragma unroll
  for (int r = 0; r < M; ++r) y[r] = 0.f;
  const float4* Sg = reinterpret_cast<const float4*>(S32) + g * (int64_t)P4 * 32 + lane;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int r = 0; r < M; ++r) {
#pragma unroll
    for (int c = r; c < M; ++c) {
      const int p = packed_index(M, r, c);
      if ((p & 3) == 0) v = __ldcs(Sg + (p >> 2) * 32);
      const float s = (p & 3) == 0 ? v.x : (p & 3) == 1 ? v.y : (p & 3) == 2 ? v.z : v.w;
      y[r] = fmaf(s, xl[c], y[r]);
      if (c != r) y[c] = fmaf(s, xl[r], y[c]);
    }
  }
  float* t = tr[wid];
#pragma unroll
  for (int r = 0; r < M; ++r) t[lane * MP + r] = y[r];
  __syncwarp();
  if (wact) {
    const int64_t nvalid = (ne - g * 32) < 32 ? (ne - g * 32) : 32;
    float* dst = slot + g * 32 * (int64_t)M;
    for (int idx = lane; idx < nvalid * M; idx += 32) dst[idx] = t[(idx / M) * MP + idx % M];
  }
  Acc2 a;
#pragma unroll
  for (int r = 0; r < M; ++r) a.dot(xl[r], y[r]);
  if constexpr (TWO) {
    cg2_end_a<4>(o2, a);
    timing_end(pqo);
  } else if (pqo.part) {
    pq_epilogue(pqo, a.value());
  }
}

// f(0), .., f(N - 1) with compile-time arguments: loops too long for the unroller keep register arrays
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// ---------------------------------------------------------------- FP16 operator copy
// Packed symmetric S_K in binary16 with one FP32 scale per element: S_K ~ sc16[e] * S16,
// sc16[e] = max |S_K| (so every stored value lies in [-1, 1]). Layout [group][P8][lane][8]:
// one 16-byte load per lane carries 8 consecutive packed entries.
template <int DIM, int K>
struct Packed16 {
  static constexpr int M = Dims<DIM, K>::M;
  static constexpr int P = M * (M + 1) / 2;
  static constexpr int P8 = (P + 7) / 8;
};

// Trace gather table of the FP16 apply: gface[e][f] = the id of face f of element e where it
// carries trace unknowns (an interior face), else -1; rows past the last element are -1
// (n = whole 32-element groups x NFC).
static __global__ void gface_kernel(int64_t n, int64_t nval, const int32_t* __restrict__ elem_face,
                                    const int32_t* __restrict__ face_bnd, int32_t* __restrict__ gface) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    int v = -1;
    if (t < nval) {
      const int f = elem_face[t];
      if (f >= 0 && face_bnd[f] < 0) v = f;
    }
    gface[t] = v;
  }
}

// Shared memory of the FP16 apply, per warp: the staged traces of the next group (row stride
// XS floats; each face run is copied by 8-byte asynchronous copies when NF is even, else
// 4-byte ones) and the transpose buffer of the slot write (row stride MP).
template <int DIM, int K>
struct Apply16Cfg {
  static constexpr int NF = Dims<DIM, K>::NF, M = Dims<DIM, K>::M;
  static constexpr int CPB = NF % 2 == 0 ? 8 : 4;
  static constexpr int XS = CPB == 8 ? M + 2 : M + 1;
  static constexpr int MP = M + 1;
  static constexpr int WARPS = 4;
  static constexpr size_t SMEM = sizeof(float) * WARPS * 32 * (XS + MP);
};

// slot = S_K x_K with the FP16 copy (FP32 accumulation, the element scale applied once at the
// end), one thread per element, one warp per group of 32 elements. Persistent: warps stride
// over the groups, and the traces of a warp's next group are gathered into shared memory by
// asynchronous copies (from gface, read one more group ahead) while the current group's S16
// streams in, so the gather latency is off the streaming path.
template <int DIM, int K>
__global__ void __launch_bounds__(128, 4) apply16_kernel(int64_t ne, const int32_t* __restrict__ gface,
                                                      const __half* __restrict__ S16, const float* __restrict__ sc16,
                                                      const float* __restrict__ x, float* __restrict__ slot,
                                                      const int* __restrict__ done, PqOut pqo) {
  using D = Dims<DIM, K>;
  using PK = Packed16<DIM, K>;
  using C = Apply16Cfg<DIM, K>;
  constexpr int NF = D::NF, M = D::M, NFC = D::NFC, P8 = PK::P8, XS = C::XS, MP = C::MP, CPB = C::CPB;
  extern __shared__ __align__(16) float a16sm[];
  if (done && *done) return;
  timing_start(pqo, global_ns());
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float* t = a16sm + wid * 32 * (XS + MP) + 32 * XS;
  const unsigned xrow = (unsigned)__cvta_generic_to_shared(a16sm + wid * 32 * (XS + MP) + lane * XS);
  const float* xrow_g = a16sm + wid * 32 * (XS + MP) + lane * XS;
  const int64_t ngroups = (ne + 31) / 32;
  const int64_t nw = (int64_t)gridDim.x * C::WARPS;
  int gf[NFC];
  auto load_gf = [&](int64_t gg) {
#pragma unroll
    for (int f = 0; f < NFC; ++f) gf[f] = gg < ngroups ? gface[(gg * 32 + lane) * NFC + f] : -1;
  };
  // this lane's traces into its own row (zeros where gf < 0); only this lane reads the row
  auto issue = [&]() {
#pragma unroll
    for (int f = 0; f < NFC; ++f) {
      const float* src = gf[f] >= 0 ? x + (int64_t)gf[f] * NF : x;
      const unsigned nb = gf[f] >= 0 ? CPB : 0;
#pragma unroll
      for (int j = 0; j < NF * 4 / CPB; ++j)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(xrow + 4 * f * NF + CPB * j),
                     "l"(src + (CPB / 4) * j), "n"(CPB), "r"(nb)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  int64_t g = (int64_t)blockIdx.x * C::WARPS + wid;
  load_gf(g);
  issue();
  load_gf(g + nw);
  Acc2 a;
  for (; g < ngroups; g += nw) {
    const int64_t e = g * 32 + lane;
    const float scl = e < ne ? sc16[e] : 0.f;
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    float xl[M], y[M];
#pragma unroll
    for (int r = 0; r < M; ++r) xl[r] = xrow_g[r];
    issue();              // the next group's traces
    load_gf(g + 2 * nw);  // and the group after it's gather table
#pragma unroll
    for (int r = 0; r < M; ++r) y[r] = 0.f;
    const uint4* Sg = reinterpret_cast<const uint4*>(S16) + g * (int64_t)P8 * 32 + lane;
    float sv[8];
#pragma unroll
    for (int r = 0; r < M; ++r) {
#pragma unroll
      for (int c = r; c < M; ++c) {
        const int p = packed_index(M, r, c);
        if ((p & 7) == 0) {
          const uint4 u = __ldcs(Sg + (p >> 3) * 32);
          const unsigned w4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float2 f2 = __half22float2(*reinterpret_cast<const __half2*>(&w4[h]));
            sv[2 * h] = f2.x;
            sv[2 * h + 1] = f2.y;
          }
        }
        const float s = sv[p & 7];
        y[r] = fmaf(s, xl[c], y[r]);
        if (c != r) y[c] = fmaf(s, xl[r], y[c]);
      }
    }
#pragma unroll
    for (int r = 0; r < M; ++r) {
      y[r] *= scl;
      t[lane * MP + r] = y[r];
      a.dot(xl[r], y[r]);
    }
    __syncwarp();
    const int64_t nvalid = (ne - g * 32) < 32 ? (ne - g * 32) : 32;
    float* dst = slot + g * 32 * (int64_t)M;
    for (int idx = lane; idx < nvalid * M; idx += 32) dst[idx] = t[(idx / M) * MP + idx % M];
    __syncwarp();   // the transpose buffer is rewritten by the next group
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if (pqo.part) pq_epilogue(pqo, a.value());
}

// FP32 vectors are padded to a multiple of 4 entries (padding: zero, dinv = 0) and
// processed as float4.
__device__ __forceinline__ float4 f4fma(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ float4 f4mul(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }


// inner solve start from x = 0: r = b, z = Dinv r, p = z; partials (rz, rr)
static __global__ void cg32_init_kernel(int64_t n4, const float4* __restrict__ b, const float4* __restrict__ dinv,
                                 float4* __restrict__ x, float4* __restrict__ r, float4* __restrict__ z,
                                 float4* __restrict__ p, float2* __restrict__ part) {
  Acc2 a[2];   // (r, z), (r, r)
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
    const float4 rv = b[t];
    const float4 zv = f4mul(dinv[t], rv);
    x[t] = make_float4(0.f, 0.f, 0.f, 0.f); r[t] = rv; z[t] = zv; p[t] = zv;
    a[0].dot4(rv, zv); a[1].dot4(rv, rv);
  }
  block_pairs<2, 8>(a);
  if (threadIdx.x < 2) part[threadIdx.x * gridDim.x + blockIdx.x] = make_float2(a[threadIdx.x].s, a[threadIdx.x].c);
}

// rtol_dev (may be null): the relative tolerance read on the device instead of rtol
static __global__ void cg32_init_scalars(int nb, const float2* __restrict__ part, double rtol, CgScal* sc, Cg2State* st,
                                         const double* __restrict__ rtol_dev) {
  Acc2 a[2];
  sum_pairs<2, 8>(part, nb, a);
  if (threadIdx.x == 0) {
    const double tol = rtol_dev ? *rtol_dev : rtol, rr = a[1].value(), t2 = tol * tol * rr;
    sc->rho[0] = a[0].value(); sc->rho[1] = 0; sc->bb = rr; sc->rr = rr;
    sc->tol2 = t2;
    sc->iters = 0;
    sc->done = sc->halt[0] = sc->halt[1] = (rr == 0.0) ? 1 : 0;
    st->rho[0] = st->rho[1] = make_float2(a[0].s, a[0].c);
    st->tol2 = make_float2((float)t2, (float)(t2 - (double)(float)t2));
    st->beta = 0.f;
    st->it[0] = st->it[1] = 0;
  }
}

// The update of the Krylov iteration with q = sgn K p formed from the slots (the face pass
// is folded in): q = sgn (slot0 + slot1) on interior faces (0 on the boundary),
// x += alpha p, r -= alpha q, z = Dinv r; partials (r.z, r.r). alpha = rho / pq with pq
// from the apply's reduction. Vectors are processed as float4 (coalesced); the two slot
// values of each entry are gathered by runs within a face. Two float4
// per trip, and the face flags and slot pairs loaded before the branch on them, keep two
// independent load chains in flight per thread; a thread visits its entries in the same order
// as with one float4 per trip, so the sums are the same.
template <class LD>
__device__ __forceinline__ float4 q_entries4(int64_t t, int64_t nfe, float sgn, const int2* __restrict__ face_slot2,
                                             const int32_t* __restrict__ face_bnd, const float* __restrict__ slot) {
  // V consecutive entries never leave a face: one face lookup and two V-wide loads serve them
  constexpr int NF = LD::NF, V = NF % 4 == 0 ? 4 : NF % 2 == 0 ? 2 : 1, G = 4 / V;
  const int64_t d0 = 4 * t;
  uint32_t f = (uint32_t)(d0 / NF);   // n_faces * NF < 2^32
  int mm = (int)(d0 - (int64_t)f * NF);
  uint32_t fi[G];
  int mi[G], fb[G];
  int2 fs[G];
  bool ok[G];
#pragma unroll
  for (int i = 0; i < G; ++i) {
    fi[i] = f;
    mi[i] = mm;
    mm += V;
    if (mm == NF) { mm = 0; ++f; }
  }
#pragma unroll
  for (int i = 0; i < G; ++i) {
    ok[i] = d0 + V * i < nfe;
    fb[i] = ok[i] ? face_bnd[fi[i]] : 0;
    fs[i] = ok[i] ? face_slot2[fi[i]] : make_int2(0, 0);
  }
  float q[4];
#pragma unroll
  for (int i = 0; i < G; ++i) {
    float a[V], b[V];
#pragma unroll
    for (int v = 0; v < V; ++v) a[v] = b[v] = 0.f;
    if (ok[i] && fb[i] < 0) {
      const float *sa = slot + (int64_t)fs[i].x * NF + mi[i], *sb = slot + (int64_t)fs[i].y * NF + mi[i];
      if constexpr (V == 4) {
        const float4 u = *reinterpret_cast<const float4*>(sa), w = *reinterpret_cast<const float4*>(sb);
        a[0] = u.x; a[1] = u.y; a[2] = u.z; a[3] = u.w;
        b[0] = w.x; b[1] = w.y; b[2] = w.z; b[3] = w.w;
      } else if constexpr (V == 2) {
        const float2 u = *reinterpret_cast<const float2*>(sa), w = *reinterpret_cast<const float2*>(sb);
        a[0] = u.x; a[1] = u.y;
        b[0] = w.x; b[1] = w.y;
      } else {
        a[0] = *sa;
        b[0] = *sb;
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) q[V * i + v] = sgn * (a[v] + b[v]);
  }
  return make_float4(q[0], q[1], q[2], q[3]);
}

// where q's four entries of a float4 come from: the two slots of an interior face, or slot positions
// per entry (dslot[2 t], dslot[2 t + 1]; -1: boundary)
template <class LD>
struct QFaces {
  int64_t nfe;
  const int2* face_slot2;
  const int32_t* face_bnd;
  __device__ __forceinline__ float4 at(int64_t t, float sgn, const float* slot) const {
    return q_entries4<LD>(t, nfe, sgn, face_slot2, face_bnd, slot);
  }
};
struct QSlots {
  int64_t n;
  const int32_t* dslot;
  __device__ __forceinline__ float4 at(int64_t t, float sgn, const float* slot) const {
    float q[4];
    int2 d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = 4 * t + i < n ? reinterpret_cast<const int2*>(dslot)[4 * t + i] : make_int2(-1, -1);
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = d[i].x >= 0 ? sgn * (slot[d[i].x] + slot[d[i].y]) : 0.f;
    return make_float4(q[0], q[1], q[2], q[3]);
  }
};

// TWO: kernel B of a two-kernel iteration (alpha from A's partials, p advanced here); else p is the
// direction and (p, q) complete in pq_in.
// (The first trip's loads are issued before alpha is formed.)
template <class Q, bool TWO>
__global__ void __launch_bounds__(256, 3) cg32_update_f_kernel(int64_t n4, float sgn, int parity, Q qsrc,
                                                               const float* __restrict__ slot, float4* __restrict__ p,
                                                               const float4* __restrict__ dinv, float4* __restrict__ x,
                                                               float4* __restrict__ r, float4* __restrict__ z,
                                                               const double* __restrict__ pq_in,
                                                               float2* __restrict__ part, const CgScal* __restrict__ sc,
                                                               Cg2Args o2) {
  constexpr int U = TWO ? 1 : 2;
  if constexpr (!TWO) {
    if (sc->done) return;
  }
  float4 pv[U], xv[U], rv[U], dv[U], qv[U], zv[U];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  auto load = [&] {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t tu = t + u * stride;
      if (tu < n4) {
        pv[u] = p[tu];
        if constexpr (TWO) zv[u] = z[tu];
        xv[u] = x[tu]; rv[u] = r[tu]; dv[u] = dinv[tu];
        qv[u] = qsrc.at(tu, sgn, slot);
      }
    }
  };
  float al, beta = 0.f;
  bool first = true;
  if constexpr (TWO) {
    load();
    const int over = sc->done, k = o2.st->it[parity];
    const float2 rho = o2.st->rho[parity ^ 1];
    beta = o2.st->beta;
    Acc2 pq[1];
    sum_pairs<1, 8>(o2.partA, o2.na, pq);
    if (over) return;
    al = pair_ratio(rho, make_float2(sgn * pq[0].s, sgn * pq[0].c));
    first = k == 0;
  } else {
    load();
    al = (float)cta_ratio(sc->rho[parity], *pq_in);
  }
  Acc2 a[2];   // (r, z), (r, r)
  while (t < n4) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t tu = t + u * stride;
      if (tu >= n4) break;
      if constexpr (TWO) {
        pv[u] = first ? zv[u] : f4fma(beta, pv[u], zv[u]);
        p[tu] = pv[u];
      }
      x[tu] = f4fma(al, pv[u], xv[u]);
      const float4 rn = f4fma(-al, qv[u], rv[u]);
      const float4 zn = f4mul(dv[u], rn);
      r[tu] = rn;
      z[tu] = zn;
      a[0].dot4(rn, zn);
      a[1].dot4(rn, rn);
    }
    t += U * stride;
    load();
  }
  block_pairs<2, 8>(a);
  if (threadIdx.x < 2) {
    float2* o = TWO ? o2.partB : part;
    o[threadIdx.x * gridDim.x + blockIdx.x] = make_float2(a[threadIdx.x].s, a[threadIdx.x].c);
  }
}

// as cg_direction_kernel, FP32 vectors (float4). PART: double (interleaved sums), or float2 (compensated
// pairs [2][nb], as in the two-kernel iteration): the FP64 sums of every CTA and a division in every
// thread were most of this kernel's time, 196,608 tets, k = 3: 11.7 us, now 7.8 us
template <class PART>
__global__ void __launch_bounds__(256) cg32_direction_kernel(int64_t n4, int nb, int parity, int iter,
                                                             const PART* __restrict__ part, const float4* __restrict__ z,
                                                             float4* __restrict__ p, CgScal* sc, int maxit,
                                                             cudaGraphConditionalHandle h) {
  if (sc->halt[parity]) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      sc->halt[parity ^ 1] = 1;
      if (iter < 0) cudaGraphSetConditional(h, 0u);
    }
    return;
  }
  __shared__ double rzs, rrs;
  __shared__ float bes;
  if constexpr (std::is_same<PART, float2>::value) {
    Acc2 a[2];
    sum_pairs<2, 8>(part, nb, a);
    if (threadIdx.x == 0) {
      rzs = a[0].value();
      rrs = a[1].value();
    }
  } else {
    __shared__ double red[8];
    const double rz0 = reduce_partials(part + 0, nb, 2, red);
    const double rr0 = reduce_partials(part + 1, nb, 2, red);
    if (threadIdx.x == 0) {
      rzs = rz0;
      rrs = rr0;
    }
  }
  if (threadIdx.x == 0) bes = (float)(rzs / sc->rho[parity]);
  __syncthreads();
  const double rz = rzs, rr = rrs;
  const bool conv = rr <= sc->tol2;
  const int it = iter >= 0 ? iter + 1 : sc->iters + 1;
  if (!conv && (iter < 0 || it < maxit)) {
    const float be = bes;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (; t + 3 * stride < n4; t += 4 * stride) {
      float4 pv[4], zv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) { pv[u] = p[t + u * stride]; zv[u] = z[t + u * stride]; }
#pragma unroll
      for (int u = 0; u < 4; ++u) p[t + u * stride] = f4fma(be, pv[u], zv[u]);
    }
    for (; t < n4; t += stride) p[t] = f4fma(be, p[t], z[t]);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sc->rho[parity ^ 1] = rz;
    sc->rr = rr;
    sc->iters = it;
    const int done = conv ? 1 : (it >= maxit ? 2 : 0);
    if (done) sc->done = sc->halt[parity ^ 1] = done;
    if (iter < 0) cudaGraphSetConditional(h, done ? 0u : 1u);
  }
}

// FP64 refinement residual rho = b - (sgn K) lam = b - sgn sum slots64 (interior), partials |rho|^2, |b|^2
static __global__ void refine_residual_kernel(int64_t nf, int NF, double sgn, const int32_t* __restrict__ face_slot,
                                       const int32_t* __restrict__ face_bnd, const double* __restrict__ zslot,
                                       const double* __restrict__ b, double* __restrict__ rho,
                                       double* __restrict__ part, const int* __restrict__ skip) {
  if (skip && *skip) return;   // rho and the partials are already in place
  __shared__ double red[8];
  const int64_t n = nf * NF;
  double rr = 0, bb = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t f = (uint32_t)t / (uint32_t)NF;   // n < 2^32
    const int mm = (int)((uint32_t)t - f * (uint32_t)NF);
    double v = 0.0;
    if (face_bnd[f] < 0) {
      const double bv = b[t];
      v = bv - sgn * face_sum(face_slot, zslot, f, mm, NF);
      bb += bv * bv;
    }
    rho[t] = v;
    rr += v * v;
  }
  double s;
  s = block_sum256(rr, red); if (threadIdx.x == 0) part[blockIdx.x * 2 + 0] = s;
  s = block_sum256(bb, red); if (threadIdx.x == 0) part[blockIdx.x * 2 + 1] = s;
}

struct RefScal {
  double rr, bb, scale;
};

static __global__ void refine_scalars(int nb, const double* __restrict__ part, RefScal* rs) {
  __shared__ double red[8];
  const double rr = reduce_partials(part + 0, nb, 2, red);
  const double bb = reduce_partials(part + 1, nb, 2, red);
  if (threadIdx.x == 0) {
    rs->rr = rr; rs->bb = bb;
    rs->scale = rr > 0.0 ? 1.0 / sqrt(rr) : 1.0;
  }
}

// b32 = rho * scale (inner right-hand side of unit norm)
static __global__ void to32_scaled_kernel(int64_t n, const double* __restrict__ rho, const RefScal* __restrict__ rs,
                                   float* __restrict__ b32) {
  const double s = rs->scale;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    b32[t] = (float)(rho[t] * s);
}

// lam += delta / scale on interior faces (delta is zero on boundary faces)
static __global__ void refine_update_kernel(int64_t nf, int NF, const int32_t* __restrict__ face_bnd,
                                     const float* __restrict__ delta, const RefScal* __restrict__ rs,
                                     double* __restrict__ lam) {
  const double inv = cta_ratio(1.0, rs->scale);
  const int64_t n = nf * NF;   // < 2^32
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    if (face_bnd[(uint32_t)t / (uint32_t)NF] < 0) lam[t] += (double)delta[t] * inv;
}

static __global__ void to32_kernel(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    b[t] = (float)a[t];
}

}  // namespace hdg

namespace hdg {

// ================================================================ double-float (FP64-class on the FP32 pipe)
// A value is the unevaluated sum h + l of two floats (|l| <= ulp(h)/2): about 48 significant
// bits. Products use the exact FMA error of h*h, sums the TwoSum error, so dot products keep
// the accuracy of FP64 evaluation to ~1e-14 relative on GB300's 58x faster FP32 pipe.
struct df2 {
  float h, l;
};

__device__ __forceinline__ df2 df_from(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

// hi = fl32(v), lo = fl32(v - hi), bit for bit as the FP64 conversions give them, on the integer
// pipe: the four FP64 instructions of the other route cost a copy kernel more than its bytes do
// (to_df_kernel on 33 M entries: 0.234 -> 0.090 ms).
__device__ __forceinline__ void split_f64(double v, float& hi, float& lo) {
  const unsigned hw = (unsigned)__double2hiint(v), lw = (unsigned)__double2loint(v);
  const int ex = (int)((hw >> 20) & 0x7ffu);
  if (ex < 960 || ex > 1140) {   // zero, tiny, huge, infinite: by conversion
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
    return;
  }
  const unsigned m = ((hw & 0xfffffu) << 3) | (lw >> 29), rem = lw & 0x1fffffffu;
  const unsigned up = rem > 0x10000000u || (rem == 0x10000000u && (m & 1u)) ? 1u : 0u;   // nearest, ties to even
  const unsigned sign = hw & 0x80000000u;
  hi = __uint_as_float(sign | ((((unsigned)(ex - 896) << 23) | m) + up));
  // the signed remainder in units of the last FP64 place, rounded once
  const float rl = (float)((int)rem - (int)(up << 29)) * __uint_as_float((unsigned)(ex - 948) << 23);
  lo = sign ? 0.f - rl : rl;   // an exact value leaves +0, as v - hi does
}

// (double)h + (double)l for a normalised pair, the same bits, on the integer pipe: l in units of the
// last place of the FP64 result is rounded to an integer and added to the widened significand of h.
__device__ __forceinline__ double join_f64(float h, float l) {
  const unsigned hb = __float_as_uint(h);
  const int eh = (int)((hb >> 23) & 0xffu);
  if (eh >= 80 && eh < 255) {
    const float ls = l * __uint_as_float((unsigned)(306 - eh) << 23);   // exact: a power of two
    const long long m = ((long long)((hb & 0x7fffffu) | 0x800000u) << 29) + __float2int_rn((int)hb < 0 ? -ls : ls);
    if (m > (1ll << 52) && fabsf(ls) < 1073741824.f)
      return __hiloint2double((int)((hb & 0x80000000u) | ((unsigned)(m >> 32) - 0x100000u + ((unsigned)(eh + 896) << 20))),
                              (int)(unsigned)m);
  }
  // zero, tiny, not finite, a sum below the binade of h, or one that rounded up to its edge: the places there
  // are half as far apart
  return (double)h + (double)l;
}

// compensated accumulator of sum_i a_i b_i with a_i, b_i double-floats
struct DfAcc {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void fma(df2 a, df2 b) {
    const float p = a.h * b.h;
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
    const float t = s + p;
    const float bb = t - s;
    c += ((s - (t - bb)) + (p - bb)) + e;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

__device__ __forceinline__ df2 df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ df2 df_mul(df2 a, df2 b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
  const float s = p + e;
  return {s, e - (s - p)};
}
__device__ __forceinline__ df2 df_add(df2 a, df2 b) {
  df2 s = df_two_sum(a.h, b.h);
  const float err = s.l + (a.l + b.l);
  const float h = s.h + err;
  return {h, err - (h - s.h)};
}
// normalised value of a compensated accumulator
__device__ __forceinline__ df2 df_of(const DfAcc& a) { return df_two_sum(a.s, a.c); }

// conversions of the local solves, on the integer pipe (see split_f64)
__device__ __forceinline__ df2 dfl_from(double x) {
  df2 v;
  split_f64(x, v.h, v.l);
  return v;
}
__device__ __forceinline__ double dfl_to(df2 v) { return join_f64(v.h, v.l); }

// Double-float copy of S_K for the refinement apply, element-contiguous and diagonal-major:
// element e holds [hi | lo], each PD = 4 * P4 floats, entry (r, r + s) of the upper triangle at
// off(s) + r with off(s) = packed_index(M, s, s) (the s-th superdiagonal follows the first s
// ones). hi = fl32(S), lo = fl32(S - hi).
__host__ __device__ constexpr int diag_off(int M, int s) { return packed_index(M, s, s); }

// FP64-accurate refinement apply on the FP32 pipe: zslot[e][r] = sum_c S_K[r][c] x_K[c] with
// S_K = hi + lo from the diagonal-major copy and x split into double-floats. CTA = EPB
// elements, one thread per (element, row); persistent over groups of EPB elements, the
// copies of the next group staged in shared memory with 16-byte asynchronous copies while the
// current one is computed (two stages). At step s thread r takes column c = (r + s) mod M: the
// superdiagonal s at row r when c >= r, else the superdiagonal M - s at row c, so the threads
// of an element read two runs of consecutive words.
template <int DIM, int K>
struct ApplyDfCfg {
  static constexpr int M = Dims<DIM, K>::M;
  static constexpr int EPB = 4;
  static constexpr int NT = EPB * M;
  static constexpr int PD = Packed<DIM, K>::P4 * 4;
  static constexpr int CH = EPB * 2 * PD / 4;                   // 16-byte chunks per group
  static constexpr int STAGE = EPB * 2 * PD;                     // floats per stage
  static constexpr size_t SMEM = sizeof(float) * 2 * STAGE + sizeof(df2) * EPB * M;
};

template <int DIM, int K>
__global__ void __launch_bounds__(ApplyDfCfg<DIM, K>::NT) apply_df_kernel(DevMesh mesh, const float* __restrict__ Sdf,
                                                                         const double* __restrict__ x,
                                                                         double* __restrict__ zslot, int64_t ngroups,
                                                                         const int* __restrict__ skip) {
  using D = Dims<DIM, K>;
  using C = ApplyDfCfg<DIM, K>;
  if (skip && *skip) return;   // the residual this apply serves is already in place
  constexpr int NF = D::NF, M = D::M, NFC = D::NFC, EPB = C::EPB, PD = C::PD;
  extern __shared__ __align__(16) float dsm[];
  df2* lx = reinterpret_cast<df2*>(dsm + 2 * C::STAGE);   // [EPB][M]
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(dsm);
  // the copy is padded to whole 32-element groups, so every chunk of a group is in bounds
  auto issue = [&](int64_t g, int stage) {
    const char* src = reinterpret_cast<const char*>(Sdf + g * EPB * 2 * PD);
    const unsigned dst = sbase + (unsigned)(stage * C::STAGE * sizeof(float));
    for (int i = threadIdx.x; i < C::CH; i += C::NT)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16 * i), "l"(src + 16 * i) : "memory");
  };
  int64_t g = blockIdx.x;
  if (g >= ngroups) return;
  issue(g, 0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  const int el = threadIdx.x / M, r = threadIdx.x % M;
  // this thread's trace entry of group gg (gathered one group ahead, off the compute path)
  auto gather = [&](int64_t gg) {
    double v = 0.0;
    const int64_t ee = gg * EPB + el;
    if (gg < ngroups && ee < mesh.ne) {
      const int f = mesh.elem_face[ee * NFC + r / NF];
      if (mesh.face_bnd[f] < 0) v = x[(int64_t)f * NF + r % NF];
    }
    return v;
  };
  double vnext = gather(g);
  for (int it = 0; g < ngroups; ++it, g += gridDim.x) {
    const int cur = it & 1;
    if (g + gridDim.x < ngroups) issue(g + gridDim.x, cur ^ 1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const int64_t e = g * EPB + el;
    lx[el * M + r] = df_from(vnext);
    vnext = gather(g + gridDim.x);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    if (e < mesh.ne) {
      const float* hi = dsm + cur * C::STAGE + el * 2 * PD;
      const float* lo = hi + PD;
      const df2* ex = lx + el * M;
      DfAcc acc;
#pragma unroll
      for (int s = 0; s < M; ++s) {
        const int c = r + s;
        const bool up = c < M;
        const int pos = up ? diag_off(M, s) + r : diag_off(M, M - s) + (c - M);
        acc.fma(df2{hi[pos], lo[pos]}, ex[up ? c : c - M]);
      }
      zslot[e * M + r] = acc.value();
    }
    __syncthreads();   // the stage just read is the next prefetch target
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

}  // namespace hdg
