// Device-side building blocks shared by the kernels of libfeasm
// (fe_kernels.cu) and the batched persistent driver (fe_batch.cu): cell
// integration of a block of cells, exact FP64 accumulation helpers, and the
// parameter blocks of both phases.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "fe_fixed.cuh"
#include "fe_launch.h"

namespace feasm {

constexpr int kCellThreads = 256;
constexpr int kScatterWarps = 8;




struct CellParams {
  int64_t n_cells;
  int nq, cpb, qblock, nq1d;
  const double* xv;
  const double* w;
  const double* xq;
  const double* phi;
  const float2* phi2;  // [nq][nb] phihat as FP32 hi + lo (hi + lo == phihat to ~2^-48)
  const double* dphi;
  const float* dphi32;
  const double* coef;
  // the fixed-point form (fe_fixed.cuh): sqrt(w_q) dphi_a 2^(60 - lm_a) as 30-bit limbs [nq][nb][3], the
  // exponents lm_a (sum_d |sqrt(w_q) dphi_(a,d)(q)| < 2^lm_a at every point) [nb]
  const int2* dfix;
  const int* fix_lm;
  double f[3];
  double lam_hat, mu_hat;
  void* ke;
  double* fe;
  int* err;
};

__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
// Two values rounded to BF16 (nearest even) by one paired conversion.
__device__ __forceinline__ void round_bf16_pair(float& x, float& y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  x = __low2float(h);
  y = __high2float(h);
}

// Trilinear map Phi(x) = a0 + a1 x + a2 y + a3 z + a4 xy + a5 xz + a6 yz + a7 xyz
// (the Q1 geometry of the cell written in monomials). Its Jacobian at a
// point, the cofactor matrix and the determinant, all FP64:
//   J[k][d] = dPhi_k / dxhat_d,  cof[k][d] = cofactor of J[k][d],
//   det J = sum_d J[0][d] cof[0][d],  J^{-T} = cof / det.
__device__ __forceinline__ void geometry_at(const double* a, double x, double y, double z, double cof[9],
                                            double* det) {
  double J[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double a1 = a[0 + k], a2 = a[3 + k], a3 = a[6 + k], a4 = a[9 + k], a5 = a[12 + k], a6 = a[15 + k],
                 a7 = a[18 + k];
    J[k][0] = a1 + a4 * y + a5 * z + a7 * (y * z);
    J[k][1] = a2 + a4 * x + a6 * z + a7 * (x * z);
    J[k][2] = a3 + a5 * x + a6 * y + a7 * (x * y);
  }
  cof[0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
  cof[1] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
  cof[2] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
  cof[3] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
  cof[4] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
  cof[5] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
  cof[6] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
  cof[7] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
  cof[8] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
  *det = J[0][0] * cof[0] + J[0][1] * cof[1] + J[0][2] * cof[2];
}

// Monomial coefficients a1..a7 (3 components each) from the 8 vertices in
// x-fastest order.
__device__ __forceinline__ void trilinear_coefficients(const double* x, int k, double* a) {
  const double x0 = x[k], x1 = x[3 + k], x2 = x[6 + k], x3 = x[9 + k], x4 = x[12 + k], x5 = x[15 + k],
               x6 = x[18 + k], x7 = x[21 + k];
  const double d10 = x1 - x0, d32 = x3 - x2, d54 = x5 - x4, d76 = x7 - x6, d20 = x2 - x0, d64 = x6 - x4;
  a[0 + k] = d10;
  a[3 + k] = d20;
  a[6 + k] = x4 - x0;
  a[9 + k] = d32 - d10;
  a[12 + k] = d54 - d10;
  a[15 + k] = d64 - d20;
  a[18 + k] = (d76 - d54) - (d32 - d10);
}

// Compensated (Kahan) addition of a block partial into (sum, carry).
template <typename T>
__device__ __forceinline__ void kahan_add(T& sum, T& carry, T part) {
  const T y = part - carry;
  const T t = sum + y;
  carry = (t - sum) - y;
  sum = t;
}

// One block integrates `cpb` cells in FP64 (paper: Eq. fematrix, Eq.
// shape_grad, the element loop of the element-matrix computation):
//   1. geometry at every quadrature point,
//   2. cofactor gradients gh_a = cof(J) gradhat(phihat_a), so that
//      grad(phi_a) = gh_a / det J,
//   3. G^{ij}_{ab} = sum_q (w_q / det J_q) gh_{a,i} gh_{b,j}, and
//      Poisson   K_ab = kappa sum_i G^{ii}_{ab},
//      elasticity K_(a,i),(b,j) = E (lam^ G^{ij}_ab + mu^ G^{ji}_ab + mu^ d_ij sum_k G^{kk}_ab),
//   4. cell vector f_(a,i) = f_i sum_q w_q det J_q phihat_a(x_q).
// Cell matrices are stored row-major with row stride NLP (16-byte aligned
// rows). Shared memory: vertex coordinates [cpb][24], trilinear coefficients
// [cpb][21], per-point geometry [cpb][nq][11] (cofactors, w/det, w*det), the
// cofactor gradients [cpb][nq][3][nb].
//
// Plain FP64 arithmetic: the path of quadrature rules other than (p+1)^3 (HOLD)
// and of the cells that cell_block_fixed does not take (without HOLD: the
// gradients are formed per node pair instead of held in shared memory, so
// that the layout fits the fixed-point kernel's).
template <int P, int NC, bool HOLD>
__device__ __noinline__ void cell_block_plain(const CellParams& prm, int64_t e0, int ncell, double* smem) {
  constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  constexpr int NL = NC * NB;
  constexpr int NLP = (NL + 3) & ~3;
  const int cpb = prm.cpb, nq = prm.nq;
  double* sx = smem;
  double* sa = sx + cpb * 24;
  double* geo = sa + cpb * 21;
  double* g = geo + cpb * nq * 11;
  const int tid = threadIdx.x;

  for (int i = tid; i < ncell * 24; i += blockDim.x) sx[i] = prm.xv[e0 * 24 + i];
  __syncthreads();
  for (int i = tid; i < ncell * 3; i += blockDim.x) trilinear_coefficients(sx + (i / 3) * 24, i % 3, sa + (i / 3) * 21);
  __syncthreads();
  for (int i = tid; i < ncell * nq; i += blockDim.x) {
    const int c = i / nq, q = i % nq;
    double cof[9], det;
    geometry_at(sa + c * 21, prm.xq[3 * q], prm.xq[3 * q + 1], prm.xq[3 * q + 2], cof, &det);
    if (!(det > 0.0)) atomicOr(prm.err, kErrNegJacobian);
    const double wq = prm.w[q];
    double* gm = geo + size_t(i) * 11;
#pragma unroll
    for (int t = 0; t < 9; ++t) gm[t] = cof[t];
    gm[9] = wq / det;
    gm[10] = wq * det;
  }
  __syncthreads();
  auto gradient = [&](const double* gm, int q, int a, int k) {
    const double* dp = prm.dphi + (size_t(q) * NB + a) * 3;
    return gm[3 * k] * dp[0] + gm[3 * k + 1] * dp[1] + gm[3 * k + 2] * dp[2];
  };
  if (HOLD) {
    for (int i = tid; i < ncell * nq * NB; i += blockDim.x) {
      const int a = i % NB, cq = i / NB, q = cq % nq;
#pragma unroll
      for (int k = 0; k < 3; ++k) g[(size_t(cq) * 3 + k) * NB + a] = gradient(geo + size_t(cq) * 11, q, a, k);
    }
    __syncthreads();
  }
  for (int i = tid; i < ncell * NB * NB; i += blockDim.x) {
    const int c = i / (NB * NB), ab = i % (NB * NB), a = ab / NB, b = ab % NB;
    const double* gm = geo + size_t(c) * nq * 11;
    const int64_t e = e0 + c;
    const double coef = prm.coef[e];
    double* K = reinterpret_cast<double*>(prm.ke) + e * NL * NLP;
    double S[NC == 1 ? 1 : 3][3];
#pragma unroll
    for (int i2 = 0; i2 < (NC == 1 ? 1 : 3); ++i2)
#pragma unroll
      for (int j2 = 0; j2 < 3; ++j2) S[i2][j2] = 0.0;
    for (int q = 0; q < nq; ++q) {
      const double* gq = g + (size_t(c) * nq + q) * 3 * NB;
      const double s = gm[q * 11 + 9];
      double ga[3], gb[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        ga[k] = s * (HOLD ? gq[k * NB + a] : gradient(gm + q * 11, q, a, k));
        gb[k] = HOLD ? gq[k * NB + b] : gradient(gm + q * 11, q, b, k);
      }
      if (NC == 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) S[0][0] += ga[k] * gb[k];
      } else {
#pragma unroll
        for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
          for (int j2 = 0; j2 < 3; ++j2) S[NC == 1 ? 0 : i2][j2] += ga[i2] * gb[j2];
      }
    }
    if (NC == 1) {
      K[a * NLP + b] = coef * S[0][0];
    } else {
      const double lh = prm.lam_hat, mh = prm.mu_hat;
      const double tr = S[0][0] + S[1 % (NC == 1 ? 1 : 3)][1] + S[2 % (NC == 1 ? 1 : 3)][2];
#pragma unroll
      for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
        for (int j2 = 0; j2 < 3; ++j2) {
          double v = lh * S[NC == 1 ? 0 : i2][j2] + mh * S[NC == 1 ? 0 : j2][i2];
          if (i2 == j2) v += mh * tr;
          K[size_t(i2 * NB + a) * NLP + j2 * NB + b] = coef * v;
        }
    }
  }
  for (int i = tid; i < ncell * NB; i += blockDim.x) {
    const int c = i / NB, a = i % NB;
    const double* gm = geo + size_t(c) * nq * 11;
    double f = 0.0;
    for (int q = 0; q < nq; ++q) f += gm[q * 11 + 10] * prm.phi[size_t(q) * NB + a];
    double* fe = prm.fe + (e0 + c) * NL;
#pragma unroll
    for (int k = 0; k < NC; ++k) fe[k * NB + a] = prm.f[k] * f;
  }
}


// One block integrates `cpb` cells in the FP64 form with the contraction in
// fixed point (fe_fixed.cuh). FP64 arithmetic is left where it is needed, in
// the geometry of each quadrature point; GB300's FP64 pipe would take 9/2 nb^2
// nq multiply-adds per cell of elasticity otherwise. Steps:
//   1. Jacobian columns once per pair of 1D points (each depends on two of the
//      reference coordinates), per point cofactors, det J and
//      C = cof(J) / sqrt(det J) in FP64; 1/sqrt(det J) from the FP32 estimate
//      and one cubic correction (5 FP64 operations); C as 60-bit integers with
//      a power-of-two scale per point and component, and the largest of these
//      scales per cell and component (all three share one for Poisson);
//   2. operands v_(a,i)(q) = sum_d C_id sqrt(w_q) dphi_(a,d)(q) in integers (the
//      weights are in the table), rounded to kFixBits bits below the bound of
//      node a and component i in the cell;
//   3. G^ij_ab = sum_q v_(a,i) v_(b,j) in integers for node pairs a <= b, the
//      coefficient and the elasticity law in integers, one conversion to
//      double per entry, stored to (a, b) and (b, a). The lo lo products are
//      in the sums that hold squares for a = b: left out there they lower the
//      diagonal by 6e-17 of itself in every cell (displacement of a clamped
//      uniform beam of 16 x 9 x 8 cells, against extended precision: 1.0e-14
//      with them, 1.2e-13 without, 5.0e-14 with FP64 products; of 31 x 21 x 19
//      cells 1.9e-13, 1.7e-13 and 3.1e-13: few distinct entries, so that their
//      roundings do not average out);
//   4. cell vectors in FP64.
// Bound by: the integer multiply-adds of step 3 (IMAD.WIDE, 25 to 32 lanes per
// clock per SM) and the conversions to double (ALU pipe 54 % busy in Q1
// elasticity, 47 % in Q2; FP64 pipe 35 % and 8 %).
// Measured against the FP64 multiply-adds (cell_block_plain), ms: Poisson Q1
// 64^3 2.01 -> 0.42, Q2 32^3 7.44 -> 0.86, Q3 24^3 39.1 -> 4.4; elasticity Q1
// 64^3 4.31 -> 0.74, Q2 24^3 6.47 -> 0.77, Q3 12^3 10.2 -> 1.13. Error in the
// 2-norm against extended precision no larger (Q1 elasticity 6.8e-16 after
// 7.0e-16, Q2 6.7e-16 after 6.8e-16, Q3 9.2e-16 after 9.4e-16, Poisson Q2
// 5.7e-16 after 6.1e-16, Q3 8.0e-16 after 9.6e-16).
// Poisson takes a T x T tile of node pairs per thread, one tile each, and goes
// through the operands slab by slab of p2 points, so that they take little
// shared memory; elasticity takes one node pair (nine sums) per thread at a
// time.
// Returns false, with nothing written but the error bit, if a cell is out of
// the range of this form (det J <= 0, infinities, NaN, |C| outside 2^+-200,
// a nonzero coefficient outside 2^+-400): the caller then takes
// cell_block_plain, which propagates them.
// Shared memory, within cell_block_plain's layout: vertex coordinates
// [cpb][24], then in their place the per-cell scales and law multipliers;
// trilinear coefficients [cpb][21]; per point 11 doubles' space (C as 9 limb
// pairs, w det J, the scales); then the Jacobian columns [cpb][3][p2][3] and
// in their place the operands, limb pairs [cell][q][a][3].
// For the (P + 1)^3 rule (compile-time index arithmetic); other rules take
// cell_block_plain.
template <int P, int NC>
struct FixedShape {
  static constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  static constexpr int T = NB == 64 ? 4 : NB == 27 ? 3 : 2;    // Poisson tile
  static constexpr int NT = NB / T, TILES = NT * (NT + 1) / 2;
  static constexpr bool SLAB = NC == 1 && NB >= 27;            // operands slab by slab
  static constexpr bool LOLO = NB * (NC == 1 ? 3 : 1) > 30;    // 32-bit limbs with lo lo in FP32
  // threads and cells of a k_cell block (measured, 64^3 Q1, 32^3 / 24^3 Q2, 24^3 / 12^3 Q3 cells)
  static constexpr int THREADS = NC == 1 ? (NB == 8 ? 128 : NB == 27 ? 96 : 192) : (NB == 8 ? 64 : NB == 27 ? 128 : 256);
  static constexpr int CELLS = NC == 1 ? (NB == 8 ? 8 : NB == 27 ? 2 : 1) : (NB == 8 ? 7 : NB == 27 ? 2 : 1);
  static constexpr int QS = SLAB ? (P + 1) * (P + 1) : NB;     // points whose operands are held
  static constexpr long smem(int cpb) { return long(cpb) * (24 + 21 + 11 * NB + 3 * NB * QS) * 8; }
};

template <int P, int NC>
__device__ __forceinline__ bool cell_block_fixed(const CellParams& prm, int64_t e0, int ncell, double* smem) {
  using F = FixedShape<P, NC>;
  constexpr int NB = F::NB, NL = NC * NB, NLP = (NL + 3) & ~3;
  constexpr int n1d = P + 1, p2 = n1d * n1d, nq = NB, QS = F::QS;
  constexpr bool LOLO = F::LOLO;
  const int cpb = prm.cpb;
  constexpr int B = kFixBits;
  double* sx = smem;
  int4* slaw = reinterpret_cast<int4*>(smem);                  // [cpb] law multipliers as halves
  int* sexp = reinterpret_cast<int*>(slaw + cpb);              // [cpb][4] scales per component; exponent of slaw
  int64_t* smu = reinterpret_cast<int64_t*>(sexp + 4 * cpb);   // [cpb] the multiplier of the trace
  double* sa = sx + cpb * 24;
  double* geo = sa + cpb * 21;
  double* sj = geo + cpb * nq * 11;
  int2* g = reinterpret_cast<int2*>(sj);
  const int tid = threadIdx.x, nt = blockDim.x;
  bool odd = false;

  for (int i = tid; i < ncell * 24; i += nt) sx[i] = prm.xv[e0 * 24 + i];
  __syncthreads();
  for (int i = tid; i < ncell * 3; i += nt) trilinear_coefficients(sx + (i / 3) * 24, i % 3, sa + (i / 3) * 21);
  __syncthreads();
  for (int i = tid; i < ncell; i += nt) {
    sexp[4 * i] = sexp[4 * i + 1] = sexp[4 * i + 2] = 0;
    // coefficient times the law's constants (lambda, mu) as integers below 2^60
    const double cf = prm.coef[e0 + i];
    const double c0 = NC == 1 ? cf : cf * prm.lam_hat, c1 = NC == 1 ? 0.0 : cf * prm.mu_hat;
    const int w = max(__double2hiint(c0) & 0x7fffffff, __double2hiint(c1) & 0x7fffffff), eb = w >> 20;
    odd |= w != 0 && (eb < 622 || eb > 1422);
    const int ec = w == 0 ? 0 : eb - 1022;
    sexp[4 * i + 3] = ec;
    int4 m = make_int4(0, 0, 0, 0);
    if (NC == 1) {
      fix_halves(fix_quantise(c0, 61 - ec), m.x, m.y);
    } else {
      // lambda + mu, lambda - mu for the off-diagonal pairs; lambda + mu and mu for the diagonal
      const int64_t l = fix_quantise(c0, 60 - ec), u = fix_quantise(c1, 60 - ec);
      fix_halves(l + u, m.x, m.y);
      fix_halves(l - u, m.z, m.w);
      smu[i] = u;
    }
    slaw[i] = m;
  }
  for (int i = tid; i < ncell * 9 * p2; i += nt) {
    const int c = i / (9 * p2), r = i % (9 * p2), d = r / (3 * p2), rem = r % (3 * p2), pr = rem / 3, k = rem % 3;
    const double* a = sa + c * 21;
    const double u = prm.xq[3 * (pr % n1d)], v = prm.xq[3 * (pr / n1d)];
    const int o0 = 3 * d, ou = d == 2 ? 12 : 9, ov = d == 0 ? 12 : 15;
    sj[i] = fma(fma(a[18 + k], v, a[ou + k]), u, fma(a[ov + k], v, a[o0 + k]));
  }
  __syncthreads();
  for (int i = tid; i < ncell * nq; i += nt) {
    const int c = i / nq, q = i % nq;
    const int ix = q % n1d, iy = (q / n1d) % n1d, iz = q / p2;
    const double* jc = sj + c * 9 * p2;
    double J[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      J[k][0] = jc[(0 * p2 + iy + n1d * iz) * 3 + k];
      J[k][1] = jc[(1 * p2 + ix + n1d * iz) * 3 + k];
      J[k][2] = jc[(2 * p2 + ix + n1d * iy) * 3 + k];
    }
    double cof[9];
    cof[0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    cof[1] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    cof[2] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    cof[3] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    cof[4] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    cof[5] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    cof[6] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    cof[7] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    cof[8] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double det = J[0][0] * cof[0] + J[0][1] * cof[1] + J[0][2] * cof[2];
    if (!(det > 0.0)) atomicOr(prm.err, kErrNegJacobian);
    int k2;
    const double y = fix_rsqrt(det, k2, odd);
    const double t = fix_scale2(y, -k2);
    double* gm = geo + size_t(i) * 11;
    gm[9] = prm.w[q] * det;
    int m[3];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      cof[j] *= t;
      const int h = __double2hiint(cof[j]) & 0x7fffffff;
      m[j / 3] = j % 3 == 0 ? h : max(m[j / 3], h);
    }
    if (NC == 1) m[0] = m[1] = m[2] = max(m[0], max(m[1], m[2]));
    int pack = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int eb = m[j] >> 20;                               // |C_j.| < 2^(eb - 1022)
      odd |= eb != 0 && (eb < 822 || eb > 1222);
      const int ee = eb == 0 ? 0 : (eb - 821) & 0x1ff;         // 1..401; 0: the row is zero
      pack |= ee << (9 * j);
      if (NC == 3 || j == 0) atomicMax(sexp + c * 4 + j, ee);
#pragma unroll
      for (int d = 0; d < 3; ++d)
        reinterpret_cast<int2*>(gm)[3 * j + d] = fix_limbs<30>(fix_quantise(cof[3 * j + d], 60 - (eb - 1022)));
    }
    *reinterpret_cast<int*>(gm + 10) = pack;
  }
  if (__syncthreads_or(odd)) return false;
  // |C| < 2^scale_of in the cell
  auto scale_of = [&](int c, int j) { return sexp[c * 4 + (NC == 1 ? 0 : j)] - 201; };
  // operands of the points [q0, q0 + QS): v_(a,i) = operand times 2^(B - scale_of(i) - lm_a)
  auto operands = [&](int q0) {
    for (int i = tid; i < ncell * QS * NB; i += nt) {
      const int a = i % NB, c = i / (NB * QS), q = q0 + (i / NB) % QS;
      const double* gm = geo + (c * nq + q) * 11;
      const int2* C = reinterpret_cast<const int2*>(gm);
      const int pack = *reinterpret_cast<const int*>(gm + 10);
      const int2* dp = prm.dfix + (q * NB + a) * 3;
      const int2 d0 = __ldg(dp), d1 = __ldg(dp + 1), d2 = __ldg(dp + 2);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        FixAcc<30> s;
        s.zero();
        s.add(C[3 * k], d0);
        s.add(C[3 * k + 1], d1);
        s.add(C[3 * k + 2], d2);
        const int sh = min(60 - B + sexp[c * 4 + (NC == 1 ? 0 : k)] - ((pack >> (9 * k)) & 0x1ff), 62);
        g[i * 3 + k] = fix_limbs<LOLO ? 32 : 30>(s.get_shifted(sh));
      }
    }
  };
  if constexpr (NC == 1) {
    constexpr int T = F::T;
    // one tile per thread (the launch has at least cpb * TILES threads)
    const int c = tid / F::TILES;
    const bool has = c < ncell;
    int ta = 0, tb = 0;
    if (has) fix_pair(tid % F::TILES, ta, tb);
    const int a0 = ta * T, b0 = tb * T;
    FixAcc<LOLO ? 32 : 30> S[T][T];
    float L[T][T];
    int64_t sq[T] = {};  // lo lo of the tile's diagonal
#pragma unroll
    for (int u = 0; u < T; ++u)
#pragma unroll
      for (int v = 0; v < T; ++v) S[u][v].zero(), L[u][v] = 0.f;
    for (int q0 = 0; q0 < nq; q0 += QS) {
      if (q0) __syncthreads();
      operands(q0);
      __syncthreads();
      if (has) {
        const int2* gq = g + c * QS * NB * 3;
        for (int q = 0; q < QS; ++q, gq += NB * 3) {
          if (q > 0 && q % (kFixDrainEvery / 3) == 0) {
#pragma unroll
            for (int u = 0; u < T; ++u)
#pragma unroll
              for (int v = 0; v < T; ++v) S[u][v].drain();
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            int2 va[T], vb[T];
#pragma unroll
            for (int u = 0; u < T; ++u) va[u] = gq[(a0 + u) * 3 + k], vb[u] = gq[(b0 + u) * 3 + k];
            if (LOLO) {
              float fa[T], fb[T];
#pragma unroll
              for (int u = 0; u < T; ++u) fa[u] = float(va[u].y), fb[u] = float(vb[u].y);
#pragma unroll
              for (int u = 0; u < T; ++u)
#pragma unroll
                for (int v = 0; v < T; ++v) L[u][v] = fmaf(fa[u], fb[v], L[u][v]);
            }
#pragma unroll
            for (int u = 0; u < T; ++u)
#pragma unroll
              for (int v = 0; v < T; ++v) S[u][v].add(va[u], vb[v]);
            if (!LOLO) {
#pragma unroll
              for (int u = 0; u < T; ++u) mad_wide(sq[u], va[u].y, vb[u].y);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < T; ++u)
#pragma unroll
          for (int v = 0; v < T; ++v) S[u][v].drain();
      }
    }
    if (has) {
      const int64_t e = e0 + c;
      const int4 m = slaw[c];
      uint32_t mag = 0;
#pragma unroll
      for (int u = 0; u < T; ++u)
#pragma unroll
        for (int v = 0; v < T; ++v) {
          if (LOLO) S[u][v].add_low(L[u][v]);
          if (!LOLO && u == v) S[u][v].add_low(sq[u]);
          mag |= S[u][v].magnitude();
        }
      const int sh = fix_shift(mag);
      const int ex = 5 + 2 * (LOLO ? 32 : 30) - sh - 2 * (B - scale_of(c, 0)) + sexp[c * 4 + 3];
      int la[T], lb[T];
#pragma unroll
      for (int u = 0; u < T; ++u) la[u] = __ldg(prm.fix_lm + a0 + u), lb[u] = __ldg(prm.fix_lm + b0 + u);
      double* K = reinterpret_cast<double*>(prm.ke) + e * NL * NLP;
#pragma unroll
      for (int u = 0; u < T; ++u)
#pragma unroll
        for (int v = 0; v < T; ++v) {
          const double r = fix_to_double(fix_mul(S[u][v].get(sh), m.x, m.y), fix_exponent(ex + la[u] + lb[v]));
          K[(a0 + u) * NLP + b0 + v] = r;
          K[(b0 + v) * NLP + a0 + u] = r;
        }
    }
  } else {
    operands(0);
    __syncthreads();
    constexpr int NP = NB * (NB + 1) / 2;
    for (int i = tid; i < ncell * NP; i += nt) {
      const int c = i / NP;
      int a, b;
      fix_pair(i % NP, a, b);
      FixAcc<LOLO ? 32 : 30> S[3][3];
      float L[3][3];
      int64_t sq[3] = {};  // lo lo of the diagonal sums
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) S[u][v].zero(), L[u][v] = 0.f;
      const int2* ga = g + (c * nq * NB + a) * 3;
      const int2* gb = g + (c * nq * NB + b) * 3;
      constexpr int DQ = nq % 12 == 0 ? 12 : nq % 9 == 0 ? 9 : 8;
      static_assert(DQ <= kFixDrainEvery && nq % DQ == 0, "drain");
      for (int q0 = 0; q0 < nq; q0 += DQ) {
#pragma unroll 4
        for (int q = 0; q < DQ; ++q, ga += NB * 3, gb += NB * 3) {
          int2 va[3], vb[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) va[k] = ga[k], vb[k] = gb[k];
          if (LOLO) {
            float fa[3], fb[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) fa[k] = float(va[k].y), fb[k] = float(vb[k].y);
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
              for (int v = 0; v < 3; ++v) L[u][v] = fmaf(fa[u], fb[v], L[u][v]);
          }
#pragma unroll
          for (int u = 0; u < 3; ++u)
#pragma unroll
            for (int v = 0; v < 3; ++v) S[u][v].add(va[u], vb[v]);
          if (!LOLO) {
#pragma unroll
            for (int k = 0; k < 3; ++k) mad_wide(sq[k], va[k].y, vb[k].y);
          }
        }
#pragma unroll
        for (int u = 0; u < 3; ++u)
#pragma unroll
          for (int v = 0; v < 3; ++v) S[u][v].drain();
      }
      // the nine sums shifted to just below 2^61, then the law
      int s[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) s[k] = B - scale_of(c, k);
      const int smin = min(s[0], min(s[1], s[2]));
      uint32_t mag = 0;
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          if (LOLO) S[u][v].add_low(L[u][v]);
          if (!LOLO && u == v) S[u][v].add_low(sq[u]);
          mag |= S[u][v].magnitude();
        }
      const int sh = fix_shift(mag);
      const int64_t e = e0 + c;
      const int4 m = slaw[c];
      const int ex = 5 + 2 * (LOLO ? 32 : 30) - sh + sexp[c * 4 + 3] + __ldg(prm.fix_lm + a) + __ldg(prm.fix_lm + b);
      double* K = reinterpret_cast<double*>(prm.ke) + e * NL * NLP;
      auto put = [&](int u, int v, double r) {
        K[(u * NB + a) * NLP + v * NB + b] = r;
        K[(v * NB + b) * NLP + u * NB + a] = r;
      };
      // K^ij = lambda G^ij + mu G^ji through the sum and difference of the two
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int v = u + 1; v < 3; ++v) {
          const int64_t x = S[u][v].get(sh), z = S[v][u].get(sh);
          const int64_t p = fix_mul(x + z, m.x, m.y), d = fix_mul(x - z, m.z, m.w);
          const int field = fix_exponent(ex - s[u] - s[v]);
          put(u, v, fix_to_double(p + d, field));
          put(v, u, fix_to_double(p - d, field));
        }
      // K^ii = (lambda + mu) G^ii + mu tr G, the diagonal sums in the coarsest of their units
      int64_t t[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int n = min(2 * (s[k] - smin), 62);
        t[k] = S[k][k].get(sh);
        if (n > 0) t[k] = ((t[k] >> (n - 1)) + 1) >> 1;
      }
      int mh, ml;
      fix_halves(smu[c], mh, ml);
      const int64_t tr = fix_mul(t[0] + t[1] + t[2], mh, ml);
#pragma unroll
      for (int k = 0; k < 3; ++k) put(k, k, fix_to_double(fix_mul(t[k], m.x, m.y) + tr, fix_exponent(ex + 1 - 2 * smin)));
    }
  }
  for (int i = tid; i < ncell * NB; i += nt) {
    const int c = i / NB, a = i % NB;
    const double* gm = geo + c * nq * 11 + 9;
    double f = 0.0;
    for (int q = 0; q < nq; ++q) f += gm[q * 11] * prm.phi[q * NB + a];
    double* fe = prm.fe + (e0 + c) * NL;
#pragma unroll
    for (int k = 0; k < NC; ++k) fe[k * NB + a] = prm.f[k] * f;
  }
  return true;
}

// Cell integration of one block of cells in the FP64 form.
template <int P, int NC>
__device__ __forceinline__ void cell_block_fp64(const CellParams& prm, int64_t e0, int ncell, double* smem) {
  if (prm.nq1d != P + 1) {
    cell_block_plain<P, NC, true>(prm, e0, ncell, smem);
  } else if (!cell_block_fixed<P, NC>(prm, e0, ncell, smem)) {
    cell_block_plain<P, NC, false>(prm, e0, ncell, smem);
  }
}

// Exact FP64 accumulation without FP64 arithmetic. The FP64 pipe of this GPU
// is a small fraction of its FP32/INT32 rate, so each nonzero is summed in
// 64-bit integer fixed point: every term is split into sign, exponent and
// integer mantissa, the mantissas are aligned to the largest exponent of the
// nonzero (the largest term's leading bit at bit 57, so that up to 32 terms
// cannot overflow) and added as int64, and the integer sum is rounded once to
// the nearest double. Bits lost in the alignment are below 2^-57 of the
// largest term, so the result is at least as accurate as sequential FP64
// additions, is independent of the order of the terms, and is bitwise
// reproducible. A nonzero with a single FP32 term takes the exact FP32->FP64
// conversion, done on the integer bits.
template <typename TK>
struct FxTraits;
template <>
struct FxTraits<float> {
  // value = mant * 2^(ex - 150), mant < 2^24; aligned mantissa MSB at bit 57
  static constexpr int kShift0 = 34, kScale = 184;
  __device__ static __forceinline__ void split(float x, uint64_t& m, int& ex, bool& neg) {
    const uint32_t u = __float_as_uint(x);
    neg = (u >> 31) != 0;
    int e = int((u >> 23) & 0xffu);
    uint32_t mm = u & 0x7fffffu;
    if (e) mm |= 0x800000u; else e = 1;
    m = mm;
    ex = e;
  }
};
template <>
struct FxTraits<double> {
  // value = mant * 2^(ex - 1075), mant < 2^53; aligned mantissa MSB at bit 57
  static constexpr int kShift0 = 5, kScale = 1080;
  __device__ static __forceinline__ void split(double x, uint64_t& m, int& ex, bool& neg) {
    const uint64_t u = uint64_t(__double_as_longlong(x));
    neg = (u >> 63) != 0;
    int e = int((u >> 52) & 0x7ffu);
    uint64_t mm = u & 0xfffffffffffffull;
    if (e) mm |= 1ull << 52; else e = 1;
    m = mm;
    ex = e;
  }
};

// Rounds the integer S * 2^scale to the nearest double (ties to even).
__device__ __forceinline__ double fx_to_double(int64_t S, int scale) {
  if (S == 0) return 0.0;
  const bool neg = S < 0;
  const uint64_t mag = neg ? uint64_t(-S) : uint64_t(S);
  int lz = __clzll(static_cast<long long>(mag));
  const uint64_t norm = mag << lz;
  uint64_t mant = norm >> 11;
  const uint32_t rem = uint32_t(norm & 0x7ffu);
  if (rem > 0x400u || (rem == 0x400u && (mant & 1u))) ++mant;
  if (mant >> 53) {
    mant >>= 1;
    --lz;
  }
  const int biased = 63 - lz + scale + 1023;
  if (biased <= 0) return neg ? -0.0 : 0.0;
  if (biased >= 2047) return neg ? -__longlong_as_double(0x7ff0000000000000ll) : __longlong_as_double(0x7ff0000000000000ll);
  const uint64_t bits = (uint64_t(neg) << 63) | (uint64_t(biased) << 52) | (mant & 0xfffffffffffffull);
  return __longlong_as_double(static_cast<long long>(bits));
}

// Exact FP32 -> FP64 conversion on the integer bits (normal numbers and zero).
__device__ __forceinline__ bool f32_to_f64_bits(float x, double& out) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t e = (u >> 23) & 0xffu;
  if ((u & 0x7fffffffu) == 0) {
    out = (u >> 31) ? -0.0 : 0.0;
    return true;
  }
  if (e == 0 || e == 0xffu) return false;
  const uint64_t bits = (uint64_t(u >> 31) << 63) | (uint64_t(e + 896u) << 52) | (uint64_t(u & 0x7fffffu) << 29);
  out = __longlong_as_double(static_cast<long long>(bits));
  return true;
}

// Sum of n terms produced by get(t), t = 0..n-1, accumulated exactly as above.
template <typename TK, typename Get>
__device__ __forceinline__ double fx_sum(int n, Get get) {
  using Tr = FxTraits<TK>;
  if (n == 1) {
    const TK x = get(0);
    if (sizeof(TK) == 8) return double(x);
    double d;
    if (f32_to_f64_bits(float(x), d)) return d;
  }
  int emax = 1;
  for (int t = 0; t < n; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(get(t), m, ex, ng);
    if (m != 0 && ex > emax) emax = ex;
  }
  int64_t S = 0;
  for (int t = 0; t < n; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(get(t), m, ex, ng);
    const int sh = Tr::kShift0 - (emax - ex);
    const uint64_t a = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> (-sh)) : 0ull);
    S += ng ? -int64_t(a) : int64_t(a);
  }
  return fx_to_double(S, emax - Tr::kScale);
}


// fx_sum of N terms held in registers (zeros pad a shorter list): the same
// fixed-point sum and rounding, so the same result, without a second pass
// over memory.
template <int N>
__device__ __forceinline__ double fx_sum_regs(const double (&v)[N]) {
  using Tr = FxTraits<double>;
  int emax = 1;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(v[t], m, ex, ng);
    if (m != 0 && ex > emax) emax = ex;
  }
  int64_t S = 0;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(v[t], m, ex, ng);
    const int sh = Tr::kShift0 - (emax - ex);
    const uint64_t a = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> (-sh)) : 0ull);
    S += ng ? -int64_t(a) : int64_t(a);
  }
  return fx_to_double(S, emax - Tr::kScale);
}

// One-pass form of the same sum, term by term in the given order: a 64-bit
// integer S with an exponent e (value S 2^(e - 1080)); a term is its mantissa
// shifted left by 5 (leading bit at bit 57, room for 32 terms), and the smaller
// of accumulator and term is shifted right to the larger exponent before the
// integer addition. Bits lost are below 2^-57 of the largest term so far. The
// shift rounds down, which would be a bias if every sum of a matrix did so (with
// coefficients that differ by 2^8 and more between cells the sum of all entries
// was up to 3.8 times what independent roundings allow; cut off towards zero
// still 1.8 times, as the diagonal has more terms than the others). So half of
// the rows, by a hash of the first cell-matrix row they sum (the same in every
// pattern that keeps the row), sum the negated terms: one instruction per term,
// where rounding each shift would take four.
struct FxChain {
  int64_t S;
  int e;
  // 0, or -1 where the row whose first slot (cell-matrix row) is `slot` sums the negated terms
  __device__ __forceinline__ static int flip_of(int slot) { return int(uint32_t(slot) * 0x9e3779b1u) >> 31; }
  __device__ __forceinline__ static FxChain term(double x, int flip) {
    const int hi = __double2hiint(x), lo = __double2loint(x), eb = (hi >> 20) & 0x7ff;
    const uint32_t mh = uint32_t(hi & 0xfffff) | (eb != 0 ? 0x100000u : 0u);
    const int64_t m = int64_t((uint64_t(__funnelshift_l(uint32_t(lo), mh, 5)) << 32) | (uint32_t(lo) << 5));
    const int64_t sg = int64_t((hi >> 31) ^ flip);
    return FxChain{(m ^ sg) - sg, eb};  // (denormals: half of their value, but odd() unless nothing of them is left)
  }
  __device__ __forceinline__ void add(const FxChain& t) {
    const int m = max(e, t.e);
    S = shift_down(S, m - e) + shift_down(t.S, m - t.e);
    e = m;
  }
  // x / 2^d rounded down, d of any size (shr clamps it, >> in C++ does not)
  __device__ __forceinline__ static int64_t shift_down(int64_t x, int d) {
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));
    return r;
  }
  // near the ends of the exponent range (infinities, NaN, denormals): the sum is redone with fx_sum
  __device__ __forceinline__ bool odd() const { return (e < 80 && S != 0) || e > 2000; }
  // the row's sum rounded to the nearest double (ties to even); not if odd()
  __device__ __forceinline__ double round(int flip) const {
    const uint64_t s = uint64_t(S >> 63);
    const uint64_t mag = (uint64_t(S) ^ s) - s;
    const int lz = __clzll(static_cast<long long>(mag));
    const uint64_t norm = mag << (lz & 63);
    const uint32_t nh = uint32_t(norm >> 32), nl = uint32_t(norm);
    const uint32_t rem = nl & 0x7ffu, last = (nl >> 11) & 1u;
    uint64_t bits = (uint64_t(uint32_t(63 - lz + e - 1080 + 1022) << 20) << 32) +
                    ((uint64_t(nh >> 11) << 32) | __funnelshift_r(nl, nh, 11)) + (rem + last > 0x400u ? 1u : 0u);
    bits |= (s ^ uint64_t(int64_t(flip))) & 0x8000000000000000ull;
    return __longlong_as_double(static_cast<long long>(mag == 0 ? 0ull : bits));
  }
};

struct ScatterParams {
  int64_t n_rows;
  int nl, nlp;
  const int64_t* row_ptr;
  const uint8_t* cnt;
  const int64_t* code_ptr;
  const uint16_t* codes;
  const uint16_t* pos;
  const int64_t* slot_ptr;
  const int32_t* slots;
  const int32_t* ncode;  // codes per row (constrained patterns), or nullptr: slots * nl
  unsigned long long* sched;  // [2] item counters of the dynamic schedule, zero between launches
  const void* ke;
  const double* fe;
  double* values;
  double* rhs;
  int ke_bytes, code_bytes, warp_bytes, acc_stride;
};

constexpr unsigned kFull = 0xffffffffu;

// Dynamic assignment of work items (CSR rows, or the rows of one node) to the
// warps of a scatter launch. A warp takes `grab` consecutive items at a time
// from a counter in device memory (one atomicAdd by lane 0) and holds its next
// grab in reserve, so that the atomic's latency hides behind the current
// items. Rows differ in cost (a node lies in 1, 2, 4 or 8 cells, in a pattern
// that repeats every few tens of rows and shifts wherever rows are dropped);
// any static cyclic schedule lets that pattern line up with the warp index
// for some meshes and warp counts, so that a few warps collect the expensive
// rows. Taking items on demand balances the warps to within one grab, while
// the items in flight still form one contiguous window of rows. Every warp
// calls finish() once at the end; the last one resets both counters (next
// item, finished warps) to zero for the next launch on the stream.
struct ItemStream {
  unsigned long long* ctr;
  int64_t n, u, end, nxt;
  int grab;
  __device__ __forceinline__ int64_t take(int lane) const {
    unsigned long long b = 0;
    if (lane == 0) b = atomicAdd(ctr, static_cast<unsigned long long>(grab));
    return static_cast<int64_t>(__shfl_sync(kFull, b, 0));
  }
  __device__ __forceinline__ ItemStream(unsigned long long* c, int64_t n_items, int grab_size, int lane)
      : ctr(c), n(n_items), grab(grab_size) {
    u = take(lane);
    end = u + grab < n ? u + grab : n;
    nxt = take(lane);
  }
  __device__ __forceinline__ bool valid() const { return u < n; }
  // the item after the current one (>= n: no more); takes a new reserve grab when needed
  __device__ __forceinline__ void advance(int lane) {
    if (u + 1 < end) {
      ++u;
    } else {
      u = nxt;
      end = u + grab < n ? u + grab : n;
      nxt = u < n ? take(lane) : u;
    }
  }
  __device__ __forceinline__ void finish(int64_t n_warps, int lane) const {
    if (lane == 0) {
      __threadfence();
      if (atomicAdd(ctr + 1, 1ull) == static_cast<unsigned long long>(n_warps - 1)) {
        atomicExch(ctr, 0ull);
        atomicExch(ctr + 1, 0ull);
      }
    }
  }
};


// Exact FP32 -> FP64 conversion on the integer bits (denormals included),
// without the FP64 pipe; infinities and NaNs take the hardware conversion.
static __device__ __noinline__ double f2d_slow(float x) { return double(x); }
__device__ __forceinline__ double f32_to_f64_exact(float x) {
  double d;
  if (f32_to_f64_bits(x, d)) return d;
  if ((__float_as_uint(x) & 0x7f800000u) == 0x7f800000u) return f2d_slow(x);
  uint64_t m;
  int ex;
  bool ng;
  FxTraits<float>::split(x, m, ex, ng);
  return fx_to_double(ng ? -int64_t(m) : int64_t(m), ex - 150);
}

// FP32 -> FP64, exact, for zero and normal numbers, in 32-bit integer
// operations: the high word is the sign, the exponent rebiased by
// 1023 - 127 = 896 and the top 20 mantissa bits, i.e. sign | ((|x| >> 3) +
// (896 << 20)); the low word holds the last 3 mantissa bits, |x| << 29.
__device__ __forceinline__ double f32_to_f64_normal(float x) {
  const uint32_t u = __float_as_uint(x), mag = u & 0x7fffffffu, sgn = u & 0x80000000u;
  const uint32_t hw = mag == 0 ? sgn : (sgn | ((mag >> 3) + 0x38000000u));
  return __hiloint2double(int(hw), int(mag << 29));
}

// True for zero and FP32-normal x (exponent field 1..254).
__device__ __forceinline__ bool f32_zero_or_normal(float x) {
  const uint32_t mag = __float_as_uint(x) & 0x7fffffffu;
  return mag == 0 || mag - 0x00800000u < 0x7f000000u;
}

// hi + lo of a double-float accumulator, rounded once to the nearest double:
// both parts convert exactly on the integer bits and one FP64 addition rounds
// their exact sum (lo == 0 keeps hi, sign of zero included). Branch-free; a
// warp vote sends the whole warp to the general conversion in the rare case of
// a denormal part. All 32 lanes of the warp must call it.
__device__ __forceinline__ double df_to_double(float hi, float lo) {
  double dh, dl;
  if (__all_sync(kFull, f32_zero_or_normal(hi) && f32_zero_or_normal(lo))) {
    dh = f32_to_f64_normal(hi);
    dl = f32_to_f64_normal(lo);
  } else {
    dh = f32_to_f64_exact(hi);
    dl = f32_to_f64_exact(lo);
  }
  const double sum = __dadd_rn(dh, dl);
  return lo == 0.f ? dh : sum;
}


// FP64 -> FP32 round to nearest even on the integer bits (zero and
// FP32-normal results; values that would under- or overflow FP32 take the
// hardware conversion, out of line). Keeps the conversions of the FP64 geometry off the FP64 pipe.
static __device__ __noinline__ float d2f_slow(double x) { return __double2float_rn(x); }
__device__ __forceinline__ float d2f_rn(double x) {
  const uint64_t u = uint64_t(__double_as_longlong(x));
  const int e = int((u >> 52) & 0x7ffu) - 896;
  if (e <= 0 || e >= 255) {
    if ((u << 1) == 0) return __uint_as_float(uint32_t(u >> 63) << 31);
    return d2f_slow(x);  // out of line: FP64-pipe instructions on a predicated path still occupy the pipe
  }
  const uint64_t mant = u & 0xfffffffffffffull;
  uint32_t body = (uint32_t(e) << 23) | uint32_t(mant >> 29);
  const uint32_t rem = uint32_t(mant & 0x1fffffffu);
  if (rem > 0x10000000u || (rem == 0x10000000u && (body & 1u))) ++body;  // carries into the exponent
  return __uint_as_float((uint32_t(u >> 63) << 31) | body);
}

// FP64 -> FP32 round to nearest even on the 32-bit words of x, branch-free, for
// a result that is zero or an FP32 normal number; `odd` is set for inputs
// outside that range (the tile's geometry is then recomputed with the general
// conversions). A rounding at the top of the range that carries into infinity
// comes out exact without the flag.
__device__ __forceinline__ float d2f_fast(double x, bool& odd) {
  const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
  const uint32_t ahi = hi & 0x7fffffffu;
  const int e = int(ahi >> 20) - 896;
  const bool zero = (ahi | lo) == 0;
  odd |= (e <= 0 || e >= 255) && !zero;
  uint32_t body = (uint32_t(e) << 23) | ((ahi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t rem = lo & 0x1fffffffu;
  body += (rem > 0x10000000u || (rem == 0x10000000u && (body & 1u))) ? 1u : 0u;
  return __uint_as_float((hi & 0x80000000u) | (zero ? 0u : body));
}

// x - d2f_fast(x), the part of x below its FP32 rounding, itself rounded to
// FP32, on the 32-bit words: the low 29 mantissa bits minus the rounding
// carry, times 2^(exponent - 1075), normalised on the integer bits. For x with
// an FP32-normal rounding; `odd` is set where the result leaves the FP32
// normal range (the tile is then recomputed with the general conversions).
__device__ __forceinline__ float d2f_rest(double x, bool& odd) {
  const uint32_t hi = uint32_t(__double2hiint(x)), lo = uint32_t(__double2loint(x));
  const int E = int((hi & 0x7fffffffu) >> 20);
  const uint32_t rem = lo & 0x1fffffffu;
  const uint32_t body = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const bool up = rem > 0x10000000u || (rem == 0x10000000u && (body & 1u));
  // r = rem - up 2^29, |r| <= 2^28; the value is r 2^(E - 1075), sign of x, negated if up
  const uint32_t m = up ? (0x20000000u - rem) : rem;
  const int lz = __clz(m | 1u);            // >= 3
  const int sh = lz - 8;                   // normalise the leading 1 to bit 23
  const int rs = sh < 0 ? -sh : 1;         // 25..29 significant bits: round to nearest even
  const uint32_t t = m >> rs, rb = m & ((1u << rs) - 1u), half = 1u << (rs - 1);
  const uint32_t rnd = t + ((rb > half || (rb == half && (t & 1u))) ? 1u : 0u);
  const bool carry = sh < 0 && (rnd >> 24) != 0;
  const uint32_t mm = sh >= 0 ? (m << sh) : (carry ? rnd >> 1 : rnd);
  const int er = E - 948 + (31 - lz) + (carry ? 1 : 0);  // biased exponent of m 2^(E - 1075)
  odd |= m != 0 && (er <= 0 || er >= 255);
  const uint32_t sgn = (hi & 0x80000000u) ^ (up ? 0x80000000u : 0u);
  return __uint_as_float(m == 0 ? 0u : (sgn | (uint32_t(er) << 23) | (mm & 0x7fffffu)));
}

// TF32 rounding of x (to nearest, ties away from zero), the hi part of the
// 3xTF32 split; the lo part is to_tf32(x - hi).
__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Exact sum of N FP32 terms held in registers, rounded once to FP64 (the
// fixed-point accumulation of fx_sum), on the integer bits.
template <int N>
__device__ __forceinline__ double fx_sum_regs_f32(const float (&v)[N]) {
  using Tr = FxTraits<float>;
  int emax = 1;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(v[t], m, ex, ng);
    if (m != 0 && ex > emax) emax = ex;
  }
  int64_t S = 0;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    uint64_t m;
    int ex;
    bool ng;
    Tr::split(v[t], m, ex, ng);
    const int sh = Tr::kShift0 - (emax - ex);
    const uint64_t a = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> (-sh)) : 0ull);
    S += ng ? -int64_t(a) : int64_t(a);
  }
  return fx_to_double(S, emax - Tr::kScale);
}

// Shared-memory layout of the FP32/BF16 cell block (byte offsets; host and
// device agree on it through this one function). Regions: vertex coordinates
// [cpb][24] and trilinear coefficients [cpb][21] (FP64), the Jacobian columns
// [cpb][3][n1d^2][3] (FP64), the products u v of the 1D points [n1d^2] (FP64),
// w det J as hi + lo [cpb][nq] (float2), FP32 cofactors and w/det J
// [cpb][nq][12], then the operands: for nb <= 27 the scaled and plain
// cofactor gradients as float4 [cpb][nq][nb] each, else the plain gradients
// [cpb][nq][3][nb] (float).
struct MixedLayout {
  long x, a, jc, uv, djw, geo32, ga, gb, bytes;
};
__host__ __device__ inline MixedLayout mixed_layout(int cpb, int nq, int n1d, int nb) {
  MixedLayout L;
  const long p2 = long(n1d) * n1d;
  L.x = 0;
  L.a = L.x + long(cpb) * 24 * 8;
  L.jc = L.a + long(cpb) * 21 * 8;
  L.uv = L.jc + long(cpb) * 9 * p2 * 8;
  L.djw = (L.uv + p2 * 8 + 15) & ~15l;
  L.geo32 = (L.djw + long(cpb) * nq * 8 + 15) & ~15l;
  L.ga = L.geo32 + long(cpb) * nq * 48;
  if (nb <= 27) {
    L.gb = L.ga + long(cpb) * nq * nb * 16;
    L.bytes = L.gb + long(cpb) * nq * nb * 16;
  } else {
    L.gb = L.ga;
    L.bytes = L.ga + long(cpb) * nq * 3 * nb * 4;
  }
  return L;
}

// Threads and cells of a k_cell block in the FP32 and BF16 forms with the
// (p+1)^3 rule (0: 256 threads and cells_per_block). Small blocks overlap each
// other's phases: Poisson Q1 64^3 0.297 -> 0.278 ms, Q2 32^3 0.470 -> 0.438 (FP32)
// and 0.414 -> 0.391 (BF16); Q3 has one tile per thread.
template <int P, int NC, int PREC>
struct WideShape {
  static constexpr int THREADS = NC == 1 ? (P == 2 && PREC == 1 ? 192 : 128) : 0;
  static constexpr int CELLS = NC == 1 ? (P == 1 ? 8 : P == 2 && PREC == 1 ? 2 : 1) : 0;
};

// One block integrates `cpb` cells for the FP32 (PREC 1) and BF16 (PREC 2)
// forms; same steps as cell_block_fp64, with the geometry FP64 and everything
// after it FP32:
//   * each Jacobian column of the trilinear map depends on two of the three
//     reference coordinates only (column d is linear in the other two and
//     bilinear in their product), so it is evaluated once per pair of 1D
//     points of the tensor rule, n1d^2 instead of n1d^3 times (FP64);
//   * per quadrature point: cofactors and det J (FP64), rounded once to FP32
//     on the integer bits; w/det J as the FP32 quotient of the rounded values;
//     w det J as an FP32 hi + lo pair;
//   * gradients gh_a = cof gradhat(phihat_a) in FP32, stored as (w/det) gh_a
//     and gh_a (rounded to BF16 for PREC 2), so that a product of one point
//     costs one load per side;
//   * PREC 1 sums the points in blocks of `qblock` (one z-slab of the rule)
//     with Kahan compensation between blocks; PREC 2 sums plainly;
//   * the cell vector sum_q (w det J)_q phihat_a(x_q) in double-float
//     arithmetic (products with fmaf error terms, TwoSum accumulation),
//     rounded once to FP64.
template <int P, int NC, int PREC, bool WIDE>
__device__ __forceinline__ void cell_block_mixed(const CellParams& prm, int64_t e0, int ncell, double* smem) {
  constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  constexpr int NL = NC * NB;
  constexpr int NLP = (NL + 3) & ~3;
  constexpr bool VEC = NB <= 27;
  const int cpb = prm.cpb, nq = prm.nq, n1d = prm.nq1d, p2 = n1d * n1d;
  // Q3 Poisson with the 4^3 rule: operands and contraction slab by slab (below)
  constexpr bool Q3P = NC == 1 && NB == 64;
  const bool slabs = Q3P && n1d == P + 1;
  const MixedLayout L = mixed_layout(cpb, nq, n1d, NB);
  unsigned char* base = reinterpret_cast<unsigned char*>(smem);
  double* sx = reinterpret_cast<double*>(base + L.x);
  double* sa = reinterpret_cast<double*>(base + L.a);
  double* sj = reinterpret_cast<double*>(base + L.jc);
  double* suv = reinterpret_cast<double*>(base + L.uv);
  float2* djw = reinterpret_cast<float2*>(base + L.djw);
  float* geo32 = reinterpret_cast<float*>(base + L.geo32);
  float4* gA = reinterpret_cast<float4*>(base + L.ga);
  float4* gB = reinterpret_cast<float4*>(base + L.gb);
  float* g = reinterpret_cast<float*>(base + L.ga);
  const int tid = threadIdx.x;

  for (int i = tid; i < ncell * 24; i += blockDim.x) sx[i] = prm.xv[e0 * 24 + i];
  __syncthreads();
  // trilinear coefficients; u v of the 1D point pairs (the 1D rule is the x
  // coordinates of the first n1d points)
  for (int i = tid; i < ncell * 3 + p2; i += blockDim.x) {
    if (i < ncell * 3) {
      trilinear_coefficients(sx + (i / 3) * 24, i % 3, sa + (i / 3) * 21);
    } else {
      const int pr = i - ncell * 3;
      suv[pr] = prm.xq[3 * (pr % n1d)] * prm.xq[3 * (pr / n1d)];
    }
  }
  __syncthreads();
  // Jacobian columns: J[k][d] at the pair (u, v) of the other two coordinates
  // (in axis order): d = 0: a1 + a4 y + a5 z + a7 yz; d = 1: a2 + a4 x + a6 z +
  // a7 xz; d = 2: a3 + a5 x + a6 y + a7 xy (coefficients a1..a7 at offsets
  // 0, 3, .., 18 of the component).
  for (int i = tid; i < ncell * 9 * p2; i += blockDim.x) {
    const int c = i / (9 * p2), r = i % (9 * p2), d = r / (3 * p2), rem = r % (3 * p2), pr = rem / 3, k = rem % 3;
    const double* a = sa + c * 21;
    const double u = prm.xq[3 * (pr % n1d)], v = prm.xq[3 * (pr / n1d)];
    const int o0 = 3 * d, ou = d == 2 ? 12 : 9, ov = d == 0 ? 12 : 15;
    sj[i] = fma(a[18 + k], suv[pr], fma(a[ov + k], v, fma(a[ou + k], u, a[o0 + k])));
  }
  __syncthreads();
  for (int i = tid; i < ncell * nq; i += blockDim.x) {
    const int c = i / nq, q = i % nq;
    const int ix = q % n1d, iy = (q / n1d) % n1d, iz = q / p2;
    const double* jc = sj + c * 9 * p2;
    double J[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      J[k][0] = jc[(0 * p2 + iy + n1d * iz) * 3 + k];
      J[k][1] = jc[(1 * p2 + ix + n1d * iz) * 3 + k];
      J[k][2] = jc[(2 * p2 + ix + n1d * iy) * 3 + k];
    }
    double cof[9];
    cof[0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    cof[1] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    cof[2] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    cof[3] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    cof[4] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    cof[5] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    cof[6] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    cof[7] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    cof[8] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double det = J[0][0] * cof[0] + J[0][1] * cof[1] + J[0][2] * cof[2];
    if (!(det > 0.0)) atomicOr(prm.err, kErrNegJacobian);
    const double wq = prm.w[q];
    float* g32 = geo32 + size_t(i) * 12;
#pragma unroll
    for (int t = 0; t < 9; ++t) g32[t] = d2f_rn(cof[t]);
    g32[9] = d2f_rn(wq) / d2f_rn(det);
    const double wd = wq * det;
    const float hi = d2f_rn(wd);
    djw[i] = make_float2(hi, d2f_rn(wd - f32_to_f64_exact(hi)));
  }
  __syncthreads();
  for (int i = tid; i < (slabs ? 0 : ncell * nq * NB); i += blockDim.x) {
    const int a = i % NB, cq = i / NB, q = cq % nq;
    const float4* gq4 = reinterpret_cast<const float4*>(geo32 + size_t(cq) * 12);
    const float4 c0 = gq4[0], c1 = gq4[1], c2 = gq4[2];
    const float* dp = prm.dphi32 + (size_t(q) * NB + a) * 3;
    const float d0 = dp[0], d1 = dp[1], d2 = dp[2];
    float g0 = fmaf(c0.z, d2, fmaf(c0.y, d1, c0.x * d0));
    float g1 = fmaf(c1.y, d2, fmaf(c1.x, d1, c0.w * d0));
    float g2 = fmaf(c2.x, d2, fmaf(c1.w, d1, c1.z * d0));
    if (VEC) {
      const float s = c2.y;
      float a0 = s * g0, a1 = s * g1, a2 = s * g2;
      if (PREC == 2) {
        round_bf16_pair(a0, a1);
        round_bf16_pair(a2, g0);
        round_bf16_pair(g1, g2);
      }
      gA[i] = make_float4(a0, a1, a2, 0.f);
      gB[i] = make_float4(g0, g1, g2, 0.f);
    } else {
      float* gg = g + size_t(cq) * 3 * NB;
      gg[a] = g0;
      gg[NB + a] = g1;
      gg[2 * NB + a] = g2;
    }
  }
  __syncthreads();
  const int qb = PREC == 1 ? prm.qblock : nq;
  if constexpr (Q3P) {
    // Per slab of 16 points (the Kahan block): every thread forms gradients,
    // plain and times w/det, [q][component][node]; then each thread adds the
    // slab's products to its TA x 4 tile of node pairs, (TA + 4) / 4 16-byte
    // loads per 4 TA multiply-adds. The same operations in the same order per
    // entry as one pair per thread. The operands of a whole cell at once (48 KB)
    // with a 4 x 2 tile, 18 loads and 12 products w/det gh per 24 multiply-adds,
    // were bound by those: 24^3 cells 0.975 -> 0.638 ms, now bound by issue (66 %,
    // 60 % of the instructions multiply-adds).
    if (slabs) {
      constexpr int TA = WIDE ? 8 : 4, QS = (P + 1) * (P + 1);
      float* ga = g;
      float* gb = g + QS * 3 * NB;
      const int ta = tid / (NB / 4), tb = tid % (NB / 4);
      const bool has = ta < NB / TA;
      float sum[TA][4], carry[TA][4], part[TA][4];
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) sum[u][v] = carry[u][v] = part[u][v] = 0.f;
      for (int q0 = 0; q0 < nq; q0 += QS) {
        if (q0) __syncthreads();
        for (int i = tid; i < QS * NB / 4; i += blockDim.x) {  // four nodes per thread
          const int a = (i % (NB / 4)) * 4, ql = i / (NB / 4), q = q0 + ql;
          const float4* gq4 = reinterpret_cast<const float4*>(geo32 + q * 12);
          const float4 c0 = gq4[0], c1 = gq4[1], c2 = gq4[2];
          const float4* dp = reinterpret_cast<const float4*>(prm.dphi32 + (q * NB + a) * 3);
          const float4 e0v = __ldg(dp), e1v = __ldg(dp + 1), e2v = __ldg(dp + 2);
          const float d[12] = {e0v.x, e0v.y, e0v.z, e0v.w, e1v.x, e1v.y, e1v.z, e1v.w, e2v.x, e2v.y, e2v.z, e2v.w};
          float gk[3][4], sk[3][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float d0 = d[3 * u], d1 = d[3 * u + 1], d2 = d[3 * u + 2];
            gk[0][u] = fmaf(c0.z, d2, fmaf(c0.y, d1, c0.x * d0));
            gk[1][u] = fmaf(c1.y, d2, fmaf(c1.x, d1, c0.w * d0));
            gk[2][u] = fmaf(c2.x, d2, fmaf(c1.w, d1, c1.z * d0));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              sk[k][u] = c2.y * gk[k][u];
              if (PREC == 2) round_bf16_pair(sk[k][u], gk[k][u]);
            }
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            *reinterpret_cast<float4*>(ga + (ql * 3 + k) * NB + a) = make_float4(sk[k][0], sk[k][1], sk[k][2], sk[k][3]);
            *reinterpret_cast<float4*>(gb + (ql * 3 + k) * NB + a) = make_float4(gk[k][0], gk[k][1], gk[k][2], gk[k][3]);
          }
        }
        __syncthreads();
        if (has) {
          if (PREC == 1) {
#pragma unroll
            for (int u = 0; u < TA; ++u)
#pragma unroll
              for (int v = 0; v < 4; ++v) part[u][v] = 0.f;
          }
#pragma unroll 4
          for (int r = 0; r < QS * 3; ++r) {
            float x[TA], y[4];
#pragma unroll
            for (int u = 0; u < TA; u += 4) {
              const float4 A = *reinterpret_cast<const float4*>(ga + r * NB + ta * TA + u);
              x[u] = A.x, x[u + 1] = A.y, x[u + 2] = A.z, x[u + 3] = A.w;
            }
            const float4 Bv = *reinterpret_cast<const float4*>(gb + r * NB + tb * 4);
            y[0] = Bv.x, y[1] = Bv.y, y[2] = Bv.z, y[3] = Bv.w;
#pragma unroll
            for (int u = 0; u < TA; ++u)
#pragma unroll
              for (int v = 0; v < 4; ++v) part[u][v] = fmaf(x[u], y[v], part[u][v]);
          }
          if (PREC == 1) {
#pragma unroll
            for (int u = 0; u < TA; ++u)
#pragma unroll
              for (int v = 0; v < 4; ++v) kahan_add(sum[u][v], carry[u][v], part[u][v]);
          }
        }
      }
      if (has && ncell > 0) {
        const float coef = d2f_rn(prm.coef[e0]);
        float* K = reinterpret_cast<float*>(prm.ke) + e0 * NL * NLP;
#pragma unroll
        for (int u = 0; u < TA; ++u) {
          float r[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) r[v] = coef * (PREC == 1 ? sum[u][v] : part[u][v]);
          *reinterpret_cast<float4*>(K + (ta * TA + u) * NLP + tb * 4) = make_float4(r[0], r[1], r[2], r[3]);
        }
      }
    }
  }
  if constexpr (NC == 1) {
    // Poisson: each thread sums a TA x TB tile of node pairs, so that one
    // point's loads (TA + TB gradients, w/det) serve TA TB products per
    // component; per pair the same slab-blocked (Kahan) sum as one pair per
    // thread.
    constexpr int TA = NB == 64 ? 4 : NB == 27 ? 3 : 2, TB = NB == 64 ? 2 : TA;  // 4 x 2 for Q3: fewer registers
    constexpr int NTA = NB / TA, NTB = NB / TB;
    static_assert(NB % TA == 0 && NB % TB == 0, "tile");
    for (int i = tid; i < (slabs ? 0 : ncell * NTA * NTB); i += blockDim.x) {
      const int c = i / (NTA * NTB), tt = i % (NTA * NTB), a0 = (tt / NTB) * TA, b0 = (tt % NTB) * TB;
      const int64_t e = e0 + c;
      const float coef = d2f_rn(prm.coef[e]);
      float sum[TA][TB], carry[TA][TB];
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int v = 0; v < TB; ++v) sum[u][v] = carry[u][v] = 0.f;
      for (int q0 = 0; q0 < nq; q0 += qb) {
        float part[TA][TB];
#pragma unroll
        for (int u = 0; u < TA; ++u)
#pragma unroll
          for (int v = 0; v < TB; ++v) part[u][v] = 0.f;
        const int q1 = q0 + qb < nq ? q0 + qb : nq;
        for (int q = q0; q < q1; ++q) {
          float ga[3][TA], gb[3][TB];
          if (VEC) {
#pragma unroll
            for (int u = 0; u < TA; ++u) {
              const float4 A = gA[(size_t(c) * nq + q) * NB + a0 + u];
              ga[0][u] = A.x, ga[1][u] = A.y, ga[2][u] = A.z;
            }
#pragma unroll
            for (int v = 0; v < TB; ++v) {
              const float4 B = gB[(size_t(c) * nq + q) * NB + b0 + v];
              gb[0][v] = B.x, gb[1][v] = B.y, gb[2][v] = B.z;
            }
          } else {
            const float* gq = g + (size_t(c) * nq + q) * 3 * NB;
            const float sq = geo32[(size_t(c) * nq + q) * 12 + 9];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
#pragma unroll
              for (int u = 0; u < TA; ++u) {
                ga[k][u] = sq * gq[k * NB + a0 + u];
                if (PREC == 2) ga[k][u] = round_bf16(ga[k][u]);
              }
#pragma unroll
              for (int v = 0; v < TB; ++v) {
                gb[k][v] = gq[k * NB + b0 + v];
                if (PREC == 2) gb[k][v] = round_bf16(gb[k][v]);
              }
            }
          }
#pragma unroll
          for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int u = 0; u < TA; ++u)
#pragma unroll
              for (int v = 0; v < TB; ++v) part[u][v] = fmaf(ga[k][u], gb[k][v], part[u][v]);
        }
#pragma unroll
        for (int u = 0; u < TA; ++u)
#pragma unroll
          for (int v = 0; v < TB; ++v) {
            if (PREC == 1) kahan_add(sum[u][v], carry[u][v], part[u][v]); else sum[u][v] += part[u][v];
          }
      }
      float* K = reinterpret_cast<float*>(prm.ke) + e * NL * NLP;
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int v = 0; v < TB; ++v) K[(a0 + u) * NLP + b0 + v] = coef * sum[u][v];
    }
  }
  if constexpr (NC == 3) {
    // Nine Gram sums per node pair. Q3 takes two node pairs (a0, b), (a0 + 1, b)
    // per thread, which share the loads of b and w/det; per entry the same
    // operations in the same order. 12^3 Q3 cells: 0.471 -> 0.417 ms (a 2 x 2 tile
    // in 154 registers: 0.416, unrolled over the points 0.434).
    constexpr int TU = VEC ? 1 : 2;
    constexpr int MA = NB / TU;
    for (int i = tid; i < ncell * MA * NB; i += blockDim.x) {
      const int c = i / (MA * NB), ab = i % (MA * NB), a0 = (ab / NB) * TU, b = ab % NB;
      const int64_t e = e0 + c;
      const float coef = d2f_rn(prm.coef[e]);
      float* K = reinterpret_cast<float*>(prm.ke) + e * NL * NLP;
      float S[TU][3][3], C[TU][3][3];
#pragma unroll
      for (int u = 0; u < TU; ++u)
#pragma unroll
        for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
          for (int j2 = 0; j2 < 3; ++j2) S[u][i2][j2] = C[u][i2][j2] = 0.f;
      for (int q0 = 0; q0 < nq; q0 += qb) {
        float G[TU][3][3];
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
          for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
            for (int j2 = 0; j2 < 3; ++j2) G[u][i2][j2] = 0.f;
        const int q1 = q0 + qb < nq ? q0 + qb : nq;
        for (int q = q0; q < q1; ++q) {
          float ga[TU][3], gb[3];
          if constexpr (VEC) {
            const float4 A = gA[(size_t(c) * nq + q) * NB + a0], B = gB[(size_t(c) * nq + q) * NB + b];
            ga[0][0] = A.x, ga[0][1] = A.y, ga[0][2] = A.z;
            gb[0] = B.x, gb[1] = B.y, gb[2] = B.z;
          } else {
            const float* gq = g + (size_t(c) * nq + q) * 3 * NB;
            const float sc = geo32[(size_t(c) * nq + q) * 12 + 9];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const float2 A = *reinterpret_cast<const float2*>(gq + k * NB + a0);
              ga[0][k] = sc * A.x;
              ga[TU - 1][k] = sc * A.y;
              gb[k] = gq[k * NB + b];
              if (PREC == 2) {
#pragma unroll
                for (int u = 0; u < TU; ++u) ga[u][k] = round_bf16(ga[u][k]);
                gb[k] = round_bf16(gb[k]);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < TU; ++u)
#pragma unroll
            for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
              for (int j2 = 0; j2 < 3; ++j2) G[u][i2][j2] = fmaf(ga[u][i2], gb[j2], G[u][i2][j2]);
        }
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
          for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
            for (int j2 = 0; j2 < 3; ++j2) {
              if (PREC == 1) kahan_add(S[u][i2][j2], C[u][i2][j2], G[u][i2][j2]); else S[u][i2][j2] += G[u][i2][j2];
            }
      }
      const float lh = d2f_rn(prm.lam_hat), mh = d2f_rn(prm.mu_hat);
#pragma unroll
      for (int u = 0; u < TU; ++u) {
        const float tr = S[u][0][0] + S[u][1][1] + S[u][2][2];
#pragma unroll
        for (int i2 = 0; i2 < 3; ++i2)
#pragma unroll
          for (int j2 = 0; j2 < 3; ++j2) {
            float v = lh * S[u][i2][j2] + mh * S[u][j2][i2];
            if (i2 == j2) v += mh * tr;
            K[size_t(i2 * NB + a0 + u) * NLP + j2 * NB + b] = coef * v;
          }
      }
    }
  }
  for (int i = tid; i < ncell * NB; i += blockDim.x) {
    const int c = i / NB, a = i % NB;
    float sh = 0.f, sl = 0.f;
    for (int q = 0; q < nq; ++q) {
      const float2 w2 = djw[c * nq + q], p2v = prm.phi2[size_t(q) * NB + a];
      const float ph = w2.x * p2v.x;
      const float pe = fmaf(w2.x, p2v.x, -ph) + (w2.x * p2v.y + w2.y * p2v.x);
      const float sum = sh + ph;
      const float bp = sum - sh;
      const float err = (sh - (sum - bp)) + (ph - bp);
      sh = sum;
      sl += err + pe;
    }
    const double f = sl == 0.f ? f32_to_f64_exact(sh) : __dadd_rn(f32_to_f64_exact(sh), f32_to_f64_exact(sl));
    double* fe = prm.fe + (e0 + c) * NL;
#pragma unroll
    for (int k = 0; k < NC; ++k) fe[k * NB + a] = prm.f[k] * f;
  }
}

// Cell integration of one block of cells in the given precision.
// WIDE: a k_cell block (threads of WideShape), not one of the batched kernel (256 threads).
template <int P, int NC, int PREC, bool WIDE = false>
__device__ __forceinline__ void cell_block(const CellParams& prm, int64_t e0, int ncell, double* smem) {
  if constexpr (PREC == 0) {
    cell_block_fp64<P, NC>(prm, e0, ncell, smem);
  } else {
    cell_block_mixed<P, NC, PREC, WIDE>(prm, e0, ncell, smem);
  }
}

// How a scatter reads the cell matrices, which depends on when they are written:
// kBefore, by a kernel that ended before this launch began: the non-coherent
// read-only path (ld.global.nc asks for data that nobody writes while the
// reading grid exists); kOverlap, by a kernel that this launch overlaps and
// waits for (griddepcontrol.wait): ordinary loads, which neither the compiler nor
// the hardware may move before the wait; kSameLaunch, by other blocks of this
// launch (the batched driver): bypassing L1 (ld.global.cg).
enum class KeWritten { kBefore, kOverlap, kSameLaunch };
template <KeWritten W, typename T>
__device__ __forceinline__ T ld_ke(const T* p) {
  if constexpr (W == KeWritten::kSameLaunch) return __ldcg(p);
  else if constexpr (W == KeWritten::kOverlap) return *p;
  else return __ldg(p);
}

// One batch of the slot-wise double-float scatter of k_scatter_slots (see
// there): B slots from s_begin, R rows per item (R = 3: the rows of one node,
// local rows i * NL / R + a of each cell), accumulator rows of stride rs with
// a private dummy per lane at index `dummy`. The first contribution of a
// nonzero (flag bit 15 of pos; every entry of slot 0) stores (v, 0); later
// ones add with TwoSum.
template <int NL, int R, KeWritten W = KeWritten::kBefore>
struct SlotScatter {
  static constexpr KeWritten kWritten = W;
  static constexpr int CH = (NL + 31) / 32;
  static constexpr int NBR = NL / R;  // local-row offset between the rows of one node
  static constexpr int LOADS = CH * (R + 1);
  // slots per batch: 4 where the loads of a batch fit the registers (measured on
  // the Q1 node rows: 4 slots per batch at five blocks per SM beat 8 at four)
  static constexpr int SB = LOADS <= 8 ? 4 : LOADS <= 16 ? 2 : 1;

  // One batch of B slots starting at slot s_begin.
  template <int B, bool IDX32>
  __device__ __forceinline__ static void batch(const ScatterParams& p, const float* ke, const uint16_t* pos,
                                               int my_slot, int s_begin, float2* acc, int rs, int dummy, int lane) {
    float x[B][CH][R];
    int kk[B][CH];
#pragma unroll
    for (int t = 0; t < B; ++t) {
      const int s = s_begin + t;
      const int sid = __shfl_sync(kFull, my_slot, s);
      const float* krow = IDX32 ? ke + uint32_t(sid) * uint32_t(p.nlp) : ke + int64_t(sid) * p.nlp;
      const uint16_t* prow = pos + s * NL;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int k = int(W == KeWritten::kSameLaunch ? __ldcg(prow + c * 32) : __ldg(prow + c * 32));
        kk[t][c] = (c < CH - 1 || c * 32 + lane < NL) ? k : dummy;
#pragma unroll
        for (int i = 0; i < R; ++i) x[t][c][i] = ld_ke<W>(krow + i * NBR * p.nlp + c * 32);
      }
    }
#pragma unroll
    for (int t = 0; t < B; ++t) {
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int raw = kk[t][c];
        const int k = raw & 0x7fff;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          float2* ai = acc + i * rs;
          const float v = (c < CH - 1 || c * 32 + lane < NL) ? x[t][c][i] : 0.f;
          if (s_begin + t == 0) {
            ai[k] = make_float2(v, 0.f);
          } else {
            const float2 a = (raw & 0x8000) ? make_float2(0.f, 0.f) : ai[k];
            const float sum = a.x + v;
            const float bp = sum - a.x;
            const float err = (a.x - (sum - bp)) + (v - bp);
            ai[k] = make_float2(sum, a.y + err);
          }
        }
      }
      __syncwarp();
    }
  }
};


}  // namespace feasm
