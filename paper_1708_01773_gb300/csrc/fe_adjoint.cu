// The compliance adjoint of libfeasm (sm_103a).
#include <type_traits>

#include "fe_device.cuh"

namespace feasm {

// ---------------------------------------------------------------------------
// Compliance adjoint: one thread per cell. For fixed u the sensitivity of
// c = u^T A u to the cell coefficient is the cell energy of u per unit
// coefficient, evaluated per quadrature point from grad u (Eq. fematrix,
// Eq. shape_grad) without forming A^K:
//   Poisson    |grad u|^2,
//   elasticity lam^ (div u)^2 + 2 mu^ eps(u):eps(u),
// times w_q det J_q. T is the arithmetic of the strain (FP64 or FP32); the
// geometry and the sums over points are FP64.
struct AdjParams {
  int64_t n_cells;
  int nq;
  const double* xv;
  const double* w;
  const double* xq;
  const double* dphi;
  const float* dphi32;
  const int32_t* cell_dofs;
  const double* u;
  const double* coef;
  double grad_scale, lam_hat, mu_hat;
  double* g;
  double* partials;
  int* err;
};

constexpr int kAdjThreads = kAdjointBlock;

// FP32 strain energy density from the reference gradient and cof / det.
template <int NC>
__device__ __forceinline__ float strain_density(const float (&gr)[NC][3], const float (&cs)[9], float lh, float mh2) {
          float gu[NC][3];
  #pragma unroll
          for (int c = 0; c < NC; ++c)
  #pragma unroll
            for (int k = 0; k < 3; ++k) gu[c][k] = gr[c][0] * cs[3 * k] + gr[c][1] * cs[3 * k + 1] + gr[c][2] * cs[3 * k + 2];
          float dens;
          if (NC == 1) {
            dens = gu[0][0] * gu[0][0] + gu[0][1] * gu[0][1] + gu[0][2] * gu[0][2];
          } else {
            const float div = gu[0][0] + gu[1 % NC][1] + gu[2 % NC][2];
            float ee = 0.f;
  #pragma unroll
            for (int k = 0; k < 3; ++k)
  #pragma unroll
              for (int l = 0; l < 3; ++l) {
                const float eps = 0.5f * (gu[k % NC][l] + gu[l % NC][k]);
                ee += eps * eps;
              }
            dens = lh * (div * div) + mh2 * ee;
          }
  return dens;
}

// The block's share of the compliance, in a fixed order.
__device__ __forceinline__ void adjoint_partial(const AdjParams& p, int64_t e, double energy, double* red) {
  if (p.partials == nullptr) return;
  red[threadIdx.x] = (e < p.n_cells) ? p.coef[e] * energy : 0.0;
  __syncthreads();
  for (int off = kAdjThreads / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) p.partials[blockIdx.x] = red[0];
}

// Energy of one cell in the FP64 form (a: trilinear coefficients of the geometry, ue: u at the cell's DOFs).
template <int P, int NC>
__device__ __forceinline__ double cell_energy_fp64(const AdjParams& p, const double (&a)[21],
                                                   const double (&ue)[NC * (P + 1) * (P + 1) * (P + 1)]) {
  constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  double energy = 0.0;
  for (int q = 0; q < p.nq; ++q) {
    double cof[9], det;
    geometry_at(a, p.xq[3 * q], p.xq[3 * q + 1], p.xq[3 * q + 2], cof, &det);
    if (!(det > 0.0)) atomicOr(p.err, kErrNegJacobian);
    // reference gradient of each component of u
    double gr[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c) gr[c][0] = gr[c][1] = gr[c][2] = 0.0;
    const double* dq = p.dphi + size_t(q) * NB * 3;
#pragma unroll 4
    for (int b = 0; b < NB; ++b) {
      const double d0 = dq[3 * b], d1 = dq[3 * b + 1], d2 = dq[3 * b + 2];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const double uc = ue[c * NB + b];
        gr[c][0] += uc * d0;
        gr[c][1] += uc * d1;
        gr[c][2] += uc * d2;
      }
    }
    // physical gradient: (grad u)_{c,k} = sum_d gr[c][d] cof[k][d] / det
    const double inv = 1.0 / det;
    double cs[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) cs[t] = cof[t] * inv;
    double gu[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int k = 0; k < 3; ++k) gu[c][k] = gr[c][0] * cs[3 * k] + gr[c][1] * cs[3 * k + 1] + gr[c][2] * cs[3 * k + 2];
    double dens;
    if (NC == 1) {
      dens = gu[0][0] * gu[0][0] + gu[0][1] * gu[0][1] + gu[0][2] * gu[0][2];
    } else {
      const double div = gu[0][0] + gu[1 % NC][1] + gu[2 % NC][2];
      double ee = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          const double eps = 0.5 * (gu[k % NC][l] + gu[l % NC][k]);
          ee += eps * eps;
        }
      dens = p.lam_hat * (div * div) + 2.0 * p.mu_hat * ee;
    }
    energy += p.w[q] * det * dens;
  }
  return energy;
}

template <int P, int NC, typename T>
__global__ void __launch_bounds__(kAdjThreads) k_adjoint(AdjParams p) {
  constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  constexpr int NL = NC * NB;
  __shared__ double red[kAdjThreads];
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  double energy = 0.0;
  if (e < p.n_cells) {
    double x[24], a[21];
#pragma unroll
    for (int i = 0; i < 24; ++i) x[i] = p.xv[e * 24 + i];
#pragma unroll
    for (int k = 0; k < 3; ++k) trilinear_coefficients(x, k, a);
    if constexpr (std::is_same<T, float>::value) {
      // FP32 strain, FP64 geometry and sums: the conversions run on the
      // integer bits, w/det J and the physical gradients in FP32, one FP64
      // multiply-add per point accumulates w det J times the energy density
      // (GB300's FP64 pipe is the limit of this kernel).
      float ue[NL];
#pragma unroll
      for (int l = 0; l < NL; ++l) ue[l] = d2f_rn(p.u[p.cell_dofs[e * NL + l]]);
      const float lh = d2f_rn(p.lam_hat), mh2 = 2.f * d2f_rn(p.mu_hat);
      for (int q = 0; q < p.nq; ++q) {
        double cof[9], det;
        geometry_at(a, p.xq[3 * q], p.xq[3 * q + 1], p.xq[3 * q + 2], cof, &det);
        if (!(det > 0.0)) atomicOr(p.err, kErrNegJacobian);
        float gr[NC][3];
#pragma unroll
        for (int c = 0; c < NC; ++c) gr[c][0] = gr[c][1] = gr[c][2] = 0.f;
        const float* dq = p.dphi32 + size_t(q) * NB * 3;
#pragma unroll 4
        for (int b = 0; b < NB; ++b) {
          const float d0 = dq[3 * b], d1 = dq[3 * b + 1], d2 = dq[3 * b + 2];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const float uc = ue[c * NB + b];
            gr[c][0] = fmaf(uc, d0, gr[c][0]);
            gr[c][1] = fmaf(uc, d1, gr[c][1]);
            gr[c][2] = fmaf(uc, d2, gr[c][2]);
          }
        }
        const float rdet = 1.f / d2f_rn(det);
        float cs[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) cs[t] = d2f_rn(cof[t]) * rdet;
        energy = fma(p.w[q] * det, f32_to_f64_exact(strain_density<NC>(gr, cs, lh, mh2)), energy);
      }
      p.g[e] = p.grad_scale * energy;
    } else {
    T ue[NL];
#pragma unroll
    for (int l = 0; l < NL; ++l) ue[l] = T(p.u[p.cell_dofs[e * NL + l]]);
    energy = cell_energy_fp64<P, NC>(p, a, ue);
    p.g[e] = p.grad_scale * energy;
    }
  }
  adjoint_partial(p, e, energy, red);
}

// Sums the per-block partials in a fixed order (one block).
__global__ void k_sum_partials(const double* partials, int n, double* out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += partials[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// 2^-k with |x| 2^-k in [1, 2) for the largest |x| of n values (1 where that is
// zero or not finite), k added to `sum` `times` times; exact.
__device__ __forceinline__ void scale_to_one(double* x, int n, int times, int* sum) {
  double m = 0.0;
  for (int i = 0; i < n; ++i) m = fmax(m, fabs(x[i]));
  const int k = m > 0.0 && m < INFINITY ? ilogb(m) : 0;
  for (int i = 0; i < n; ++i) x[i] = scalbn(x[i], -k);
  *sum += times * k;
}

// The same, out of line, for a cell that k_adjoint_q1 does not take (x: its
// vertices, dofs: its DOFs): u and the geometry scaled by powers of two, so that
// only the result may leave the range. (The parameters one by one: a reference to
// the kernel's would keep them in memory, 5 % of the FP32 form's time.)
template <int NC>
static __device__ __noinline__ double cell_energy_scaled(const double* x, const double* u, const int32_t* dofs,
                                                         const double* xq, const double* w, const double* dphi,
                                                         double lam_hat, double mu_hat, int* err) {
  AdjParams p;
  p.nq = 8;
  p.xq = xq;
  p.w = w;
  p.dphi = dphi;
  p.lam_hat = lam_hat;
  p.mu_hat = mu_hat;
  p.err = err;
  double a[21], ue[NC * 8];
#pragma unroll
  for (int k = 0; k < 3; ++k) trilinear_coefficients(x, k, a);
  for (int l = 0; l < NC * 8; ++l) ue[l] = u[dofs[l]];
  int k = 0;
  scale_to_one(a, 21, 1, &k);
  scale_to_one(ue, NC * 8, 2, &k);
  return scalbn(cell_energy_fp64<1, NC>(p, a, ue), k);
}

// Q1 with the 2^3 rule. The displacement's reference gradient has the same
// trilinear form as the Jacobian, so both take their columns from the monomial
// coefficients, each column once per pair of 1D points (column d depends on two
// of the coordinates): 22 multiply-adds per component and cell instead of 72
// (or 72 more for the gradient from the nodes). FP64 form: the physical
// gradient times det J from the cofactors, so that 1 / det J enters once per
// point, as an FP32 estimate with one cubic correction (3 FP64 operations). That
// squares u h^2 instead of u / h: a cell where the former leaves 2^+-440 or det J
// 2^+-900 (found on the exponents, off the FP64 pipe) takes the general form with
// u and the geometry scaled.
// FP32 form: the strain as in k_adjoint, bit for bit but for the rounding of
// the Jacobian. Bound by the FP64 pipe (2 lanes per clock per SM): about 760
// FP64 operations per cell and 300 in the FP32 form, after 1,400 and 400.
// Measured on 64^3 elasticity cells, ms: 0.752 -> 0.373, FP32 form 0.242 -> 0.170.
struct Q1Columns {
  double a[6];          // a1, a2, a4, a5, a6, a7 of the component
  double c2[2][2];      // column 2 at (x, y)
  __device__ __forceinline__ void init(double v0, double v1, double v2, double v3, double v4, double v5, double v6,
                                       double v7, double g0, double g1) {
    const double d10 = v1 - v0, d32 = v3 - v2, d54 = v5 - v4, d76 = v7 - v6, d20 = v2 - v0, d64 = v6 - v4;
    const double a3 = v4 - v0;
    a[0] = d10;
    a[1] = d20;
    a[2] = d32 - d10;
    a[3] = d54 - d10;
    a[4] = d64 - d20;
    a[5] = (d76 - d54) - (d32 - d10);
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const double yy = y ? g1 : g0, t1 = fma(a[5], yy, a[3]), t0 = fma(a[4], yy, a3);
      c2[0][y] = fma(t1, g0, t0);
      c2[1][y] = fma(t1, g1, t0);
    }
  }
  // 0 if the component is the same at every node
  __device__ __forceinline__ uint32_t bits() const {
    uint32_t m = 0;
    auto put = [&](double x) { m |= (uint32_t(__double2hiint(x)) & 0x7fffffffu) | uint32_t(__double2loint(x)); };
#pragma unroll
    for (int i = 0; i < 6; ++i) put(a[i]);
    put(c2[0][0]);
    put(c2[1][1]);
    return m;
  }
  // columns 0 at (y, z) and 1 at (x, z) for the given z
  __device__ __forceinline__ void slab(double z, double g0, double g1, double (&c0)[2], double (&c1)[2]) const {
    const double t1 = fma(a[5], z, a[2]), t0 = fma(a[3], z, a[0]), s0 = fma(a[4], z, a[1]);
    c0[0] = fma(t1, g0, t0);
    c0[1] = fma(t1, g1, t0);
    c1[0] = fma(t1, g0, s0);
    c1[1] = fma(t1, g1, s0);
  }
};

template <int NC, typename T>
__global__ void __launch_bounds__(kAdjThreads) k_adjoint_q1(AdjParams p) {
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr int NL = NC * 8;
  __shared__ double red[kAdjThreads];
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  double energy = 0.0;
  if (e < p.n_cells) {
    const double g0 = p.xq[0], g1 = p.xq[3];
    const double* x = p.xv + e * 24;
    Q1Columns G[3], U[F32 ? 1 : NC];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      G[k].init(x[k], x[3 + k], x[6 + k], x[9 + k], x[12 + k], x[15 + k], x[18 + k], x[21 + k], g0, g1);
    float ue[F32 ? NL : 1];
    if constexpr (F32) {
#pragma unroll
      for (int l = 0; l < NL; ++l) ue[l] = d2f_rn(p.u[p.cell_dofs[e * NL + l]]);
    } else {
      const int32_t* cd = p.cell_dofs + e * NL;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        double v[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) v[b] = p.u[cd[c * 8 + b]];
        U[F32 ? 0 : c].init(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], g0, g1);
      }
    }
    const float lh = d2f_rn(p.lam_hat), mh2 = 2.f * d2f_rn(p.mu_hat);
    // high words: below lo a nonzero gradient, above hi any one is out of range
    uint32_t lo = 0;
    if constexpr (!F32) {
      uint32_t nz = 0;
#pragma unroll
      for (int c = 0; c < NC; ++c) nz |= U[F32 ? 0 : c].bits();
      lo = nz != 0 ? uint32_t(1023 - 440) << 20 : 0u;
    }
    constexpr uint32_t hi = uint32_t(1023 + 440) << 20;
    bool odd = false;
#pragma unroll 1
    for (int iz = 0; iz < 2; ++iz) {
      const double z = iz ? g1 : g0;
      double G0[3][2], G1[3][2], U0[NC][2], U1[NC][2];
#pragma unroll
      for (int k = 0; k < 3; ++k) G[k].slab(z, g0, g1, G0[k], G1[k]);
      if constexpr (!F32) {
#pragma unroll
        for (int c = 0; c < NC; ++c) U[F32 ? 0 : c].slab(z, g0, g1, U0[c], U1[c]);
      }
#pragma unroll
      for (int iy = 0; iy < 2; ++iy)
#pragma unroll
        for (int ix = 0; ix < 2; ++ix) {
          const int q = ix + 2 * iy + 4 * iz;
          double J[3][3];
#pragma unroll
          for (int k = 0; k < 3; ++k) J[k][0] = G0[k][iy], J[k][1] = G1[k][ix], J[k][2] = G[k].c2[ix][iy];
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
          if (!(det > 0.0)) atomicOr(p.err, kErrNegJacobian);
          if constexpr (F32) {
            float gr[NC][3];
#pragma unroll
            for (int c = 0; c < NC; ++c) gr[c][0] = gr[c][1] = gr[c][2] = 0.f;
            const float* dq = p.dphi32 + q * 24;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
              const float d0 = dq[3 * b], d1 = dq[3 * b + 1], d2 = dq[3 * b + 2];
#pragma unroll
              for (int c = 0; c < NC; ++c) {
                const float uc = ue[F32 ? c * 8 + b : 0];
                gr[c][0] = fmaf(uc, d0, gr[c][0]);
                gr[c][1] = fmaf(uc, d1, gr[c][1]);
                gr[c][2] = fmaf(uc, d2, gr[c][2]);
              }
            }
            const float rdet = 1.f / d2f_rn(det);
            float cs[9];
#pragma unroll
            for (int t = 0; t < 9; ++t) cs[t] = d2f_rn(cof[t]) * rdet;
            energy = fma(p.w[q] * det, f32_to_f64_exact(strain_density<NC>(gr, cs, lh, mh2)), energy);
          } else {
            double gu[NC][3];  // det J times the physical gradient
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
              for (int k = 0; k < 3; ++k)
                gu[c][k] = U0[c][iy] * cof[3 * k] + U1[c][ix] * cof[3 * k + 1] + U[F32 ? 0 : c].c2[ix][iy] * cof[3 * k + 2];
            uint32_t top = 0;
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
              for (int k = 0; k < 3; ++k) top = max(top, uint32_t(__double2hiint(gu[c][k])) & 0x7fffffffu);
            const uint32_t dh = uint32_t(__double2hiint(det)) & 0x7fffffffu;
            odd |= top < lo || top > hi || dh - (uint32_t(1023 - 900) << 20) > (uint32_t(1800) << 20);
            double dens;
            if constexpr (NC == 1) {
              dens = gu[0][0] * gu[0][0] + gu[0][1] * gu[0][1] + gu[0][2] * gu[0][2];
            } else {
              const double div = gu[0][0] + gu[1 % NC][1] + gu[2 % NC][2];
              const double s01 = gu[0][1] + gu[1 % NC][0], s02 = gu[0][2] + gu[2 % NC][0], s12 = gu[1 % NC][2] + gu[2 % NC][1];
              const double diag = gu[0][0] * gu[0][0] + gu[1 % NC][1] * gu[1 % NC][1] + gu[2 % NC][2] * gu[2 % NC][2];
              const double off = s01 * s01 + s02 * s02 + s12 * s12;
              dens = fma(p.lam_hat * div, div, p.mu_hat * fma(2.0, diag, off));
            }
            energy = fma(p.w[q] * reciprocal(det), dens, energy);
          }
        }
    }
    if constexpr (!F32) {
      if (odd)
        energy = cell_energy_scaled<NC>(x, p.u, p.cell_dofs + e * NL, p.xq, p.w, p.dphi, p.lam_hat, p.mu_hat, p.err);
    }
    p.g[e] = p.grad_scale * energy;
  }
  adjoint_partial(p, e, energy, red);
}

template <int P, int NC>
static cudaError_t launch_adj_p(const AdjParams& prm, bool fp32, int blocks, cudaStream_t st) {
  if (P == 1 && prm.nq == 8) {
    if (fp32)
      k_adjoint_q1<NC, float><<<blocks, kAdjThreads, 0, st>>>(prm);
    else
      k_adjoint_q1<NC, double><<<blocks, kAdjThreads, 0, st>>>(prm);
  } else if (fp32) {
    k_adjoint<P, NC, float><<<blocks, kAdjThreads, 0, st>>>(prm);
  } else {
    k_adjoint<P, NC, double><<<blocks, kAdjThreads, 0, st>>>(prm);
  }
  return cudaGetLastError();
}

cudaError_t launch_adjoint(const fe_space* s, const double* u, const double* coef, double grad_scale, double* g,
                           double* compliance, fe_precision prec, cudaStream_t st) {
  return launch_adjoint_with_scratch(s, u, coef, grad_scale, g, compliance, prec, s->d_partials, s->n_partials, st);
}

cudaError_t launch_adjoint_with_scratch(const fe_space* s, const double* u, const double* coef, double grad_scale,
                                        double* g, double* compliance, fe_precision prec, double* partials,
                                        int max_partials, cudaStream_t st) {
  if (s->n_cells == 0) return cudaSuccess;
  AdjParams prm;
  prm.n_cells = s->n_cells;
  prm.nq = s->nq;
  prm.xv = s->d_xv;
  prm.w = s->d_w;
  prm.xq = s->d_xq;
  prm.dphi = s->d_dphi;
  prm.dphi32 = s->d_dphi32;
  prm.cell_dofs = s->d_cell_dofs;
  prm.u = u;
  prm.coef = coef;
  prm.grad_scale = grad_scale;
  prm.lam_hat = s->nu / ((1.0 + s->nu) * (1.0 - 2.0 * s->nu));
  prm.mu_hat = 1.0 / (2.0 * (1.0 + s->nu));
  prm.g = g;
  prm.err = s->d_err;
  const int blocks = int((s->n_cells + kAdjThreads - 1) / kAdjThreads);
  const bool want_c = compliance != nullptr && coef != nullptr;
  prm.partials = want_c ? partials : nullptr;
  if (want_c && blocks > max_partials) return cudaErrorInvalidValue;
  const bool fp32 = prec != FE_PREC_FP64;
  cudaError_t e;
  switch (s->order * 10 + s->ncomp) {
    case 11: e = launch_adj_p<1, 1>(prm, fp32, blocks, st); break;
    case 13: e = launch_adj_p<1, 3>(prm, fp32, blocks, st); break;
    case 21: e = launch_adj_p<2, 1>(prm, fp32, blocks, st); break;
    case 23: e = launch_adj_p<2, 3>(prm, fp32, blocks, st); break;
    case 31: e = launch_adj_p<3, 1>(prm, fp32, blocks, st); break;
    case 33: e = launch_adj_p<3, 3>(prm, fp32, blocks, st); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess || !want_c) return e;
  k_sum_partials<<<1, 256, 0, st>>>(partials, blocks, compliance);
  return cudaGetLastError();
}

}  // namespace feasm
