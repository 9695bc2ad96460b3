// Interior penalty DG for the Poisson problem (paper, Sect. "Non-conforming
// methods", Eq. ip_dg_formulations, Eq. mean_and_jump_ops, Eq.
// local_to_face_matrix): discontinuous Q_p, cell-local DOFs K*nb + a.
//
// GB300 form: the cell integrals come from the Poisson cell kernels of an
// internal fe_space of the same order (FP64 or FP32 form); the facet integrals
// from k_dg_facets (FP32 forms) or k_dg_facets_fixed (FP64 form): persistent
// blocks, one facet at a time, its four nb x nb blocks, or one for a boundary
// facet, through small products over the face nodes; one warp forms the next
// facet's FP64 point data while the others form the products. The facet kernel
// stores the off-diagonal blocks at their CSR places and the diagonal ones to
// scratch; k_dg_rows then writes each cell's diagonal block, the cell matrix
// plus the cell's six facet diagonal blocks in face order (fixed order:
// deterministic). Storing all four blocks to scratch and copying them in the row
// kernel moved 4 nb^2 more values per facet; with the block rows walked by
// pointers instead of divisions the FP32 form of 32^3 Q2 cells went from 2.75
// to 2.04 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "fe_device.cuh"
#include "fe_launch.h"

namespace feasm {
namespace dg {

constexpr int kSelf = 6;  // block slot code of the cell itself (0..5: the neighbour through that face)

}  // namespace dg
}  // namespace feasm

struct fe_dg {
  fe_space* s = nullptr;     // Poisson space of the same order: cell integrals, geometry, tables
  int p = 0, nb = 0;
  int64_t n_cells = 0, n_dofs = 0, nnz = 0;
  bool host_only = false;
  // interior facets: cells K+ < K-, their local faces, and for each corner (s, t)
  // of K+'s face (s, t in {0,1}, corner index s + 2t) the local vertex of K- there
  std::vector<int32_t> fplus, fminus;
  std::vector<uint8_t> fpf, fmf, fcorner;  // fcorner [n_int][4]
  std::vector<int32_t> bcell;
  std::vector<uint8_t> bface;
  // per cell: the code of each local face (interior facet i on side s: 2 i + s;
  // boundary facet j: -1 - j) and the block slots of its row in column order
  std::vector<int32_t> face_code;  // [cells][6]
  std::vector<uint8_t> slots;      // [cells][7]: face through which the neighbour is reached, or kSelf
  std::vector<uint8_t> nslot;      // [cells]
  std::vector<int64_t> row_ptr;
  std::vector<int32_t> col;
  // device
  int32_t* d_fplus = nullptr;
  int32_t* d_fminus = nullptr;
  uint8_t* d_fpf = nullptr;
  uint8_t* d_fmf = nullptr;
  uint8_t* d_fcorner = nullptr;
  int32_t* d_bcell = nullptr;
  uint8_t* d_bface = nullptr;
  int32_t* d_face_code = nullptr;
  uint8_t* d_slots = nullptr;
  uint8_t* d_nslot = nullptr;
  int64_t* d_row_ptr = nullptr;
  int32_t* d_col = nullptr;
  double* d_ones = nullptr;    // unit coefficients of the cell integrals
  double* d_fblk = nullptr;    // diagonal blocks of the interior facets [n_int][2][nb][nb]
  double* d_bblk = nullptr;    // boundary facet blocks [n_bnd][nb][nb]
  double* d_gx = nullptr;      // face Gauss rule on [0,1], p+1 points
  double* d_gw = nullptr;
  // FP64 form (FacetTables)
  int fix_lp = 0, fix_ld = 0;
  int32_t* d_fix = nullptr;
  double* d_fix_dn = nullptr;
};

namespace {

// local vertex of the corner (s, t) of local face f: xhat_d = f % 2, s along
// the lower and t along the higher of the two other axes
int face_corner_vertex(int f, int s, int t) {
  const int d = f / 2, d1 = d == 0 ? 1 : 0, d2 = d == 2 ? 1 : 2;
  return ((f % 2) << d) | (s << d1) | (t << d2);
}

int setup_dg(fe_dg* g, const fe_mesh_desc* mesh, std::string* err) {
  const int64_t nc = mesh->n_cells;
  const int nb = g->nb;
  g->face_code.assign(size_t(nc) * 6, 0);
  std::map<std::array<int32_t, 4>, std::pair<int32_t, int>> open;  // sorted face key -> (cell, face)
  for (int64_t e = 0; e < nc; ++e) {
    const int32_t* cv = mesh->cell_vertices + 8 * e;
    for (int f = 0; f < 6; ++f) {
      std::array<int32_t, 4> key;
      for (int c = 0; c < 4; ++c) key[c] = cv[face_corner_vertex(f, c & 1, c >> 1)];
      std::sort(key.begin(), key.end());
      auto it = open.find(key);
      if (it == open.end()) {
        open.emplace(key, std::make_pair(int32_t(e), f));
        continue;
      }
      // second cell on this face: an interior facet, K+ = the earlier (lower) cell
      const int32_t kp = it->second.first;
      const int fp = it->second.second;
      open.erase(it);
      const int32_t i = int32_t(g->fplus.size());
      g->fplus.push_back(kp);
      g->fminus.push_back(int32_t(e));
      g->fpf.push_back(uint8_t(fp));
      g->fmf.push_back(uint8_t(f));
      const int32_t* cvp = mesh->cell_vertices + 8 * int64_t(kp);
      for (int c = 0; c < 4; ++c) {
        const int32_t v = cvp[face_corner_vertex(fp, c & 1, c >> 1)];
        int lv = -1;
        for (int w = 0; w < 8; ++w)
          if (cv[w] == v) lv = w;
        if (lv < 0) {
          *err = "facet vertices do not match";
          return FE_ERR_INVALID_ARG;
        }
        g->fcorner.push_back(uint8_t(lv));
      }
      // K+'s face corners (s, t) = (0,0), (1,0), (0,1), (1,1) on K-'s reference
      // corners: a symmetry of the square, i.e. corner (1,1) = (1,0) + (0,1) - (0,0)
      // in every reference coordinate (the facet kernel relies on it)
      const uint8_t* fc = g->fcorner.data() + g->fcorner.size() - 4;
      for (int k = 0; k < 3; ++k) {
        const int b[4] = {(fc[0] >> k) & 1, (fc[1] >> k) & 1, (fc[2] >> k) & 1, (fc[3] >> k) & 1};
        if (b[3] != b[1] + b[2] - b[0]) {
          *err = "facet corners of the two cells are not related by a symmetry of the square";
          return FE_ERR_INVALID_ARG;
        }
      }
      g->face_code[size_t(kp) * 6 + fp] = 2 * i;
      g->face_code[size_t(e) * 6 + f] = 2 * i + 1;
    }
  }
  // what stays open is on the boundary (ascending cell, face)
  std::vector<std::pair<int32_t, int>> bnd;
  for (auto& kv : open) bnd.push_back(kv.second);
  std::sort(bnd.begin(), bnd.end());
  for (auto& b : bnd) {
    const int32_t j = int32_t(g->bcell.size());
    g->bcell.push_back(b.first);
    g->bface.push_back(uint8_t(b.second));
    g->face_code[size_t(b.first) * 6 + b.second] = -1 - j;
  }
  // block slots of each cell's rows (cells ascending) and the CSR pattern
  g->slots.assign(size_t(nc) * 7, 0);
  g->nslot.assign(nc, 0);
  g->row_ptr.assign(size_t(nc) * nb + 1, 0);
  for (int64_t e = 0; e < nc; ++e) {
    std::vector<std::pair<int32_t, int>> blk{{int32_t(e), feasm::dg::kSelf}};
    for (int f = 0; f < 6; ++f) {
      const int32_t code = g->face_code[size_t(e) * 6 + f];
      if (code < 0) continue;
      const int32_t i = code >> 1;
      blk.push_back({(code & 1) ? g->fplus[i] : g->fminus[i], f});
    }
    std::sort(blk.begin(), blk.end());
    g->nslot[e] = uint8_t(blk.size());
    for (size_t j = 0; j < blk.size(); ++j) g->slots[size_t(e) * 7 + j] = uint8_t(blk[j].second);
    for (int a = 0; a < nb; ++a)
      g->row_ptr[size_t(e) * nb + a + 1] = int64_t(blk.size()) * nb;
    for (int a = 0; a < nb; ++a)
      for (auto& b : blk)
        for (int c = 0; c < nb; ++c) g->col.push_back(int32_t(int64_t(b.first) * nb + c));
  }
  for (size_t r = 0; r + 1 < g->row_ptr.size(); ++r) g->row_ptr[r + 1] += g->row_ptr[r];
  g->nnz = g->row_ptr.back();
  if (g->nnz > INT32_MAX * int64_t(8)) {
    *err = "too many nonzeros";
    return FE_ERR_UNSUPPORTED;
  }
  return FE_OK;
}

}  // namespace

namespace feasm {
namespace dg {

// Exact FP32 -> FP64 on the integer bits: the short path for zeros and normal
// numbers, the general one otherwise.
__device__ __forceinline__ double to_f64(float x) {
  return f32_zero_or_normal(x) ? f32_to_f64_normal(x) : f32_to_f64_exact(x);
}

struct FacetParams {
  int64_t n_int, n_bnd;
  const double* xv;  // [cells][8][3]
  const int32_t* fplus;
  const int32_t* fminus;
  const uint8_t* fpf;
  const uint8_t* fmf;
  const uint8_t* fcorner;
  const int32_t* bcell;
  const uint8_t* bface;
  const double* gx;  // face Gauss points [n1] on [0,1]
  const double* gw;
  double tau, gamma;
  void* fblk;  // diagonal blocks of the interior facets [n_int][2][nb][nb], double (FP64 form) or float
  void* bblk;  // [n_bnd][nb][nb]
  double* values;  // the off-diagonal blocks go straight to their CSR places
  const uint8_t* slots;
  const uint8_t* nslot;
  const int64_t* row_ptr;
  const int2* fix;      // FP64 form: FacetTables (limbs)
  const double* fix_dn; // FP64 form: derivatives of the 1D basis at 0 and 1, [2][n1]
  int fix_lp, fix_ld;
  int* err;
};

// Where the facet's off-diagonal blocks go: entry (a, b) of the block in side
// s's rows at values[base[s] + a len[s] + b].
struct FacetOut {
  int64_t base[2];
  int len[2];
};

// (lanes 0 and 1 of the point warp, one side each)
template <int NB>
__device__ __forceinline__ void facet_out(const FacetParams& fp, int64_t cell, int face, int s, FacetOut* o) {
  const int ns = fp.nslot[cell];
  int j = 0;
  for (int k = 0; k < ns; ++k)
    if (fp.slots[cell * 7 + k] == face) j = k;
  o->base[s] = fp.row_ptr[cell * NB] + int64_t(j) * NB;
  o->len[s] = ns * NB;
}

// 1D Lagrange polynomials on the nodes m/P and their derivatives at x, in T.
template <int P, typename T>
__device__ __forceinline__ void lagrange(T x, T* v, T* d) {
#pragma unroll
  for (int m = 0; m <= P; ++m) {
    T val = T(1), der = T(0);
#pragma unroll
    for (int s = 0; s <= P; ++s) {
      if (s == m) continue;
      const T den = T(m - s) / T(P);
      der = der * ((x - T(s) / T(P)) / den) + val / den;
      val *= (x - T(s) / T(P)) / den;
    }
    v[m] = val;
    d[m] = der;
  }
}

// Shared memory of k_dg_facets for order P. The per-facet point data are
// double-buffered (the point warp fills facet n+1's while the other warps use
// facet n's): the sides' trilinear coefficients and |F| in double; cof^T n /
// det, the 1D Lagrange data, the surface elements (FP32) and the face-node
// indices. The products' operands and results (FP32) belong to the product
// warps alone.
template <int P>
struct FacetLayout {
  static constexpr int N1 = P + 1, NB = N1 * N1 * N1, NQF = N1 * N1, NBF = N1 * N1;
  static constexpr size_t S = sizeof(float);
  // one point-data buffer
  static constexpr size_t B_ACO = 0;                                      // double [2][21]
  static constexpr size_t B_AREA = B_ACO + size_t(2) * 21 * 8;           // double |F|
  static constexpr size_t B_CN = B_AREA + 8;                              // float [2][NQF][3]
  static constexpr size_t B_VD = B_CN + size_t(2) * NQF * 3 * S;          // float [2][NQF][2][3][N1]
  static constexpr size_t B_DS = B_VD + size_t(2) * NQF * 6 * N1 * S;     // float [NQF]
  static constexpr size_t B_CIDX = (B_DS + size_t(NQF) * S + 3) & ~size_t(3);  // int [2][NB]
  static constexpr size_t B_OUT = (B_CIDX + size_t(2) * NB * 4 + 7) & ~size_t(7);  // FacetOut
  static constexpr size_t B_BYTES = (B_OUT + sizeof(FacetOut) + 15) & ~size_t(15);
  static constexpr size_t PT = 0;                                         // two buffers
  static constexpr size_t GN = PT + 2 * B_BYTES;                          // [2][NQF][NB]   grad phi . n
  static constexpr size_t PF = GN + size_t(2) * NQF * NB * S;             // [2][NQF][NBF]  dS phi (face nodes)
  static constexpr size_t FF = PF + size_t(2) * NQF * NBF * S;            // [2][NQF][NBF]  phi (face nodes)
  static constexpr size_t X1 = FF + size_t(2) * NQF * NBF * S;            // [4][NBF][NB]
  static constexpr size_t YY = X1 + size_t(4) * NBF * NB * S;             // [4][NBF][NBF]
  static constexpr size_t BYTES = YY + size_t(4) * NBF * NBF * S;
};

// The facet named by id (interior facets first, then boundary facets).
struct FacetRef {
  bool interior;
  int64_t i;  // index among the interior or the boundary facets
  int ns;     // sides
  int face[2];
  int64_t cell[2];
};

__device__ __forceinline__ FacetRef facet_ref(const FacetParams& fp, int64_t id) {
  FacetRef f;
  f.interior = id < fp.n_int;
  f.i = f.interior ? id : id - fp.n_int;
  f.ns = f.interior ? 2 : 1;
  f.face[0] = f.interior ? int(fp.fpf[f.i]) : int(fp.bface[f.i]);
  f.face[1] = f.interior ? int(fp.fmf[f.i]) : 0;
  f.cell[0] = f.interior ? int64_t(fp.fplus[f.i]) : int64_t(fp.bcell[f.i]);
  f.cell[1] = f.interior ? int64_t(fp.fminus[f.i]) : 0;
  return f;
}

// Jacobian, cofactors and determinant at (x, y, z) from the trilinear
// coefficients: 45 FP64 operations.
__device__ __forceinline__ void facet_geometry(const double* a, double x, double y, double z, double (&cof)[9], double* det) {
  double J[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double a4 = a[9 + k], a5 = a[12 + k], a6 = a[15 + k], a7 = a[18 + k];
    const double t = fma(a7, z, a4);
    J[k][0] = fma(t, y, fma(a5, z, a[k]));
    J[k][1] = fma(t, x, fma(a6, z, a[3 + k]));
    J[k][2] = fma(fma(a7, y, a5), x, fma(a6, y, a[6 + k]));
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

// 1 / sqrt(x) with the FP32 estimate and one cubic correction (5 FP64
// operations) for positive normal x, else rsqrt.
static __device__ __noinline__ double rsqrt_slow(double x) { return rsqrt(x); }
__device__ __forceinline__ double rsqrt_fast(double x) {
  bool odd = false;
  int k2;
  const double y = fix_rsqrt(x, k2, odd);
  return odd ? rsqrt_slow(x) : fix_scale2(y, -k2);
}

// x with its sign flipped if neg, on the integer bits
__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? int(0x80000000u) : 0), __double2loint(x));
}

// Sum over the lanes below N of a warp (lanes from N on pass 0), in every lane
// below 2^ceil(log2 N).
template <int N>
__device__ __forceinline__ double low_lanes_sum(double v) {
  constexpr int H = N > 8 ? 8 : N > 4 ? 4 : N > 2 ? 2 : 1;
#pragma unroll
  for (int off = H; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

// Point data of facet id into buffer b (all 32 lanes of the point warp):
// each side's compact face-node index (node index along the face normal =
// the face's side) and trilinear coefficients; then one lane per (side,
// point) (2 (p+1)^2 <= 32): the reference point (side 1: each coordinate s,
// 1 - s, t, 1 - t or the face's side, read off the reference corners of K-
// that carry K+'s face corners), FP64 geometry, the physical normal and
// surface element of the point from cof(J+) nhat = det J+ J+^{-T} nhat
// (side-0 lanes; shuffled to the side-1 lane of the same point), |F| (a
// butterfly sum over the side-0 lanes), cof^T n / det and the 1D Lagrange
// data.
template <int P>
__device__ __forceinline__ void facet_points(const FacetParams& fp, int64_t id, unsigned char* b, int lane) {
  using L = FacetLayout<P>;
  constexpr int N1 = L::N1, NB = L::NB, NQF = L::NQF;
  static_assert(2 * NQF <= 32, "one lane per (side, point)");
  double* aco = reinterpret_cast<double*>(b + L::B_ACO);
  float* cnv = reinterpret_cast<float*>(b + L::B_CN);
  float* vd = reinterpret_cast<float*>(b + L::B_VD);
  float* dsw = reinterpret_cast<float*>(b + L::B_DS);
  int* cidx = reinterpret_cast<int*>(b + L::B_CIDX);
  const FacetRef f = facet_ref(fp, id);
  for (int it = lane; it < f.ns * NB; it += 32) {
    const int s = it / NB, a = it % NB, d = f.face[s] / 2;
    const int ad = (a / (d == 0 ? 1 : (d == 1 ? N1 : N1 * N1))) % N1;
    int c = -1;
    if (ad == (f.face[s] % 2) * P) {
      const int d1 = d == 0 ? 1 : 0, d2 = d == 2 ? 1 : 2;
      const int st1 = d1 == 0 ? 1 : (d1 == 1 ? N1 : N1 * N1), st2 = d2 == 0 ? 1 : (d2 == 1 ? N1 : N1 * N1);
      c = (a / st1) % N1 + N1 * ((a / st2) % N1);
    }
    cidx[s * NB + a] = c;
  }
  if (lane < 3 * f.ns) trilinear_coefficients(fp.xv + f.cell[lane / 3] * 24, lane % 3, aco + (lane / 3) * 21);
  if (f.interior && lane < 2)
    facet_out<NB>(fp, lane ? f.cell[1] : f.cell[0], lane ? f.face[1] : f.face[0], lane, reinterpret_cast<FacetOut*>(b + L::B_OUT));
  __syncwarp();
    const bool act = lane < f.ns * NQF;
    const int side = act ? lane / NQF : 0, q = lane % NQF, qs = q % N1, qt = q / N1;
    const double s = fp.gx[qs], tt = fp.gx[qt];
    // (selects, not indexing by the face's direction, so that xh, cof and
    // nd stay in registers)
    double xh[3];
    if (side == 0) {
      const int d = f.face[0] / 2;
      const double fv = double(f.face[0] % 2);
      xh[0] = d == 0 ? fv : s;
      xh[1] = d == 1 ? fv : (d == 0 ? s : tt);
      xh[2] = d == 2 ? fv : tt;
    } else {
      // the corners of K+'s face sit on K-'s reference corners v0 (s, t) =
      // (0, 0), v1 (1, 0), v2 (0, 1), v3 = v1 + v2 - v0 (a symmetry of the
      // square, checked at setup), so each reference coordinate of K-'s
      // point is v0 + (v1 - v0) s + (v2 - v0) t: one of s, 1 - s, t, 1 - t
      // or the face's side
      const int v0 = fp.fcorner[4 * f.i], v1 = fp.fcorner[4 * f.i + 1], v2 = fp.fcorner[4 * f.i + 2];
      const double sm1 = 1.0 - s, tm1 = 1.0 - tt;
      const int d = f.face[1] / 2;
      const double fv = double(f.face[1] % 2);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int b0 = (v0 >> k) & 1, d1 = ((v1 >> k) & 1) - b0, d2 = ((v2 >> k) & 1) - b0;
        xh[k] = k == d ? fv : (d1 > 0 ? s : d1 < 0 ? sm1 : d2 > 0 ? tt : d2 < 0 ? tm1 : double(b0));
      }
    }
    double cof[9], det;
    facet_geometry(aco + side * 21, xh[0], xh[1], xh[2], cof, &det);
    if (act && !(det > 0.0)) atomicOr(fp.err, kErrNegJacobian);
    // the normal of point q: cof(J+) nhat on the side-0 lane q
    const int d = f.face[0] / 2;
    const bool low = f.face[0] % 2 == 0;
    double nd[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      nd[k] = flip(d == 0 ? cof[3 * k] : (d == 1 ? cof[3 * k + 1] : cof[3 * k + 2]), low);
      nd[k] = __shfl_sync(kFull, nd[k], q);
    }
    const double l2 = nd[0] * nd[0] + nd[1] * nd[1] + nd[2] * nd[2];
    const double rl = rsqrt_fast(l2), len = l2 * rl;
    const double dsq = len * fp.gw[qs] * fp.gw[qt];
    const double ar = low_lanes_sum<NQF>(lane < NQF ? dsq : 0.0);
    if (act) {
      const double rdet = reciprocal(det);
      const double n0 = nd[0] * rl, n1 = nd[1] * rl, n2 = nd[2] * rl;
#pragma unroll
      for (int k = 0; k < 3; ++k) cnv[lane * 3 + k] = d2f_rn((cof[k] * n0 + cof[3 + k] * n1 + cof[6 + k] * n2) * rdet);
      // the 1D shape data; FP32 forms with p <= 2 evaluate them in FP32 at the
      // rounded reference point (nodes 0, 1/2, 1 exact, every Gauss point
      // and its mirror at least 0.11 from a node); for p = 3 a 4-point Gauss
      // abscissa lies 0.003 from the node 1/3, so x - 1/3 is formed in FP64
      float* vt = vd + lane * 6 * N1;  // V[k][m] at k*N1 + m, D at (3 + k)*N1 + m
      if constexpr (P <= 2) {
#pragma unroll
        for (int k = 0; k < 3; ++k) lagrange<P, float>(d2f_rn(xh[k]), vt + k * N1, vt + (3 + k) * N1);
      } else {
        double V[3][N1], D[3][N1];
#pragma unroll
        for (int k = 0; k < 3; ++k) lagrange<P, double>(xh[k], V[k], D[k]);
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int m = 0; m < N1; ++m) {
            vt[k * N1 + m] = d2f_rn(V[k][m]);
            vt[(3 + k) * N1 + m] = d2f_rn(D[k][m]);
          }
      }
      if (side == 0) dsw[q] = d2f_rn(dsq);
    }
    if (lane == 0) *reinterpret_cast<double*>(b + L::B_AREA) = ar;
}

__device__ __forceinline__ void product_barrier() { asm volatile("bar.sync 1, 96;" ::: "memory"); }

// One block of 128 threads per facet at a time, persistent, with warp roles:
//   warp 3      the point data of the block's next facet (facet_points) into
//               the other buffer;
//   warps 0-2   with facet n's point data:
//     3. per (side, point) row and node column: the normal derivative of every
//        shape function and the values of the (p+1)^2 face nodes (the other
//        shape functions vanish on the face);
//     4. the products X_{sa,sb} = sum_q dS phi^{sa}_{a'} (grad phi^{sb}_b . n)
//        (a' a face node of side sa) and Y_{sa,sb} = sum_q dS phi^{sa}_{a'} phi^{sb}_{b'};
//     5. block (sa, sb), row a, column b:
//        -s_a/2 X_{sa,sb}[a'][b] - tau s_b/2 X_{sb,sa}[b'][a] + gamma/|F| s_a s_b Y_{sa,sb}[a'][b']
//        (terms whose face node is missing are zero; boundary facets: one side,
//        s = 1 and the factor 1/2 dropped), Eq. local_to_face_matrix;
//     named barrier 1 (96 threads) between the steps.
// One block barrier per facet hands the buffers over; every thread runs the
// same facet loop, so each barrier sees all of its threads. Geometry, normals,
// |F| and the 1D shape data (for p = 3; p <= 2 forms them in FP32) in FP64,
// rounded to FP32 on the integer bits; steps 3 to 5 in FP32, diagonal blocks
// stored in FP32, the others converted exactly. GB300 issues FP64 at 2 lanes
// per clock per SM: the point warp's FP64 chain is the part the roles overlap.
template <int P>
__global__ void __launch_bounds__(128) k_dg_facets(FacetParams fp) {
  using L = FacetLayout<P>;
  constexpr int N1 = L::N1, NB = L::NB, NQF = L::NQF, NBF = L::NBF;
  constexpr int NW = 3, NBJ = (NB + 31) / 32;
  extern __shared__ __align__(16) unsigned char sm[];
  float* gn = reinterpret_cast<float*>(sm + L::GN);
  float* pf = reinterpret_cast<float*>(sm + L::PF);
  float* ff = reinterpret_cast<float*>(sm + L::FF);
  float* x1 = reinterpret_cast<float*>(sm + L::X1);
  float* yy = reinterpret_cast<float*>(sm + L::YY);
  // roles rotate with the block: warp w of every block sits on the same
  // sub-partition, and the point warps' FP64 work has to spread over all four
  const int warp = ((threadIdx.x >> 5) + blockIdx.x) & 3, lane = threadIdx.x & 31, t = warp * 32 + lane;
  const int64_t n_fac = fp.n_int + fp.n_bnd;
  // steps 3 and 5 give each product warp whole rows and each lane the columns
  // b = lane + 32 j; the tensor-product digits of those columns, once
  int bd[NBJ][3];
#pragma unroll
  for (int j = 0; j < NBJ; ++j) {
    const int bb = lane + 32 * j;
    bd[j][0] = bb % N1;
    bd[j][1] = N1 + (bb / N1) % N1;
    bd[j][2] = 2 * N1 + (bb / (N1 * N1)) % N1;
  }
  if (warp == 3 && blockIdx.x < n_fac) facet_points<P>(fp, blockIdx.x, sm + L::PT, lane);
  __syncthreads();
  int buf = 0;
  for (int64_t id = blockIdx.x; id < n_fac; id += gridDim.x, buf ^= 1) {
    if (warp == 3) {
      const int64_t nx = id + gridDim.x;
      if (nx < n_fac) facet_points<P>(fp, nx, sm + L::PT + (buf ^ 1) * L::B_BYTES, lane);
    } else {
      const unsigned char* b = sm + L::PT + buf * L::B_BYTES;
      const float* cnv = reinterpret_cast<const float*>(b + L::B_CN);
      const float* vd = reinterpret_cast<const float*>(b + L::B_VD);
      const float* dsw = reinterpret_cast<const float*>(b + L::B_DS);
      const int* cidx = reinterpret_cast<const int*>(b + L::B_CIDX);
      const double area = *reinterpret_cast<const double*>(b + L::B_AREA);
      const FacetOut* fo = reinterpret_cast<const FacetOut*>(b + L::B_OUT);
      const FacetRef f = facet_ref(fp, id);
      const int ns = f.ns;
      // the face-node index of the lane's columns on each side
      int cbl[2][NBJ];
#pragma unroll
      for (int j = 0; j < NBJ; ++j) {
        const int bb = lane + 32 * j;
        cbl[0][j] = bb < NB ? cidx[bb] : -1;
        cbl[1][j] = bb < NB && ns == 2 ? cidx[NB + bb] : -1;
      }
      // 3. row (side, point), column node b: normal derivative; value and dS
      //    value on face nodes
      for (int r = warp; r < ns * NQF; r += NW) {
        const int side = r / NQF, q = r % NQF;
        const float* V = vd + r * 6 * N1;  // values at 0..3 N1, derivatives 3 N1 further
        const float c0 = cnv[r * 3], c1 = cnv[r * 3 + 1], c2 = cnv[r * 3 + 2], dq = dsw[q];
  #pragma unroll
        for (int j = 0; j < NBJ; ++j) {
          const int b = lane + 32 * j;
          if (b < NB) {
            const float v0 = V[bd[j][0]], v1 = V[bd[j][1]], v2 = V[bd[j][2]];
            const float d0 = V[3 * N1 + bd[j][0]], d1 = V[3 * N1 + bd[j][1]], d2 = V[3 * N1 + bd[j][2]];
            gn[r * NB + b] = c0 * d0 * v1 * v2 + c1 * v0 * d1 * v2 + c2 * v0 * v1 * d2;
            const int c = side ? cbl[1][j] : cbl[0][j];
            if (c >= 0) {
              const float ph = v0 * v1 * v2;
              ff[r * NBF + c] = ph;
              pf[r * NBF + c] = dq * ph;
            }
          }
        }
      }
      product_barrier();
      // 4. X_{sa,sb} scaled by -s_a/2 (boundary: -1), row (block, face node c),
      //    column b; Y_{sa,sb} scaled by s_a s_b
      const float half = f.interior ? float(0.5) : float(1);
      for (int r = warp; r < ns * ns * NBF; r += NW) {
        const int blk = r / NBF, c = r % NBF, sa = blk >> 1, sb = blk & 1;
        float pq[NQF];
  #pragma unroll
        for (int q = 0; q < NQF; ++q) pq[q] = pf[(sa * NQF + q) * NBF + c];
        const float* g = gn + sb * NQF * NB;
        const float sc = sa ? half : -half;
  #pragma unroll
        for (int j = 0; j < NBJ; ++j) {
          const int b = lane + 32 * j;
          if (b < NB) {
            float v = float(0);
  #pragma unroll
            for (int q = 0; q < NQF; ++q) v = fma(pq[q], g[q * NB + b], v);
            x1[r * NB + b] = sc * v;
          }
        }
      }
      for (int it = t; it < ns * ns * NBF * NBF; it += 32 * NW) {
        const int blk = it / (NBF * NBF), sa = blk >> 1, sb = blk & 1, c = (it / NBF) % NBF, e = it % NBF;
        float v = float(0);
  #pragma unroll
        for (int q = 0; q < NQF; ++q) v = fma(pf[(sa * NQF + q) * NBF + c], ff[(sb * NQF + q) * NBF + e], v);
        yy[(blk * NBF + c) * NBF + e] = sa == sb ? v : -v;
      }
      product_barrier();
      // 5. the facet blocks, warp w rows a = w, w + 3, ..: X term, tau times the
      //    transposed X term of the swapped block, gamma/|F| times the Y term
      //    (entries with no face node: zero, no arithmetic)
      const float pen = d2f_rn(fp.gamma / area), tau = d2f_rn(fp.tau);
      for (int blk = 0; blk < ns * ns; ++blk) {
        const int sa = blk >> 1, sb = blk & 1;
        const float* xr = x1 + blk * NBF * NB + lane;
        const float* xt = x1 + ((sb << 1) | sa) * NBF * NB;
        const float* yr = yy + blk * NBF * NBF;
        float* diag = f.interior ? static_cast<float*>(fp.fblk) + (f.i * 2 + sa) * NB * NB : static_cast<float*>(fp.bblk) + f.i * NB * NB;
        diag += warp * NB + lane;
        const int len = sa != sb ? fo->len[sa] : 0;
        double* off = fp.values + (sa != sb ? fo->base[sa] + int64_t(warp) * len + lane : 0);
        for (int a = warp; a < NB; a += NW, diag += NW * NB, off += NW * len) {
          const int ca = cidx[sa * NB + a];
  #pragma unroll
          for (int j = 0; j < NBJ; ++j) {
            if (NB % 32 != 0 && lane + 32 * j >= NB) continue;
            const int cb = sb ? cbl[1][j] : cbl[0][j];
            float v = ca >= 0 ? xr[ca * NB + 32 * j] : float(0);
            if (cb >= 0) {
              v = fma(tau, xt[cb * NB + a], v);
              if (ca >= 0) v = fma(pen, yr[ca * NBF + cb], v);
            }
            if (sa == sb) {
              diag[32 * j] = v;
            } else {
              off[32 * j] = to_f64(v);
            }
          }
        }
      }
    }
    __syncthreads();
  }
}

// Shared memory of k_dg_facets_fixed: two point-data buffers, the tables, the
// right-hand operands and the results of one facet.
template <int P>
struct FixedFacetLayout {
  static constexpr int N1 = P + 1, NB = N1 * N1 * N1, NQF = N1 * N1, NBF = N1 * N1;
  // (odd_facets puts doubles in the place of w and ds)
  struct Points {
    FacetOut out;
    double pen;          // gamma / |F|
    int2 w[2][NQF][3];   // dS (cof^T n / det) along the face's normal axis and its two other axes
    int2 ds[NQF];        // dS
    int perm[2][NQF];    // the point's index in the side's own face rule
    int ew[2][2], ey;    // scales: |w| < 2^ew per side and kind of axis (normal, the two others), dS < 2^ey
    int odd;             // out of range: left to odd_facets
  };
  static constexpr size_t PT = 0;
  static constexpr size_t TAB = PT + 2 * ((sizeof(Points) + 15) & ~size_t(15));      // int2 [4][NQF][NBF]
  static constexpr size_t R = TAB + size_t(4) * NQF * NBF * 8;                       // int2 [2][NQF][NBF][3]
  static constexpr size_t X = R + size_t(2) * NQF * NBF * 24;                        // double [4][NBF][N1][NBF]
  static constexpr size_t Y = X + size_t(4) * NBF * NB * 8;                          // double [4][NBF][NBF]
  static constexpr size_t XB = Y + size_t(4) * NBF * NBF * 8;                        // double [4][NBF][NBF]
  static constexpr size_t DN = XB + size_t(4) * NBF * NBF * 8;                       // double [2][N1]
  static constexpr size_t NODES = DN + size_t(2) * N1 * 8;                           // uint8 [6][NB]: c | layer << 4
  static constexpr size_t BYTES = NODES + size_t(6) * NB;
};

// Face node (index along the face's two axes) and layer along its normal axis
// of node a, for local face f.
template <int N1>
__device__ __forceinline__ uint8_t face_node(int f, int a) {
  const int d = f / 2, i0 = a % N1, i1 = (a / N1) % N1, i2 = a / (N1 * N1);
  const int m = d == 0 ? i0 : d == 1 ? i1 : i2, c = d == 0 ? i1 + N1 * i2 : d == 1 ? i0 + N1 * i2 : i0 + N1 * i1;
  return uint8_t(c | (m << 4));
}

// Reference point (qs, qt) of the face rule on the given side, and the index of each coordinate among the 1D points.
template <int P>
__device__ __forceinline__ void face_point(const FacetParams& fp, const FacetRef& f, int side, int qs, int qt, double (&xh)[3],
                                           int (&at)[3]) {
  const double s = fp.gx[qs], tt = fp.gx[qt];
  const int d = side ? f.face[1] / 2 : f.face[0] / 2;
  const double fv = double(side ? f.face[1] % 2 : f.face[0] % 2);
  if (side == 0) {
    xh[0] = d == 0 ? fv : s;
    xh[1] = d == 1 ? fv : (d == 0 ? s : tt);
    xh[2] = d == 2 ? fv : tt;
    at[0] = qs;
    at[1] = d == 0 ? qs : qt;
    at[2] = qt;
  } else {
    // K-'s reference coordinates: one of s, 1 - s, t, 1 - t or the face's side (see facet_points)
    const int v0 = fp.fcorner[4 * f.i], v1 = fp.fcorner[4 * f.i + 1], v2 = fp.fcorner[4 * f.i + 2];
    const double sm1 = 1.0 - s, tm1 = 1.0 - tt;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int b0 = (v0 >> k) & 1, d1 = ((v1 >> k) & 1) - b0, d2 = ((v2 >> k) & 1) - b0;
      xh[k] = k == d ? fv : (d1 > 0 ? s : d1 < 0 ? sm1 : d2 > 0 ? tt : d2 < 0 ? tm1 : double(b0));
      at[k] = d1 > 0 ? qs : d1 < 0 ? P - qs : d2 > 0 ? qt : P - qt;
    }
  }
}

__device__ __forceinline__ double raw_double(int2 x) { return __hiloint2double(x.y, x.x); }
__device__ __forceinline__ int2 raw_int2(double x) { return make_int2(__double2loint(x), __double2hiint(x)); }

// The weights of a facet out of the fixed-point range (all 32 lanes of a product
// warp), as plain doubles: the normal scaled by a power of two before it is
// squared, and of unit length before the products.
template <int P>
__device__ __forceinline__ void facet_weights_fp64(const FacetParams& fp, const FacetRef& f,
                                                   typename FixedFacetLayout<P>::Points* b, int lane) {
  constexpr int N1 = P + 1, NQF = N1 * N1;
  const bool act = lane < f.ns * NQF;
  const int side = act ? lane / NQF : 0, q = lane % NQF, qs = q % N1, qt = q / N1, d = f.face[side] / 2, dp = f.face[0] / 2;
  const double gww = fp.gw[qs] * fp.gw[qt];
  double a[21], xh[3], cof[9], det, n[3], w[3];
  int at[3];
  for (int k = 0; k < 3; ++k) trilinear_coefficients(fp.xv + f.cell[side] * 24, k, a);
  face_point<P>(fp, f, side, qs, qt, xh, at);
  facet_geometry(a, xh[0], xh[1], xh[2], cof, &det);
  for (int k = 0; k < 3; ++k) n[k] = __shfl_sync(kFull, flip(cof[3 * k + dp], f.face[0] % 2 == 0), q);
  const double big = fmax(fabs(n[0]), fmax(fabs(n[1]), fabs(n[2])));
  const int e = big > 0.0 && big < INFINITY ? ilogb(big) : 0;
  for (int k = 0; k < 3; ++k) n[k] = scalbn(n[k], -e);
  const double len = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]), rdet = 1.0 / det, ds = scalbn(len, e) * gww;
  for (int k = 0; k < 3; ++k)
    w[k] = (cof[k] * (n[0] / len) + cof[3 + k] * (n[1] / len) + cof[6 + k] * (n[2] / len)) * rdet * ds;
  if (act) {
    b->w[side][q][0] = raw_int2(w[d]);
    b->w[side][q][1] = raw_int2(w[d == 0 ? 1 : 0]);
    b->w[side][q][2] = raw_int2(w[d == 2 ? 1 : 2]);
    if (side == 0) b->ds[q] = raw_int2(ds);
  }
  const double ar = low_lanes_sum<NQF>(lane < NQF ? ds : 0.0);
  if (lane == 0) b->pen = fp.gamma / ar;
}

// Point data of facet id for the fixed-point products (all 32 lanes of the
// point warp): the geometry of facet_points, the weights dS cof^T n / det as
// integers under one scale per side and kind of axis, dS under one, and each
// point's index in the sides' own face rules.
template <int P>
__device__ __forceinline__ void facet_points_fixed(const FacetParams& fp, int64_t id, typename FixedFacetLayout<P>::Points* b,
                                                   double* aco, int lane) {
  using L = FixedFacetLayout<P>;
  constexpr int N1 = L::N1, NB = L::NB, NQF = L::NQF;
  static_assert(2 * NQF <= 32, "one lane per (side, point)");
  const FacetRef f = facet_ref(fp, id);
  if (lane < 3 * f.ns) trilinear_coefficients(fp.xv + f.cell[lane / 3] * 24, lane % 3, aco + (lane / 3) * 21);
  if (f.interior && lane >= 30)
    facet_out<NB>(fp, lane == 31 ? f.cell[1] : f.cell[0], lane == 31 ? f.face[1] : f.face[0], lane - 30, &b->out);
  __syncwarp();
  const bool act = lane < f.ns * NQF;
  const int side = act ? lane / NQF : 0, q = lane % NQF, qs = q % N1, qt = q / N1;
  const int d = side ? f.face[1] / 2 : f.face[0] / 2;
  double xh[3];
  int at[3];
  face_point<P>(fp, f, side, qs, qt, xh, at);
  double cof[9], det;
  facet_geometry(aco + side * 21, xh[0], xh[1], xh[2], cof, &det);
  if (act && !(det > 0.0)) atomicOr(fp.err, kErrNegJacobian);
  const int dp = f.face[0] / 2;
  const bool low = f.face[0] % 2 == 0;
  double nd[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    nd[k] = (dp == 0 ? cof[3 * k] : (dp == 1 ? cof[3 * k + 1] : cof[3 * k + 2]));
    nd[k] = __shfl_sync(kFull, flip(nd[k], low), q);
  }
  const double l2 = nd[0] * nd[0] + nd[1] * nd[1] + nd[2] * nd[2];
  const double rl = rsqrt_fast(l2), gww = fp.gw[qs] * fp.gw[qt];
  const double dsq = l2 * rl * gww;
  const double ar = low_lanes_sum<NQF>(lane < NQF ? dsq : 0.0);
  // dS n = gww nd: w_k = (cof^T nd)_k gww / det
  const double sc = gww * reciprocal(det);
  double w[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) w[k] = (cof[k] * nd[0] + cof[3 + k] * nd[1] + cof[6 + k] * nd[2]) * sc;
  const double wn = d == 0 ? w[0] : d == 1 ? w[1] : w[2];
  const double ws = d == 0 ? w[1] : w[0], wt = d == 2 ? w[1] : w[2];
  auto top = [](double x) { return __double2hiint(x) & 0x7fffffff; };
  // one scale per side and kind of axis: the weights go with 1 / (the cell's
  // extent along the axis), which may differ by any factor between the two
  // cells, and the rows of a cell's nodes off the face hold nothing of the other
  int ew[2][2];
  bool odd = false;
#pragma unroll
  for (int sd = 0; sd < 2; ++sd) {
    const bool mine = act && side == sd;
    const int mn = __reduce_max_sync(kFull, mine ? top(wn) : 0) >> 20;
    const int mt = __reduce_max_sync(kFull, mine ? max(top(ws), top(wt)) : 0) >> 20;
    ew[sd][0] = mn - 1022;
    // (the tangential terms add to the normal ones: below 2^-400 of those they are nothing)
    ew[sd][1] = max(mt - 1022, max(mn - 1422, 150 - 1022));
    odd |= sd < f.ns && (mn < 150 || mn > 1900 || mt > 1900);
  }
  const int my = __reduce_max_sync(kFull, act ? top(dsq) : 0) >> 20;
  const int ey = my - 1022;
  odd |= my < 150 || my > 1900;
  if (act) {
    const int en = side ? ew[1][0] : ew[0][0], et = side ? ew[1][1] : ew[0][1];
    b->w[side][q][0] = fix_limbs<30>(fix_quantise(wn, 60 - en));
    b->w[side][q][1] = fix_limbs<30>(fix_quantise(ws, 60 - et));
    b->w[side][q][2] = fix_limbs<30>(fix_quantise(wt, 60 - et));
    if (side == 0) b->ds[q] = fix_limbs<30>(fix_quantise(dsq, 60 - ey));
    b->perm[side][q] = d == 0 ? at[1] + N1 * at[2] : d == 1 ? at[0] + N1 * at[2] : at[0] + N1 * at[1];
  }
  const double pen = fp.gamma * reciprocal(ar);
  if (lane == 0) {
    b->pen = pen;
#pragma unroll
    for (int k = 0; k < 4; ++k) b->ew[k >> 1][k & 1] = ew[k >> 1][k & 1];
    b->ey = ey;
    b->odd = odd;
  }
}

// The block's facets that are out of the fixed-point range, in plain FP64 with the
// same steps as k_dg_facets_fixed, one facet at a time by all threads of the block.
template <int P>
static __device__ __noinline__ void odd_facets(const FacetParams& fp, unsigned char* sm, double* aco) {
  using L = FixedFacetLayout<P>;
  constexpr int N1 = L::N1, NB = L::NB, NQF = L::NQF, NBF = L::NBF;
  auto* pt = reinterpret_cast<typename L::Points*>(sm + L::PT);
  const int2* tab = reinterpret_cast<const int2*>(sm + L::TAB);
  double* R = reinterpret_cast<double*>(sm + L::R);
  double* X = reinterpret_cast<double*>(sm + L::X);
  double* Y = reinterpret_cast<double*>(sm + L::Y);
  double* XB = reinterpret_cast<double*>(sm + L::XB);
  const double* Dn = reinterpret_cast<const double*>(sm + L::DN);
  const uint8_t* nodes = sm + L::NODES;
  const int t = threadIdx.x, nt = blockDim.x, lp = fp.fix_lp, ld = fp.fix_ld;
  auto value = [](int2 l, int scale) { return scalbn(double((int64_t(l.x) << 30) + l.y), -scale); };
  for (int64_t id = blockIdx.x; id < fp.n_int + fp.n_bnd; id += gridDim.x) {
    if (t < 32) facet_points_fixed<P>(fp, id, pt, aco, t);
    __syncthreads();
    if (pt->odd) {
      const FacetRef f = facet_ref(fp, id);
      const int ns = f.ns, side_bit[2] = {f.face[0] % 2, f.face[1] % 2};
      if (t < 32) facet_weights_fp64<P>(fp, f, pt, t);
      __syncthreads();
      for (int i = t; i < ns * NQF * NBF; i += nt) {
        const int c = i % NBF, sq = i / NBF, side = sq / NQF, q = sq % NQF;
        const int2* row = tab + NQF * NBF + pt->perm[side][q] * NBF + c;
        const double ph = value(row[0], 60 - lp), ps = value(row[NQF * NBF], 60 - ld), pq = value(row[2 * NQF * NBF], 60 - ld);
        R[i * 3] = raw_double(pt->w[side][q][0]) * ph;
        R[i * 3 + 1] = raw_double(pt->w[side][q][1]) * ps + raw_double(pt->w[side][q][2]) * pq;
        R[i * 3 + 2] = raw_double(pt->ds[q]) * ph;
      }
      __syncthreads();
      for (int i = t; i < ns * ns * NBF * NBF; i += nt) {
        const int c2 = i % NBF, rest = i / NBF, c = rest % NBF, blk = rest / NBF, sa = blk >> 1, sb = blk & 1;
        double s[3] = {0.0, 0.0, 0.0};
        for (int q = 0; q < NQF; ++q) {
          const double ph = value(tab[pt->perm[sa][q] * NBF + c], 59 - lp);
          const double* r = R + ((sb * NQF + q) * NBF + c2) * 3;
          for (int k = 0; k < 3; ++k) s[k] = fma(ph, r[k], s[k]);
        }
        const double half = (sa ? 1.0 : -1.0) * (f.interior ? 0.5 : 1.0);
        const int fs = side_bit[sb];
        double* x = X + (blk * NBF + c) * NB + c2;
        for (int m = 0; m < N1; ++m) x[m * NBF] = Dn[fs * N1 + m] * (half * s[0]);
        x[fs * P * NBF] += half * s[1];
        Y[i] = sa == sb ? s[2] : -s[2];
      }
      __syncthreads();
      for (int i = t; i < ns * ns * NBF * NBF; i += nt) {
        const int c2 = i % NBF, rest = i / NBF, c = rest % NBF, blk = rest / NBF, sa = blk >> 1, sb = blk & 1;
        XB[i] = pt->pen * Y[i] + (fp.tau * X[(((sb << 1) | sa) * NBF + c2) * NB + side_bit[sa] * P * NBF + c] +
                                  X[(blk * NBF + c) * NB + side_bit[sb] * P * NBF + c2]);
      }
      __syncthreads();
      for (int i = t; i < ns * ns * NB * NB; i += nt) {
        const int b = i % NB, a = (i / NB) % NB, blk = i / (NB * NB), sa = blk >> 1, sb = blk & 1;
        const int na = nodes[f.face[sa] * NB + a], nb = nodes[f.face[sb] * NB + b];
        const bool on_a = na >> 4 == side_bit[sa] * P, on_b = nb >> 4 == side_bit[sb] * P;
        const int ca = na & 15, cb = nb & 15;
        const double v = on_a && on_b ? XB[(blk * NBF + ca) * NBF + cb]
                         : on_a       ? X[(blk * NBF + ca) * NB + (nb >> 4) * NBF + cb]
                         : on_b       ? fp.tau * X[(((sb << 1) | sa) * NBF + cb) * NB + (na >> 4) * NBF + ca]
                                      : 0.0;
        double* out = sa != sb ? fp.values + pt->out.base[sa] + int64_t(a) * pt->out.len[sa]
                      : f.interior ? static_cast<double*>(fp.fblk) + (f.i * 2 + sa) * NB * NB + a * NB
                                   : static_cast<double*>(fp.bblk) + f.i * NB * NB + a * NB;
        out[b] = v;
      }
    }
    __syncthreads();
  }
}

// The facet kernel of the FP64 form: as k_dg_facets, with the products in
// fixed point (fe_fixed.cuh) and only over face nodes. The normal derivative of
// a shape function b = (layer m along the face's normal axis, face node c') at
// a face point is cn D_m phi_c' plus, on the face layer, the two tangential
// terms, with D_m the 1D derivative at the face: so
//   X_{sa,sb}[c][(m, c')] = D_m A[c][c'] + [face layer] B[c][c'],
//   A = sum_q phi_c dS cn phi_c',  B = sum_q phi_c dS (cs d_s + ct d_t) phi_c',
// and the values of phi and its tangential derivatives are those of one face
// rule, the points of the other side permuted (a face symmetry). Steps of the
// product warps (a facet whose weights leave 2^-872 .. 2^878, or are not finite, is
// left to odd_facets):
//   1. right-hand operands (side, point, face node): dS cn phi, dS (cs d_s phi +
//      ct d_t phi), dS phi as 59-bit integers;
//   2. per (block, c, c') the three sums over the points, each converted to a
//      double once; the X rows of every layer, gamma/|F| Y;
//   3. the entries between face nodes: X + tau X^T + gamma/|F| Y;
//   4. the blocks, row (block, a), column b.
// Against FP64 multiply-adds over all nb columns (18,800 per interior facet at
// p = 2 on a pipe of 2 lanes per clock per SM) 6.0 -> 1.37 ms on 32^3 Q2 cells;
// bound by the FP64 pipe (62 %: the point data, about 90 operations per facet,
// and step 2's products with D_m) and issue (55 %).
// Blocks per SM: p = 1 as many as 64 registers let in (assembly of 40^3 cells 1.84
// ms with 8, 1.94 with 7, 2.30 with 5), p = 2 seven of 72 registers (32^3 cells 2.64
// ms, 2.69 with 8, 2.68 with 6), p = 3 the three that fit the shared memory.
template <int P>
__global__ void __launch_bounds__(128, P == 1 ? 8 : P == 2 ? 7 : 3) k_dg_facets_fixed(const __grid_constant__ FacetParams fp) {
  using L = FixedFacetLayout<P>;
  constexpr int N1 = L::N1, NB = L::NB, NQF = L::NQF, NBF = L::NBF, NT = 96;
  constexpr int NW = 3, NBJ = (NB + 31) / 32;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ double aco[42];
  __shared__ int any_odd;
  using Points = typename L::Points;
  constexpr size_t PTB = (sizeof(Points) + 15) & ~size_t(15);
  int2* tab = reinterpret_cast<int2*>(sm + L::TAB);  // 59-bit phi; 60-bit phi, d_s phi, d_t phi
  int2* R = reinterpret_cast<int2*>(sm + L::R);
  double* X = reinterpret_cast<double*>(sm + L::X);
  double* Y = reinterpret_cast<double*>(sm + L::Y);
  double* XB = reinterpret_cast<double*>(sm + L::XB);
  double* Dn = reinterpret_cast<double*>(sm + L::DN);
  uint8_t* nodes = sm + L::NODES;
  const int warp = ((threadIdx.x >> 5) + blockIdx.x) & 3, lane = threadIdx.x & 31, t = warp * 32 + lane;
  const int64_t n_fac = fp.n_int + fp.n_bnd;
  const double tau = fp.tau;
  const bool symmetric = __double_as_longlong(tau) == 0x3ff0000000000000ll;  // tau == 1
  for (int i = threadIdx.x; i < 4 * NQF * NBF; i += 128) tab[i] = fp.fix[i];
  if (threadIdx.x == 0) any_odd = 0;
  for (int i = threadIdx.x; i < 2 * N1; i += 128) Dn[i] = fp.fix_dn[i];
  for (int i = threadIdx.x; i < 6 * NB; i += 128) nodes[i] = face_node<N1>(i / NB, i % NB);
  if (warp == 3 && blockIdx.x < n_fac)
    facet_points_fixed<P>(fp, blockIdx.x, reinterpret_cast<Points*>(sm + L::PT), aco, lane);
  __syncthreads();
  int buf = 0;
  for (int64_t id = blockIdx.x; id < n_fac; id += gridDim.x, buf ^= 1) {
    if (warp == 3) {
      const int64_t nx = id + gridDim.x;
      if (nx < n_fac) facet_points_fixed<P>(fp, nx, reinterpret_cast<Points*>(sm + L::PT + (buf ^ 1) * PTB), aco, lane);
    } else {
      const Points* pt = reinterpret_cast<const Points*>(sm + L::PT + buf * PTB);
      const FacetRef f = facet_ref(fp, id);
      const bool odd = pt->odd;
      if (odd && t == 0) any_odd = 1;
      const int ns = odd ? 0 : f.ns;  // (0: nothing to do here, the facet is left to odd_facets)
      // 1. right-hand operands
      for (int i = t; i < ns * NQF * NBF; i += NT) {
        const int c = i % NBF, sq = i / NBF, side = sq / NQF, q = sq % NQF;
        const int2* row = tab + NQF * NBF + pt->perm[side][q] * NBF + c;
        const int2 ph = row[0], ps = row[NQF * NBF], pq = row[2 * NQF * NBF];
        FixAcc<30> a, b, y;
        a.zero();
        b.zero();
        y.zero();
        a.add(pt->w[side][q][0], ph);
        b.add(pt->w[side][q][1], ps);
        b.add(pt->w[side][q][2], pq);
        y.add(pt->ds[q], ph);
        R[i * 3] = fix_limbs<30>(a.get_shifted(1));
        R[i * 3 + 1] = fix_limbs<30>(b.get_shifted(1));
        R[i * 3 + 2] = fix_limbs<30>(y.get_shifted(1));
      }
      product_barrier();
      // 2. the sums over the points
      for (int i = t; i < ns * ns * NBF * NBF; i += NT) {
        const int c2 = i % NBF, rest = i / NBF, c = rest % NBF, blk = rest / NBF, sa = blk >> 1, sb = blk & 1;
        FixAcc<30> a, b, y;
        a.zero();
        b.zero();
        y.zero();
#pragma unroll
        for (int q = 0; q < NQF; ++q) {
          const int2 l = tab[pt->perm[sa][q] * NBF + c];
          const int2* r = R + ((sb * NQF + q) * NBF + c2) * 3;
          a.add(l, r[0]);
          b.add(l, r[1]);
          y.add(l, r[2]);
          if (q == 8) a.drain(), b.drain(), y.drain();
        }
        a.drain();
        b.drain();
        y.drain();
        const int ga = fix_shift(a.magnitude()), gb = fix_shift(b.magnitude()), gy = fix_shift(y.magnitude());
        // X scaled by -s_a / 2 (boundary: -1), Y by s_a s_b
        const int h = f.interior ? 1 : 0;
        const int64_t ia = a.get(ga), ib = b.get(gb), iy = y.get(gy);
        const double A = fix_to_double(sa ? ia : -ia, fix_exponent(pt->ew[sb][0] + 2 * fp.fix_lp - 56 - ga - h));
        const double Bt = fix_to_double(sa ? ib : -ib, fix_exponent(pt->ew[sb][1] + fp.fix_lp + fp.fix_ld - 56 - gb - h));
        const double Yv = fix_to_double(sa == sb ? iy : -iy, fix_exponent(pt->ey + 2 * fp.fix_lp - 56 - gy));
        const int fs = sb ? f.face[1] % 2 : f.face[0] % 2;  // the face layer of side sb
        double* x = X + (blk * NBF + c) * NB + c2;
#pragma unroll
        for (int m = 0; m < N1; ++m) x[m * NBF] = Dn[fs * N1 + m] * A;
        x[fs * P * NBF] = fma(Dn[fs * N1 + fs * P], A, Bt);
        Y[i] = Yv;
      }
      product_barrier();
      // 3. entries between face nodes
      const double pen = pt->pen;
      for (int i = t; i < ns * ns * NBF * NBF; i += NT) {
        const int c2 = i % NBF, rest = i / NBF, c = rest % NBF, blk = rest / NBF, sa = blk >> 1, sb = blk & 1;
        const int la = (sa ? f.face[1] % 2 : f.face[0] % 2) * P, lb = (sb ? f.face[1] % 2 : f.face[0] % 2) * P;
        XB[i] = fma(pen, Y[i], fma(tau, X[(((sb << 1) | sa) * NBF + c2) * NB + la * NBF + c], X[(blk * NBF + c) * NB + lb * NBF + c2]));
      }
      product_barrier();
      // 4. the blocks: warp w takes rows a = w, w + 3, ...
      for (int blk = 0; blk < ns * ns; ++blk) {
        const int sa = blk >> 1, sb = blk & 1;
        const int fa = sa ? f.face[1] : f.face[0], fb = sb ? f.face[1] : f.face[0];
        double* out = sa != sb ? fp.values + pt->out.base[sa]
                      : f.interior ? static_cast<double*>(fp.fblk) + (f.i * 2 + sa) * NB * NB
                                   : static_cast<double*>(fp.bblk) + f.i * NB * NB;
        const int len = sa != sb ? pt->out.len[sa] : NB;
        out += int64_t(warp) * len + lane;
        // the lane's columns: X entries of rows on the face (XB where the column
        // is on the face too), transposed X entries of the other rows
        const double *on[NBJ], *off[NBJ];
        int stride[NBJ];
        bool bon[NBJ];
#pragma unroll
        for (int j = 0; j < NBJ; ++j) {
          const int node = lane + 32 * j < NB ? int(nodes[fb * NB + lane + 32 * j]) : 0;
          const int cb = node & 15, mb = node >> 4;
          bon[j] = mb == (fb & 1) * P;
          on[j] = bon[j] ? XB + blk * NBF * NBF + cb : X + blk * NBF * NB + mb * NBF + cb;
          stride[j] = bon[j] ? NBF : NB;
          off[j] = X + (((sb << 1) | sa) * NBF + cb) * NB;
        }
        auto rows = [&](auto unit) {
#pragma unroll 3
          for (int a = warp; a < NB; a += NW, out += NW * len) {
            const int node = nodes[fa * NB + a], ca = node & 15, ma = node >> 4;
            const bool face_row = ma == (fa & 1) * P;
#pragma unroll
            for (int j = 0; j < NBJ; ++j) {
              const double* src = face_row ? on[j] + ca * stride[j] : off[j] + ma * NBF + ca;
              double v = face_row || bon[j] ? *src : 0.0;
              if (!decltype(unit)::value && !face_row && bon[j]) v *= tau;
              if (NB % 32 == 0 || lane + 32 * j < NB) out[32 * j] = v;
            }
          }
        };
        // (an FP64 multiply costs a warp 64 clocks of its FP64 pipe, predicated off or not)
        if (symmetric) rows(std::true_type()); else rows(std::false_type());
      }
    }
    __syncthreads();
  }
  if (any_odd) odd_facets<P>(fp, sm, aco);  // (after the loop: a call among its steps costs them registers)
}

}  // namespace dg
}  // namespace feasm

namespace feasm {
namespace dg {

struct RowParams {
  int64_t n_cells;
  int nb, nlp;
  const void* ke;  // cell matrices [cells][nb][nlp], T
  const double* fe;
  const int32_t* face_code;
  const uint8_t* slots;
  const uint8_t* nslot;
  const int64_t* row_ptr;
  const void* fblk;  // facet blocks in T (the facet kernel's storage type)
  const void* bblk;
  double* values;
  double* rhs;
};

// One block per cell: the diagonal block of its block row, the cell matrix
// plus the diagonal blocks of the cell's six facets in face order (the other
// blocks are the facet kernel's). T is the storage of the cell and facet
// blocks: FP64, or FP32, whose seven terms are summed as an FP32 pair (TwoSum)
// and rounded once to FP64. The block locations are resolved once per cell
// into shared memory.
template <int NB, typename T>
__global__ void __launch_bounds__(256) k_dg_rows(RowParams rp) {
  constexpr bool F32 = std::is_same<T, float>::value;
  const T* ke = static_cast<const T*>(rp.ke);
  const T* fblk = static_cast<const T*>(rp.fblk);
  const T* bblk = static_cast<const T*>(rp.bblk);
  __shared__ const T* s_diag[6];
  __shared__ int64_t s_base;
  __shared__ int s_len;
  const int t = threadIdx.x;
  for (int64_t e = blockIdx.x; e < rp.n_cells; e += gridDim.x) {
    if (t < 6) {
      const int32_t code = rp.face_code[e * 6 + t];
      s_diag[t] = code >= 0 ? fblk + (int64_t(code >> 1) * 2 + (code & 1)) * NB * NB : bblk + int64_t(-1 - code) * NB * NB;
    } else if (t == 32) {
      const int ns = rp.nslot[e];
      int j = 0;
      while (j < ns - 1 && rp.slots[e * 7 + j] != kSelf) ++j;
      s_len = ns * NB;
      s_base = rp.row_ptr[e * NB] + int64_t(j) * NB;
    }
    __syncthreads();
    for (int ab = t; ab < NB * NB; ab += blockDim.x) {
      const int a = ab / NB, b = ab % NB;
      T x[6];
#pragma unroll
      for (int f = 0; f < 6; ++f) x[f] = s_diag[f][ab];
      T hi = ke[(e * NB + a) * int64_t(rp.nlp) + b], lo = T(0);
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        if constexpr (F32) {
          const T sum = hi + x[f], bp = sum - hi;
          lo += (hi - (sum - bp)) + (x[f] - bp);
          hi = sum;
        } else {
          hi += x[f];
        }
      }
      double v;
      if constexpr (F32) v = to_f64(hi) + to_f64(lo); else v = hi;
      rp.values[s_base + int64_t(a) * s_len + b] = v;
    }
    if (rp.rhs)
      for (int a = t; a < NB; a += blockDim.x) rp.rhs[e * NB + a] = rp.fe[e * NB + a];
    __syncthreads();
  }
}

template <int P>
cudaError_t launch(const fe_dg* g, double tau, double gamma, double* values, double* rhs, fe_precision prec,
                   const double* gx, const double* gw, cudaStream_t st) {
  constexpr int NB = (P + 1) * (P + 1) * (P + 1);
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, g->s->device);
  FacetParams fp;
  fp.n_int = int64_t(g->fplus.size());
  fp.n_bnd = int64_t(g->bcell.size());
  fp.xv = g->s->d_xv;
  fp.fplus = g->d_fplus;
  fp.fminus = g->d_fminus;
  fp.fpf = g->d_fpf;
  fp.fmf = g->d_fmf;
  fp.fcorner = g->d_fcorner;
  fp.bcell = g->d_bcell;
  fp.bface = g->d_bface;
  fp.gx = gx;
  fp.gw = gw;
  fp.tau = tau;
  fp.gamma = gamma;
  fp.fblk = g->d_fblk;
  fp.bblk = g->d_bblk;
  fp.values = values;
  fp.slots = g->d_slots;
  fp.nslot = g->d_nslot;
  fp.row_ptr = g->d_row_ptr;
  fp.fix = reinterpret_cast<const int2*>(g->d_fix);
  fp.fix_dn = g->d_fix_dn;
  fp.fix_lp = g->fix_lp;
  fp.fix_ld = g->fix_ld;
  fp.err = g->s->d_err;
  const int64_t nf = fp.n_int + fp.n_bnd;
  // a persistent grid of the resident blocks (one wave; facets cost alike)
  auto facets = [&](auto kern, size_t smem) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    int per_sm = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, smem);
    if (e != cudaSuccess) return e;
    const int fblocks = int(std::min<int64_t>(nf, int64_t(nsm) * std::max(per_sm, 1)));
    kern<<<fblocks, 128, smem, st>>>(fp);
    return cudaSuccess;
  };
  if (nf > 0) {
    const cudaError_t e = prec == FE_PREC_FP64 ? facets(k_dg_facets_fixed<P>, FixedFacetLayout<P>::BYTES)
                                               : facets(k_dg_facets<P>, FacetLayout<P>::BYTES);
    if (e != cudaSuccess) return e;
  }
  RowParams rp;
  rp.n_cells = g->n_cells;
  rp.nb = NB;
  rp.nlp = g->s->nlp;
  rp.ke = g->s->d_ke;
  rp.fe = g->s->d_fe;
  rp.face_code = g->d_face_code;
  rp.slots = g->d_slots;
  rp.nslot = g->d_nslot;
  rp.row_ptr = g->d_row_ptr;
  rp.fblk = g->d_fblk;
  rp.bblk = g->d_bblk;
  rp.values = values;
  rp.rhs = rhs;
  const int blocks = int(std::min<int64_t>(g->n_cells, int64_t(nsm) * 8));
  if (prec == FE_PREC_FP64)
    k_dg_rows<NB, double><<<blocks, 256, 0, st>>>(rp);
  else
    k_dg_rows<NB, float><<<blocks, 256, 0, st>>>(rp);
  return cudaGetLastError();
}

}  // namespace dg
}  // namespace feasm

namespace {

template <typename T>
cudaError_t upload_vec(T** dst, const std::vector<T>& src) {
  *dst = nullptr;
  if (src.empty()) return cudaSuccess;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(dst), src.size() * sizeof(T));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
}

// Tables of the FP64 facet kernel: the shape functions of the face nodes at the
// face rule's points, phi 2^(59 - lp) and phi 2^(60 - lp), and their derivatives
// along the face's two axes 2^(60 - ld), as limb pairs [4][point][node]; the 1D
// derivatives at 0 and 1.
struct FacetTables {
  int lp = 0, ld = 0;
  std::vector<int32_t> limbs;
  std::vector<double> dn;
};

FacetTables facet_tables(int p) {
  const int n1 = p + 1, n = n1 * n1;
  std::vector<double> v(size_t(n1) * n1), d(v.size());
  feasm::lagrange_1d_table(p, n1, v.data(), d.data());
  std::vector<long double> t[3];  // phi, d_s phi, d_t phi: [point][node]
  for (int q = 0; q < n; ++q)
    for (int c = 0; c < n; ++c) {
      const int qs = q % n1, qt = q / n1, cs = c % n1, ct = c / n1;
      const long double vs = v[qs * n1 + cs], vt = v[qt * n1 + ct];
      t[0].push_back(vs * vt);
      t[1].push_back((long double)d[qs * n1 + cs] * vt);
      t[2].push_back(vs * d[qt * n1 + ct]);
    }
  FacetTables ft;
  long double mp = 0, md = 0;
  for (int i = 0; i < n * n; ++i) {
    mp = std::max(mp, std::fabs(t[0][i]));
    md = std::max(md, std::fabs(t[1][i]) + std::fabs(t[2][i]));
  }
  std::frexp(1.02l * mp, &ft.lp);
  std::frexp(1.02l * md, &ft.ld);
  auto put = [&](const std::vector<long double>& x, int scale) {
    for (long double y : x) {
      const int64_t u = std::llrint(std::ldexp(y, scale)), h = (u + (int64_t(1) << 29)) >> 30;
      ft.limbs.push_back(int32_t(h));
      ft.limbs.push_back(int32_t(u - (h << 30)));
    }
  };
  put(t[0], 59 - ft.lp);
  put(t[0], 60 - ft.lp);
  put(t[1], 60 - ft.ld);
  put(t[2], 60 - ft.ld);
  for (int x = 0; x < 2; ++x)
    for (int m = 0; m < n1; ++m) {
      // derivative of the m-th Lagrange polynomial on the nodes j / p at x
      long double sum = 0;
      for (int j = 0; j < n1; ++j) {
        if (j == m) continue;
        long double z = (long double)p / (m - j);
        for (int k = 0; k < n1; ++k)
          if (k != m && k != j) z *= ((long double)(x * p - k)) / (m - k);
        sum += z;
      }
      ft.dn.push_back(double(sum));
    }
  return ft;
}

void free_dg(fe_dg* g) {
  void* ptrs[] = {g->d_fplus, g->d_fminus, g->d_fpf, g->d_fmf, g->d_fcorner, g->d_bcell, g->d_bface, g->d_face_code,
                  g->d_slots, g->d_nslot, g->d_row_ptr, g->d_col, g->d_ones, g->d_fblk, g->d_bblk, g->d_gx, g->d_gw,
                  g->d_fix, g->d_fix_dn};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (g->s) fe_space_destroy(g->s);
}

int dg_create(const fe_mesh_desc* mesh, int order, bool host_only, fe_dg** out) {
  if (!out) return feasm::set_error(FE_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (order < 1 || order > 3) return feasm::set_error(FE_ERR_INVALID_ARG, "order must be 1..3");
  fe_dg* g = new (std::nothrow) fe_dg();
  if (!g) return feasm::set_error(FE_ERR_OOM, "host allocation failed");
  int rc = host_only ? fe_space_create_host(mesh, order, 0, FE_POISSON, 0.0, &g->s)
                     : fe_space_create(mesh, order, 0, FE_POISSON, 0.0, &g->s);
  if (rc) {
    delete g;
    return rc;
  }
  g->p = order;
  g->nb = (order + 1) * (order + 1) * (order + 1);
  g->n_cells = mesh->n_cells;
  g->n_dofs = mesh->n_cells * g->nb;
  g->host_only = host_only;
  if (g->n_dofs > INT32_MAX) {
    fe_space_destroy(g->s);
    delete g;
    return feasm::set_error(FE_ERR_UNSUPPORTED, "more than 2^31-1 DG DOFs");
  }
  std::string err;
  try {
    rc = setup_dg(g, mesh, &err);
  } catch (const std::bad_alloc&) {
    rc = FE_ERR_OOM;
    err = "host allocation failed during DG setup";
  }
  if (rc) {
    fe_space_destroy(g->s);
    delete g;
    return feasm::set_error(rc, err.c_str());
  }
  if (!host_only) {
    std::vector<double> gx(order + 1), gw(order + 1), ones(std::max<int64_t>(1, g->n_cells), 1.0);
    feasm::gauss_rule(order + 1, gx.data(), gw.data());
    const size_t nbb = size_t(g->nb) * g->nb;
    cudaError_t e = upload_vec(&g->d_fplus, g->fplus);
    if (e == cudaSuccess) e = upload_vec(&g->d_fminus, g->fminus);
    if (e == cudaSuccess) e = upload_vec(&g->d_fpf, g->fpf);
    if (e == cudaSuccess) e = upload_vec(&g->d_fmf, g->fmf);
    if (e == cudaSuccess) e = upload_vec(&g->d_fcorner, g->fcorner);
    if (e == cudaSuccess) e = upload_vec(&g->d_bcell, g->bcell);
    if (e == cudaSuccess) e = upload_vec(&g->d_bface, g->bface);
    if (e == cudaSuccess) e = upload_vec(&g->d_face_code, g->face_code);
    if (e == cudaSuccess) e = upload_vec(&g->d_slots, g->slots);
    if (e == cudaSuccess) e = upload_vec(&g->d_nslot, g->nslot);
    if (e == cudaSuccess) e = upload_vec(&g->d_row_ptr, g->row_ptr);
    if (e == cudaSuccess) e = upload_vec(&g->d_col, g->col);
    if (e == cudaSuccess) e = upload_vec(&g->d_ones, ones);
    if (e == cudaSuccess) e = upload_vec(&g->d_gx, gx);
    if (e == cudaSuccess) e = upload_vec(&g->d_gw, gw);
    const FacetTables ft = facet_tables(order);
    g->fix_lp = ft.lp;
    g->fix_ld = ft.ld;
    if (e == cudaSuccess) e = upload_vec(&g->d_fix, ft.limbs);
    if (e == cudaSuccess) e = upload_vec(&g->d_fix_dn, ft.dn);
    if (e == cudaSuccess && !g->fplus.empty())
      e = cudaMalloc(&g->d_fblk, g->fplus.size() * 2 * nbb * sizeof(double));
    if (e == cudaSuccess && !g->bcell.empty()) e = cudaMalloc(&g->d_bblk, g->bcell.size() * nbb * sizeof(double));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
      free_dg(g);
      delete g;
      return feasm::set_error(e == cudaErrorMemoryAllocation ? FE_ERR_OOM : FE_ERR_CUDA, cudaGetErrorString(e));
    }
    std::vector<int32_t>().swap(g->col);  // kept on the device only
  }
  *out = g;
  return FE_OK;
}

}  // namespace

extern "C" {

int fe_dg_create(const fe_mesh_desc* mesh, int order, fe_dg** out) {
  return feasm::no_throw("fe_dg_create", [&] { return dg_create(mesh, order, false, out); });
}
int fe_dg_create_host(const fe_mesh_desc* mesh, int order, fe_dg** out) {
  return feasm::no_throw("fe_dg_create_host", [&] { return dg_create(mesh, order, true, out); });
}

int fe_dg_sizes(const fe_dg* g, int64_t* n_dofs, int64_t* nnz, int64_t* n_interior, int64_t* n_boundary) {
  if (!g) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL argument");
  if (n_dofs) *n_dofs = g->n_dofs;
  if (nnz) *nnz = g->nnz;
  if (n_interior) *n_interior = int64_t(g->fplus.size());
  if (n_boundary) *n_boundary = int64_t(g->bcell.size());
  return FE_OK;
}

int fe_dg_csr_pattern_host(const fe_dg* g, int64_t* row_ptr, int32_t* col_idx) {
  if (!g || !row_ptr || (!col_idx && g->nnz)) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL argument");
  if (!g->host_only) return feasm::set_error(FE_ERR_INVALID_ARG, "the pattern is kept on the host for host-only DG spaces; use fe_dg_csr_pattern");
  std::memcpy(row_ptr, g->row_ptr.data(), g->row_ptr.size() * sizeof(int64_t));
  if (g->nnz) std::memcpy(col_idx, g->col.data(), g->col.size() * sizeof(int32_t));
  return FE_OK;
}

int fe_dg_csr_pattern(const fe_dg* g, int64_t* row_ptr, int32_t* col_idx, void* stream) {
  if (!g || !row_ptr || (!col_idx && g->nnz)) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL argument");
  if (g->host_only) return feasm::set_error(FE_ERR_INVALID_ARG, "host-only DG space");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(row_ptr, g->d_row_ptr, (g->n_dofs + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && g->nnz)
    e = cudaMemcpyAsync(col_idx, g->d_col, g->nnz * sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
  return e == cudaSuccess ? FE_OK : feasm::set_error(FE_ERR_CUDA, cudaGetErrorString(e));
}

int fe_dg_facets_host(const fe_dg* g, int32_t* plus, int32_t* minus, uint8_t* plus_face, uint8_t* minus_face,
                      int32_t* bnd_cell, uint8_t* bnd_face) {
  if (!g) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL argument");
  const size_t ni = g->fplus.size(), nbd = g->bcell.size();
  if (plus && ni) std::memcpy(plus, g->fplus.data(), ni * sizeof(int32_t));
  if (minus && ni) std::memcpy(minus, g->fminus.data(), ni * sizeof(int32_t));
  if (plus_face && ni) std::memcpy(plus_face, g->fpf.data(), ni);
  if (minus_face && ni) std::memcpy(minus_face, g->fmf.data(), ni);
  if (bnd_cell && nbd) std::memcpy(bnd_cell, g->bcell.data(), nbd * sizeof(int32_t));
  if (bnd_face && nbd) std::memcpy(bnd_face, g->bface.data(), nbd);
  return FE_OK;
}

int fe_dg_assemble(fe_dg* g, double tau, double gamma, double source, double* csr_values, double* rhs,
                   fe_precision prec, void* stream) {
  if (!g) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL argument");
  if (g->host_only) return feasm::set_error(FE_ERR_INVALID_ARG, "host-only DG space cannot compute");
  if (prec != FE_PREC_FP64 && prec != FE_PREC_FP32 && prec != FE_PREC_BF16)
    return feasm::set_error(FE_ERR_INVALID_ARG, "unknown precision");
  if (g->nnz && !csr_values) return feasm::set_error(FE_ERR_INVALID_ARG, "NULL csr_values");
  if (!(gamma > 0.0)) return feasm::set_error(FE_ERR_INVALID_ARG, "gamma must be positive");
  if (g->n_cells == 0) return FE_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const double f[3] = {source, 0.0, 0.0};
  if (int rc = feasm::cell_stage(g->s, g->d_ones, f, prec, st)) return rc;
  cudaError_t e;
  switch (g->p) {
    case 1: e = feasm::dg::launch<1>(g, tau, gamma, csr_values, rhs, prec, g->d_gx, g->d_gw, st); break;
    case 2: e = feasm::dg::launch<2>(g, tau, gamma, csr_values, rhs, prec, g->d_gx, g->d_gw, st); break;
    default: e = feasm::dg::launch<3>(g, tau, gamma, csr_values, rhs, prec, g->d_gx, g->d_gw, st); break;
  }
  return e == cudaSuccess ? FE_OK : feasm::set_error(FE_ERR_CUDA, cudaGetErrorString(e));
}

void fe_dg_destroy(fe_dg* g) {
  if (!g) return;
  if (g->host_only) {
    if (g->s) fe_space_destroy(g->s);
  } else {
    free_dg(g);
  }
  delete g;
}

}  // extern "C"
