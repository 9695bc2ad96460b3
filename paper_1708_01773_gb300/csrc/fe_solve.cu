// Self-adjoint compliance of a clamped structure (not in the paper; it uses
// the paper's assembly with strong Dirichlet conditions, Sect. "Strong
// imposition of boundary conditions"): K(E) u = f on the free DOFs, c = f^T u
// and dc/dE_K = -u_K^T (A^K / E_K) u_K. The free system is solved by the
// conjugate gradient method with the Jacobi preconditioner, in FP64, with
// every reduction in a fixed order (the result is deterministic on any GPU).
//
// The iterations run in one cooperative kernel (k_pcg), a block per SM, up to
// kChunk of them per launch. Per iteration three grid-wide exchanges:
//   q = A p, block partials of p.q               -> alpha
//   x += alpha p, r -= alpha q, z = D^-1 r;
//   partials of r.z and r.r                      -> beta, convergence
//   p = z + beta p                               -> every p in place
// A block's partial sums and its arrival are one store (see Exchange), so an
// exchange costs one trip through L2. As three kernels per iteration on a fixed
// grid of 1216 blocks, launched from the host with a look at the residual every
// 8 iterations, a small system spent most of its time in launches and in
// summing 1216 partials per block. Measured per iteration, us: 811,200 rows 230 ->
// 183 (FP64 pipe and HBM), 136,000 rows 77 -> 49, 41,000 rows 48 -> 23.4, 3,900 rows
// 43 -> 15 (latency of the exchanges and of dependent FP64 operations).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "fe_device.cuh"
#include "fe_launch.h"

namespace feasm {
namespace solve {

constexpr int kBlock = 256;
constexpr int kGridBlocks = 1216;  // elementwise grid (152 SMs x 8), fixed
constexpr int kCheckEvery = 8;     // iterations between convergence checks
constexpr int kChunk = 256;        // iterations per launch of k_pcg at most
// Partial sums of k_pcg: virtual blocks of kPcgThreads threads, at most one per
// SM on GB300 (a smaller grid loops over them), their number a function of the
// system's size alone, so that the sums and with them every result do not
// depend on the SM count (where every virtual block has an SM; fewer SMs take
// the form that keeps its vectors in memory, which sums in another order).
constexpr int kVirtual = 152;
constexpr int kPcgThreads = 1024;
constexpr long long kPcgWait = 1ll << 31;  // clock cycles before a wait gives up

// device scalars
enum { S_RZ = 0, S_IT = 1, S_RR = 2, S_BB = 3, S_FLAG = 4, kScalars = 8 };
// S_FLAG bits
constexpr int kFlagNotSpd = 1, kFlagTimeout = 2, kFlagDiverged = 4;

struct CgParams {
  int64_t n;
  const int64_t* row_ptr;
  const int32_t* col;
  const double* val;
  const double* b;
  double* x;
  double* r;
  double* z;
  double* p;
  double* q;
  double* dinv;
  double* part_a;  // [kGridBlocks] r.z at init
  double* part_b;  // exchange slots of k_pcg: [6][kVirtual][2], over part_c
  double* part_c;  // [kGridBlocks] b.b at init
  double* s;       // [kScalars]
};

// Fixed-order block reduction of one value per thread; the result is valid in
// thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(kFull, v, off);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kBlock / 32; ++w) t += sh[w];
  __syncthreads();
  return t;
}

// Sum of the kGridBlocks partials in a fixed order, by one warp (every lane
// ends with the same value).
__device__ __forceinline__ double sum_partials(const double* part) {
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int i = lane; i < kGridBlocks; i += 32) v += part[i];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

// x = 0, r = b, z = D^-1 b, p = z; partials of r.z and b.b. The diagonal of
// each row is found by binary search (columns ascending).
__global__ void __launch_bounds__(kBlock) k_cg_init(CgParams p) {
  __shared__ double sh[kBlock / 32];
  double rz = 0.0, bb = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * kBlock + threadIdx.x; i < p.n; i += int64_t(gridDim.x) * kBlock) {
    int64_t lo = p.row_ptr[i], hi = p.row_ptr[i + 1] - 1;
    double d = 0.0;
    while (lo <= hi) {
      const int64_t mid = (lo + hi) >> 1;
      const int64_t c = p.col[mid];
      if (c == i) { d = p.val[mid]; break; }
      if (c < i) lo = mid + 1; else hi = mid - 1;
    }
    if (!(d > 0.0)) atomicOr(reinterpret_cast<unsigned long long*>(p.s + S_FLAG), 0ull | kFlagNotSpd);
    const double di = d > 0.0 ? 1.0 / d : 0.0;
    const double bi = p.b[i];
    p.dinv[i] = di;
    p.x[i] = 0.0;
    p.r[i] = bi;
    p.z[i] = di * bi;
    p.p[i] = di * bi;
    rz += bi * (di * bi);
    bb += bi * bi;
  }
  const double a = block_sum(rz, sh);
  const double c = block_sum(bb, sh);
  if (threadIdx.x == 0) {
    p.part_a[blockIdx.x] = a;
    p.part_c[blockIdx.x] = c;
  }
}

// rz (buffer 0) and b.b from the init partials; one warp.
__global__ void k_cg_init_sums(CgParams p) {
  const double rz = sum_partials(p.part_a);
  const double bb = sum_partials(p.part_c);
  if (threadIdx.x == 0) {
    p.s[S_RZ] = rz;
    p.s[S_BB] = bb;
    p.s[S_RR] = bb;
  }
}

// Sums of two values over the lanes of a warp in a fixed order: a in lane 0, b
// in lane 16 (5 FP64 additions for both: each takes a warp 64 clocks).
__device__ __forceinline__ double pair_sum(double a, double b) {
  const bool up = (threadIdx.x & 16) != 0;
  const double give = up ? a : b, keep = up ? b : a;
  double v = keep + __shfl_xor_sync(kFull, give, 16);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  return v;
}

// Grid-wide exchange of up to two sums. Every virtual block has a slot of two
// doubles in each of kSets sets; a slot holds the sentinel (all bits set, a NaN
// no arithmetic produces) until its block stores its partial sums there, which
// is also its arrival. Warp 0 of every block waits for all slots (a 16-byte load
// each, all in flight) and adds them in the same fixed order. Sets rotate: a
// block empties its slot of the previous exchange once it has seen every slot
// of the current one, when all blocks are done with the previous.
// Only every third exchange publishes other data (p) and has the fences for it
// (PUBLISH; a fence costs a few thousand clocks): the sums travel in the slots
// themselves. A slot emptied at exchange t + 1 is used again at t + 6, with a
// fence of its block in between, so nobody can find the old sums there.
// Waits are bounded; a block whose wait runs out gives up, so do then the others.
struct Exchange {
  double* slots;
  int nv;  // virtual blocks in use
  int t = 0;
  bool gave_up = false;
  static constexpr unsigned long long kEmpty = ~0ull;
  static constexpr int PER = (kVirtual + 31) / 32;
  static constexpr int kSets = 6;

  __device__ __forceinline__ double* slot(int set, int vb) const { return slots + (set * kVirtual + vb) * 2; }
  // Thread 0 of the block: the partial sums of virtual block vb. PUBLISH: all
  // earlier writes of the block (before a __syncthreads) are visible to whoever
  // sees it in a finish of that kind.
  template <bool PUBLISH>
  __device__ __forceinline__ void put(int vb, double a, double b) {
    if (PUBLISH) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    asm volatile("st.volatile.global.v2.f64 [%0], {%1, %2};" ::"l"(slot(t % kSets, vb)), "d"(a), "d"(b) : "memory");
  }
  // All threads of the block, after put() for each of its virtual blocks.
  // step(a, b, out) turns the two sums into up to two values for all threads; it
  // runs in one thread (an FP64 division by every warp of the block would take
  // its FP64 pipes longer than the exchange).
  template <bool PUBLISH, typename Step>
  __device__ __forceinline__ void finish(double* out, double* sh, Step step) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      const long long t0 = clock64();
      unsigned long long v[PER][2];
      bool wait = true, bad = false;
      while (wait && !bad) {
        wait = false;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const int vb = lane + 32 * k;
          v[k][0] = v[k][1] = 0;
          if (vb < nv) asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(v[k][0]), "=l"(v[k][1]) : "l"(slot(t % kSets, vb)) : "memory");
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) wait |= v[k][0] == kEmpty || v[k][1] == kEmpty;
        bad = wait && clock64() - t0 > kPcgWait;
      }
      bad = __any_sync(kFull, bad);
      if (PUBLISH) asm volatile("fence.acq_rel.gpu;" ::: "memory");
      double a = 0.0, b = 0.0;
      if (!PUBLISH) {
        a = __longlong_as_double(static_cast<long long>(v[0][0]));
        b = __longlong_as_double(static_cast<long long>(v[0][1]));
#pragma unroll
        for (int k = 1; k < PER; ++k) {
          if (32 * k >= nv) break;
          a += __longlong_as_double(static_cast<long long>(v[k][0]));
          b += __longlong_as_double(static_cast<long long>(v[k][1]));
        }
        a = pair_sum(a, b);
        b = __shfl_sync(kFull, a, 16);
      }
      if (lane == 0) {
        step(a, b, sh);
        sh[2] = bad ? 1.0 : 0.0;
        for (int vb = blockIdx.x; vb < nv; vb += gridDim.x)
          asm volatile("st.volatile.global.v2.u64 [%0], {%1, %1};" ::"l"(slot((t + kSets - 1) % kSets, vb)), "l"(kEmpty) : "memory");
      }
    }
    __syncthreads();
    out[0] = sh[0];
    out[1] = sh[1];
    gave_up = sh[2] != 0.0;
    ++t;
  }
};

// (on the integer bits, off the FP64 pipe)
__device__ __forceinline__ bool is_finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// a / b from 1 / b; at the ends of the exponent range, where 1 / b overflows or
// loses bits (loads of the order of 1e-150), the division
static __device__ __noinline__ double quotient_slow(double a, double b) { return a / b; }
__device__ __forceinline__ double quotient(double a, double b, double inv_b) {
  const int eb = (__double2hiint(b) >> 20) & 0x7ff;
  return eb < 2 || eb > 2044 ? quotient_slow(a, b) : a * inv_b;
}

// Up to n_it PCG iterations (see the head of this file), ending early at a
// check (every kCheckEvery iterations) that finds ||r|| <= rtol ||b|| or a
// matrix that is not positive definite, and at once where p.q, r.z or r.r is not
// finite: such a sum does not recover, and no later residual may pass for a
// converged one. Cooperative launch: every block is resident. Virtual block vb
// owns rows [n vb / nv, n (vb + 1) / nv).
//
// GB300 issues FP64 at 2 lanes per clock per SM and charges a warp instruction
// in full (64 clocks of its sub-partition) whatever its active lanes; that
// shapes everything here:
//   SpMV       a group of G lanes takes one row (a warp 32 / G consecutive
//              rows), each lane summing every G-th nonzero, then a log2(G)-step
//              xor butterfly. G = 4 takes the 81 entries of an interior Q1
//              elasticity row in 21 rounds with 3 idle slots; G = 2 where that
//              lets a block's 257 to 512 rows run in one pass of its 32 warps
//              (Q1 elasticity, us per iteration with G = 2 / 4: 270 rows a block
//              23.4 / 24.8, 376 rows 26.7 / 26.7, 494 rows 29.2 / 28.9; Poisson,
//              323 rows 19.0 / 19.5); 8 for rows of more than 128 entries;
//   sums       the threads' values go through shared memory to one warp per sum
//              (butterflies in all 32 warps: 160 warp additions a sum);
//   scalars    alpha and beta in one thread.
// RES: at most one row per thread (n <= 152 x 1024): x, r, p and D^-1 of the row
// stay in the thread's registers from iteration to iteration, q in shared
// memory; only p goes to memory. 41,000 rows: 27 -> 23.4 us per iteration, of which the SpMV
// takes 13k of 49k clocks (11k at the FP64 pipe's rate) and the three exchanges
// 7k to 9k each (a store, its way through L2 to 152 pollers, nine dependent FP64
// additions).
template <int G, bool RES>
__global__ void __launch_bounds__(kPcgThreads, 1) k_pcg(CgParams p, int nv, int n_it, double rtol) {
  constexpr int RPW = 32 / G;  // rows per warp pass
  constexpr int U = 7;         // loads in flight per lane
  constexpr int W = kPcgThreads / 32;
  __shared__ double red[2][kPcgThreads];
  __shared__ double sq[RES ? kPcgThreads : 1];
  __shared__ double bc[3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = lane % G, slot = lane / G;
  Exchange x;
  x.slots = p.part_b;
  x.nv = nv;
  // (thread 0's copies are the ones that count)
  double rz = p.s[S_RZ], rr = 0.0;
  const double bb = p.s[S_BB];
  bool not_spd = false, diverged = false;
  auto row0 = [&](int vb) { return p.n * vb / nv; };
  // block sums of a and (TWO) b over the first `lim` threads (a multiple of 32)
  // in a fixed order, then the block's arrival
  auto block_put = [&](int vb, int lim, double a, double b, auto two) {
    constexpr bool TWO = decltype(two)::value;
    red[0][tid] = a;
    if (TWO) red[1][tid] = b;
    __syncthreads();
    if (warp < (TWO ? 2 : 1)) {
      double s0 = red[warp][lane], s1 = 0.0;
      for (int k = 32; k < lim; k += 64) {
        s1 += red[warp][lane + k];
        if (k + 32 < lim) s0 += red[warp][lane + k + 32];
      }
      s0 += s1;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s0 += __shfl_xor_sync(kFull, s0, off);
      if (TWO && warp == 1 && lane == 0) bc[1] = s0;
      a = s0;
    }
    if (TWO) __syncthreads();
    if (tid == 0) x.template put<false>(vb, a, TWO ? bc[1] : 0.0);
    if (vb + int(gridDim.x) < nv) __syncthreads();
  };
  const std::true_type two;
  const std::false_type one;
  // RES: this thread's row (one virtual block per block)
  const int64_t own0 = row0(blockIdx.x);
  const int own = int(row0(blockIdx.x + 1) - own0);
  const bool has = RES && tid < own;
  double xv = 0.0, rv = 0.0, pv = 0.0, di = 0.0;
  if (has) {
    xv = p.x[own0 + tid];
    rv = p.r[own0 + tid];
    pv = p.p[own0 + tid];
    di = p.dinv[own0 + tid];
  }
  double got[2];
  int it = 0;
  while (it < n_it) {
    for (int vb = blockIdx.x; vb < nv; vb += gridDim.x) {
      const int64_t r0 = row0(vb), r1 = row0(vb + 1);
      double pq = 0.0;
      for (int64_t base = r0 + warp * RPW; base < r1; base += W * RPW) {
        const int64_t i = base + slot;
        int64_t k0 = 0;
        int len = 0;
        if (i < r1) {
          k0 = p.row_ptr[i];
          len = int(p.row_ptr[i + 1] - k0);
        }
        const double* val = p.val + k0;
        const int32_t* col = p.col + k0;
        double acc = 0.0;
        for (int k = j; k < len; k += G * U) {
          double v[U];
          int c[U];
#pragma unroll
          for (int t = 0; t < U; ++t) {
            const int kk = k + t * G;
            v[t] = kk < len ? __ldg(val + kk) : 0.0;
            c[t] = kk < len ? __ldg(col + kk) : 0;
          }
          // past the row's end v = 0 and c = 0: the multiply-add adds an exact zero
#pragma unroll
          for (int t = 0; t < U; ++t) acc = fma(v[t], p.p[c[t]], acc);
        }
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(kFull, acc, off);
        if (j == 0 && i < r1) {
          if (RES) {
            sq[i - r0] = acc;
          } else {
            p.q[i] = acc;
            pq += p.p[i] * acc;
          }
        }
      }
      if (RES) {
        __syncthreads();
        block_put(vb, (own + 31) & ~31, has ? pv * sq[tid] : 0.0, 0.0, one);
      } else {
        block_put(vb, kPcgThreads, pq, 0.0, one);
      }
    }
    const double inv_rz = warp == 0 ? reciprocal(rz) : 0.0;  // (thread 0's, while the others arrive)
    x.template finish<false>(got, bc, [&](double pq, double, double* o) {
      not_spd |= !(pq > 0.0) && rz > 0.0;
      diverged |= !is_finite(pq);
      o[0] = pq > 0.0 ? quotient(rz, pq, reciprocal(pq)) : 0.0;
    });
    if (x.gave_up) break;
    const double alpha = got[0];
    double zv = 0.0;
    for (int vb = blockIdx.x; vb < nv; vb += gridDim.x) {
      double s_rz = 0.0, s_rr = 0.0;
      if (RES) {
        if (warp * 32 < own) {  // (whole warps: lanes past the end hold zeros)
          xv = fma(alpha, pv, xv);
          rv = fma(-alpha, has ? sq[tid] : 0.0, rv);
          zv = di * rv;
          s_rz = rv * zv;
          s_rr = rv * rv;
        }
        block_put(vb, (own + 31) & ~31, s_rz, s_rr, two);
      } else {
        const int64_t r1 = row0(vb + 1);
        for (int64_t i = row0(vb) + tid; i < r1; i += kPcgThreads) {
          p.x[i] = fma(alpha, p.p[i], p.x[i]);
          const double ri = fma(-alpha, p.q[i], p.r[i]);
          const double zi = p.dinv[i] * ri;
          p.r[i] = ri;
          p.z[i] = zi;
          s_rz += ri * zi;
          s_rr += ri * ri;
        }
        block_put(vb, kPcgThreads, s_rz, s_rr, two);
      }
    }
    ++it;
    x.template finish<false>(got, bc, [&](double rz_new, double rr_new, double* o) {
      o[0] = rz > 0.0 ? quotient(rz_new, rz, inv_rz) : 0.0;
      rz = rz_new;
      rr = rr_new;
      diverged |= !is_finite(rz) || !is_finite(rr);
      const bool check = it % kCheckEvery == 0 || it == n_it;
      o[1] = diverged || (check && (not_spd || !(sqrt(rr / bb) > rtol))) ? 1.0 : 0.0;
    });
    if (x.gave_up || got[1] != 0.0) break;
    const double beta = got[0];
    for (int vb = blockIdx.x; vb < nv; vb += gridDim.x) {
      if (RES) {
        if (warp * 32 < own) pv = fma(beta, pv, zv);
        if (has) p.p[own0 + tid] = pv;
      } else {
        const int64_t r1 = row0(vb + 1);
        for (int64_t i = row0(vb) + tid; i < r1; i += kPcgThreads) p.p[i] = fma(beta, p.p[i], p.z[i]);
      }
      __syncthreads();
      if (tid == 0) x.template put<true>(vb, 0.0, 0.0);
    }
    x.template finish<true>(got, bc, [](double, double, double*) {});
    if (x.gave_up) break;
  }
  if (has) {
    p.x[own0 + tid] = xv;
    p.r[own0 + tid] = rv;
  }
  if (blockIdx.x == 0 && tid == 0) {
    p.s[S_RZ] = rz;
    p.s[S_RR] = rr;
    p.s[S_IT] = double(it);
    const int flags = (not_spd ? kFlagNotSpd : 0) | (diverged ? kFlagDiverged : 0) | (x.gave_up ? kFlagTimeout : 0);
    if (flags)
      atomicOr(reinterpret_cast<unsigned long long*>(p.s + S_FLAG), static_cast<unsigned long long>(flags));
  }
}

// u[g] = x[label[g]] for free DOFs, 0 for fixed ones.
__global__ void __launch_bounds__(kBlock) k_expand(const int32_t* label, int64_t n_dofs, const double* x, double* u) {
  for (int64_t g = int64_t(blockIdx.x) * kBlock + threadIdx.x; g < n_dofs; g += int64_t(gridDim.x) * kBlock) {
    const int32_t l = label[g];
    u[g] = l >= 0 ? x[l] : 0.0;
  }
}

__global__ void __launch_bounds__(kBlock) k_dot(const double* a, const double* b, int64_t n, double* part) {
  __shared__ double sh[kBlock / 32];
  double v = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * kBlock + threadIdx.x; i < n; i += int64_t(gridDim.x) * kBlock)
    v += a[i] * b[i];
  const double t = block_sum(v, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void k_dot_final(const double* part, double* out) {
  const double v = sum_partials(part);
  if (threadIdx.x == 0) *out = v;
}

}  // namespace solve

int64_t compliance_work_doubles(int64_t n_free, int64_t nnz) {
  // values [nnz] | b [n] | x, r, z, p, q, D^-1 [6n] | partials [3 G] | scalars
  return nnz + 7 * n_free + 3 * solve::kGridBlocks + solve::kScalars;
}

int compliance_solve(const ComplianceArgs& a, cudaStream_t st) {
  using namespace solve;
  const int64_t n = a.n_free;
  double* w = a.work;
  double* val = w;
  double* b = val + a.nnz;
  CgParams p;
  p.n = n;
  p.row_ptr = a.row_ptr;
  p.col = a.col;
  p.val = val;
  p.b = b;
  p.x = b + n;
  p.r = p.x + n;
  p.z = p.r + n;
  p.p = p.z + n;
  p.q = p.p + n;
  p.dinv = p.q + n;
  p.part_a = p.dinv + n;
  p.part_c = p.part_a + 2 * kGridBlocks;
  // the exchange slots, 16-byte aligned: 6 x 152 x 2 of part_b's and part_c's 2432
  // doubles (part_c is done with before the first iteration)
  p.part_b = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(p.part_a + kGridBlocks) + 15) & ~uintptr_t(15));
  p.s = p.part_c + kGridBlocks;
  *a.iterations = 0;
  *a.rel_residual = 0.0;
  cudaError_t e = cudaMemsetAsync(p.s, 0, kScalars * sizeof(double), st);
  if (e != cudaSuccess) return set_error(FE_ERR_CUDA, "compliance: memset");
  std::vector<double> hs(kScalars);
  if (n > 0) {
    k_cg_init<<<kGridBlocks, kBlock, 0, st>>>(p);
    k_cg_init_sums<<<1, 32, 0, st>>>(p);
    e = cudaMemcpyAsync(hs.data(), p.s, kScalars * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return set_error(FE_ERR_CUDA, "compliance: PCG start");
    const double bb = hs[S_BB];
    uint64_t flag = 0;
    std::memcpy(&flag, &hs[S_FLAG], sizeof(flag));
    if (flag & kFlagNotSpd) return set_error(FE_ERR_INVALID_ARG, "compliance: a diagonal entry is not positive");
    if (!std::isfinite(bb) || !std::isfinite(hs[S_RZ]))
      return set_error(FE_ERR_INVALID_ARG, "compliance: the squared norms of the load are not finite");
    int it = 0;
    double rel = 0.0;
    if (bb > 0.0) {
      int dev = 0, nsm = 0, per_sm = 0;
      e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
      // virtual blocks: one per 32 rows up to one per SM (a function of n alone)
      int nv = int(std::min<int64_t>(kVirtual, (n + 31) / 32));
      const int64_t per_block = (n + nv - 1) / nv;
      const int lanes = a.nnz / n > 128 ? 8 : per_block > 256 && per_block <= 512 ? 2 : 4;  // per row of the SpMV
      auto kernel = [&](auto res) {
        constexpr bool R = decltype(res)::value;
        return lanes == 8 ? reinterpret_cast<const void*>(k_pcg<8, R>)
               : lanes == 2 ? reinterpret_cast<const void*>(k_pcg<2, R>)
                            : reinterpret_cast<const void*>(k_pcg<4, R>);
      };
      // vectors in registers: one row per thread and one virtual block per block
      const bool res = per_block <= kPcgThreads && nv <= nsm;
      const void* kern = res ? kernel(std::true_type()) : kernel(std::false_type());
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPcgThreads, 0);
      if (e != cudaSuccess || per_sm < 1) return set_error(FE_ERR_CUDA, "compliance: PCG launch");
      int grid = std::min(nv, nsm * per_sm);
      rel = 1.0;
      while (it < a.max_iter && rel > a.rtol) {
        int n_it = std::min(kChunk, a.max_iter - it);
        double rtol = a.rtol;
        void* args[] = {&p, &nv, &n_it, &rtol};
        auto launch = [&] {
          if (a.max_blocks > 0 && grid > a.max_blocks) return cudaErrorCooperativeLaunchTooLarge;
          return cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(kPcgThreads), args, 0, st);
        };
        e = cudaMemsetAsync(p.part_b, 0xff, Exchange::kSets * kVirtual * 2 * sizeof(double), st);
        if (e == cudaSuccess) e = launch();
        // a process that may use part of the SMs only: the form that keeps its vectors
        // in memory, whose blocks loop over the virtual blocks, with as many as fit
        while (e == cudaErrorCooperativeLaunchTooLarge && grid > 1) {
          cudaGetLastError();
          kern = kernel(std::false_type());
          grid /= 2;
          e = launch();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), p.s, kScalars * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return set_error(FE_ERR_CUDA, "compliance: PCG iteration");
        std::memcpy(&flag, &hs[S_FLAG], sizeof(flag));
        if (flag & kFlagTimeout) return set_error(FE_ERR_TIMEOUT, "compliance: a bounded device wait gave up");
        if (flag & kFlagNotSpd) return set_error(FE_ERR_INVALID_ARG, "compliance: the constrained matrix is not positive definite");
        it += int(hs[S_IT]);
        rel = std::sqrt(hs[S_RR] / bb);
        if ((flag & kFlagDiverged) || !std::isfinite(rel)) return set_error(FE_ERR_INVALID_ARG, "compliance: PCG diverged");
      }
    }  // else b = 0: the initial x = 0 is the solution
    *a.iterations = it;
    *a.rel_residual = rel;
    if (rel > a.rtol) {
      return set_error(FE_ERR_NOT_CONVERGED, "compliance: PCG reached max_iter before rtol");
    }
  }
  // u over all DOFs, c = f . x over the free DOFs
  const int eb = int(std::min<int64_t>(std::max<int64_t>(1, (a.n_dofs + kBlock - 1) / kBlock), kGridBlocks));
  k_expand<<<eb, kBlock, 0, st>>>(a.label, a.n_dofs, p.x, a.u);
  k_dot<<<kGridBlocks, kBlock, 0, st>>>(b, p.x, n, p.part_a);
  k_dot_final<<<1, 32, 0, st>>>(p.part_a, a.compliance);
  e = cudaGetLastError();
  return e == cudaSuccess ? FE_OK : set_error(FE_ERR_CUDA, "compliance: kernels");
}

}  // namespace feasm
