// Slot-wise scatter for FP64 cell matrices: the walk of k_scatter_slots
// (fe_kernels.cu) with integer accumulators; and the scatter of small systems in
// all precisions.
#include <algorithm>
#include <type_traits>

#include "fe_device.cuh"

namespace feasm {

constexpr int kSlotGrab = 4;  // items per grab

// One batch of B slots, R rows per item (see SlotScatter). A nonzero's
// accumulator is an FxChain, its sum and its exponent kept in two arrays of the
// warp's shared memory: at least as accurate as FP64 additions, which this GPU
// issues at 2 lanes per clock per SM.
template <int NL, int R, KeWritten W = KeWritten::kBefore>
struct SlotScatter64 {
  static constexpr KeWritten kWritten = W;
  static constexpr int CH = (NL + 31) / 32;
  static constexpr int NBR = NL / R;
  static constexpr int LOADS = CH * R;
  static constexpr int SB = LOADS <= 3 ? 4 : LOADS <= 4 ? 2 : 1;  // slots per batch

  template <int B, bool IDX32>
  __device__ __forceinline__ static void batch(const ScatterParams& p, const double* ke, const uint16_t* pos,
                                               int my_slot, int s_begin, int64_t* acc, int* exps, int rs, int dummy,
                                               int lane, const int (&flip)[R]) {
    double x[B][CH][R];
    int kk[B][CH];
#pragma unroll
    for (int t = 0; t < B; ++t) {
      const int s = s_begin + t;
      const int sid = __shfl_sync(kFull, my_slot, s);
      const double* krow = IDX32 ? ke + uint32_t(sid) * uint32_t(p.nlp) : ke + int64_t(sid) * p.nlp;
      const uint16_t* prow = pos + s * NL;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const bool in = c < CH - 1 || c * 32 + lane < NL;
        kk[t][c] = in ? int(__ldg(prow + c * 32)) : dummy;
#pragma unroll
        for (int i = 0; i < R; ++i) x[t][c][i] = in ? ld_ke<W>(krow + i * NBR * p.nlp + c * 32) : 0.0;
      }
    }
#pragma unroll
    for (int t = 0; t < B; ++t) {
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int raw = kk[t][c];
        const int k = raw & 0x7fff;
        const bool first = s_begin + t == 0 || (raw & 0x8000);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          int64_t* ai = acc + i * rs;
          int* ei = exps + i * rs;
          FxChain v = FxChain::term(x[t][c][i], flip[i]);
          if (!first) {
            FxChain acc{ai[k], ei[k]};
            acc.add(v);
            v = acc;
          }
          ai[k] = v.S;
          ei[k] = v.e;
        }
      }
      __syncwarp();
    }
  }
};

// The row's nonzeros whose sums are odd(), from the row's codes, one lane per
// nonzero (k_scatter's method).
static __device__ __noinline__ void row_from_codes(const ScatterParams& p, int64_t r, int64_t k0, int nnz,
                                                   const int64_t* acc, const int* exps, int lane) {
  const double* ke = reinterpret_cast<const double*>(p.ke);
  const int64_t s0 = p.slot_ptr[r];
  const uint16_t* codes = p.codes + p.code_ptr[r];
  int64_t c = 0;
  for (int kb = 0; kb < nnz; kb += 32) {
    const int64_t k = k0 + kb + lane;
    const int n = kb + lane < nnz ? int(p.cnt[k]) : 0;
    int incl = n;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += t;
    }
    const uint16_t* cp = codes + c + (incl - n);
    if (n > 0 && FxChain{acc[kb + lane], exps[kb + lane]}.odd())
      p.values[k] = fx_sum<double>(n, [&](int t) {
        const unsigned code = cp[t];
        return ke[int64_t(p.slots[s0 + ((code >> 8) & 127u)]) * p.nlp + (code & 255u)];
      });
    c += __shfl_sync(kFull, incl, 31);
  }
}

// One warp per work item: a CSR row (R = 1), or the three rows of one node
// (R = 3, Q1 elasticity), slots in ascending cell order; one rounding per
// nonzero. Sums near the ends of the exponent range (infinities, NaN,
// denormals) are redone with fx_sum over the row's destination-sorted codes.
// k_scatter_rows gives each nonzero a lane, with two passes over its 1 to 8
// terms, so that a warp's lanes wait for the one with the most. Bound by the ALU
// pipe (67 % busy, about 20 integer instructions per term); measured against
// k_scatter_rows, ms: elasticity Q1 64^3 1.60 -> 0.550, Q2 24^3 0.945 -> 0.367, Q3
// 12^3 1.20 -> 0.322; Poisson Q1 64^3 0.28 -> 0.182, Q3 24^3 0.54 -> 0.246; Stokes
// 24^3 1.15 -> 0.41.
template <int NL, int R, bool IDX32>
__global__ void __launch_bounds__(kScatterWarps * 32, 4) k_scatter_slots64(ScatterParams p) {
  using S = SlotScatter64<NL, R>;
  extern __shared__ __align__(16) unsigned char sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t* acc = reinterpret_cast<int64_t*>(sm + size_t(warp) * p.warp_bytes);
  const int rs = p.acc_stride + 32;       // accumulator row: acc_stride nonzeros, then one dummy per lane
  const int dummy = p.acc_stride + lane;  // within each accumulator row
  int* exps = reinterpret_cast<int*>(acc + R * rs);  // exponents of the accumulators
  const double* ke = reinterpret_cast<const double*>(p.ke) + lane;
  const bool want_rhs = p.rhs != nullptr;
  const int64_t n_items = p.n_rows / R;
  const int64_t n_warps = int64_t(gridDim.x) * kScatterWarps;
  ItemStream items(p.sched, n_items, kSlotGrab, lane);
  if (want_rhs) {
    // RHS entries first, statically: 32 consecutive items per warp pass, one per lane
    for (int64_t ub = (int64_t(blockIdx.x) * kScatterWarps + warp) * 32; ub < n_items; ub += n_warps * 32) {
      const int64_t uu = ub + lane;
      if (uu < n_items) {
        const int64_t ss = p.slot_ptr[uu * R];
        const int nss = int(p.slot_ptr[uu * R + 1] - ss);
        if (nss <= 8) {
          // all gathers issued at once, the sum from registers
          int sl[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) sl[t] = t < nss ? p.slots[ss + t] : 0;
#pragma unroll
          for (int i = 0; i < R; ++i) {
            double v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = t < nss ? p.fe[sl[t] + i * S::NBR] : 0.0;
            p.rhs[uu * R + i] = fx_sum_regs(v);
          }
        } else {
#pragma unroll
          for (int i = 0; i < R; ++i)
            p.rhs[uu * R + i] = fx_sum<double>(nss, [&](int t) { return p.fe[p.slots[ss + t] + i * S::NBR]; });
        }
      }
    }
  }
  int64_t u = items.u;
  int64_t s0 = 0, k0 = 0, c0 = 0;
  int ns = 0, nnz = 0, my_slot = 0;
  if (u < n_items) {
    const int64_t r = u * R;
    s0 = p.slot_ptr[r];
    ns = int(p.slot_ptr[r + 1] - s0);
    k0 = p.row_ptr[r];
    nnz = int(p.row_ptr[r + 1] - k0);
    c0 = p.code_ptr[r];
    my_slot = lane < ns ? p.slots[s0 + lane] : 0;
  }
  while (u < n_items) {
    // first-level descriptors of the next item (independent loads)
    items.advance(lane);
    const int64_t un = items.u, rn = un * R;
    int64_t s0n = 0, s1n = 0, k0n = 0, k1n = 0, c0n = 0;
    if (un < n_items) {
      s0n = p.slot_ptr[rn];
      s1n = p.slot_ptr[rn + 1];
      k0n = p.row_ptr[rn];
      k1n = p.row_ptr[rn + 1];
      c0n = p.code_ptr[rn];
    }
    const uint16_t* pos = p.pos + c0 + lane;
    int flip[R];
#pragma unroll
    for (int i = 0; i < R; ++i) flip[i] = FxChain::flip_of(__shfl_sync(kFull, my_slot, 0) + i * S::NBR);
    int sb = 0;
    while (sb < ns) {
      const int left = ns - sb;
      if (S::SB >= 4 && left >= 4) {
        S::template batch<4, IDX32>(p, ke, pos, my_slot, sb, acc, exps, rs, dummy, lane, flip);
        sb += 4;
      } else if (S::SB >= 2 && left >= 2) {
        S::template batch<2, IDX32>(p, ke, pos, my_slot, sb, acc, exps, rs, dummy, lane, flip);
        sb += 2;
      } else {
        S::template batch<1, IDX32>(p, ke, pos, my_slot, sb, acc, exps, rs, dummy, lane, flip);
        sb += 1;
      }
    }
    // second-level descriptors of the next item (its slot ids)
    const int nsn = int(s1n - s0n);
    const int my_slot_n = (un < n_items && lane < nsn) ? p.slots[s0n + lane] : 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int64_t ki = k0 + int64_t(i) * nnz;  // the rows of one node are consecutive and equally long
      bool odd = false;
      for (int j = lane; j < nnz; j += 32) {
        const FxChain v{acc[i * rs + j], exps[i * rs + j]};
        odd |= v.odd();
        p.values[ki + j] = v.round(flip[i]);
      }
      if (__any_sync(kFull, odd)) {
        __syncwarp();
        row_from_codes(p, u * R + i, ki, nnz, acc + i * rs, exps + i * rs, lane);
      }
    }
    __syncwarp();
    s0 = s0n;
    ns = nsn;
    k0 = k0n;
    nnz = int(k1n - k0n);
    c0 = c0n;
    my_slot = my_slot_n;
    u = un;
  }
  items.finish(n_warps, lane);
}

constexpr int kSmallRowsPerSm = 320;

// The scatter of a small system: warp w takes row w, its RHS entry included
// (the exact sum of fx_sum, a term per lane). The kernels for larger systems
// take rows from a counter and form the RHS entries in a pass of their own: a
// chain of dependent round trips to L2 of about 20 us, longer than the work on
// a coarse mesh (729 rows 11.7 -> 5.5 us, cold). Here the block scheduler
// balances the rows, but their row descriptors are read with nothing in flight
// beside them and nodes' rows share no loads, which costs more as the systems
// grow. Measured, us (FP32 / FP64 form), counter -> one row per warp:
//   Poisson Q1      15,625 rows 23 / 33 -> 13 / 18, 68,921 rows 42 / 60 -> 36 / 58,
//                   117,649 rows 58 / 93 -> 64 / 105
//   elasticity Q1   14,739 rows 40 / 42 -> 15 / 19, 59,049 rows 60 / 91 -> 44 / 68,
//                   107,811 rows 74 / 99 -> 76 / 122
//   elasticity Q2   27,783 rows 46 / 66 -> 26 / 44, 59,049 rows 64 / 89 -> 58 / 87,
//                   107,811 rows 97 / 138 -> 103 / 154
//   Poisson Q3      15,625 rows 27 / 33 -> 15 / 19, 39,304 rows 38 / 46 -> 23 / 38,
//                   117,649 rows 74 / 93 -> 74 / 115
// so the line is drawn at kSmallRowsPerSm rows per SM (48,640 on GB300).
// Launched to overlap the cell kernel's end: only static data is read before
// griddepcontrol.wait, and the cell kernel's data with ordinary loads.
// Per nonzero the same terms in the same order as those kernels.
template <int NL, typename TK>
__global__ void __launch_bounds__(kScatterWarps * 32) k_scatter_small(ScatterParams p) {
  constexpr bool F64 = sizeof(TK) == 8;
  constexpr KeWritten W = KeWritten::kOverlap;
  using S = std::conditional_t<F64, SlotScatter64<NL, 1, W>, SlotScatter<NL, 1, W>>;
  static_assert(S::kWritten == KeWritten::kOverlap, "this grid overlaps the kernel that writes the cell matrices");
  extern __shared__ __align__(16) unsigned char sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r = int64_t(blockIdx.x) * kScatterWarps + warp;
  if (r >= p.n_rows) return;
  float2* acc = reinterpret_cast<float2*>(sm + size_t(warp) * p.warp_bytes);
  const int rs = p.acc_stride + 32, dummy = p.acc_stride + lane;
  int64_t* acc64 = reinterpret_cast<int64_t*>(acc);
  int* exps = reinterpret_cast<int*>(acc + rs);
  const int64_t s0 = p.slot_ptr[r], k0 = p.row_ptr[r], c0 = p.code_ptr[r];
  const int ns = int(p.slot_ptr[r + 1] - s0), nnz = int(p.row_ptr[r + 1] - k0);
  const int my_slot = lane < ns ? p.slots[s0 + lane] : 0;
  const uint16_t* pos = p.pos + c0 + lane;
  const int flip[1] = {F64 ? FxChain::flip_of(__shfl_sync(kFull, my_slot, 0)) : 0};
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const TK* ke = reinterpret_cast<const TK*>(p.ke) + lane;
  double fe = 0.0;
  if (p.rhs != nullptr && lane < ns) fe = p.fe[my_slot];
  int sb = 0;
  while (sb < ns) {
    const int left = ns - sb;
    auto run = [&](auto n) {
      constexpr int B = decltype(n)::value;
      if constexpr (F64)
        S::template batch<B, true>(p, ke, pos, my_slot, sb, acc64, exps, rs, dummy, lane, flip);
      else
        S::template batch<B, true>(p, ke, pos, my_slot, sb, acc, rs, dummy, lane);
      sb += B;
    };
    if (S::SB >= 4 && left >= 4)
      run(std::integral_constant<int, 4>());
    else if (S::SB >= 2 && left >= 2)
      run(std::integral_constant<int, 2>());
    else
      run(std::integral_constant<int, 1>());
  }
  if constexpr (F64) {
    bool odd = false;
    for (int j = lane; j < nnz; j += 32) {
      const FxChain v{acc64[j], exps[j]};
      odd |= v.odd();
      p.values[k0 + j] = v.round(flip[0]);
    }
    if (__any_sync(kFull, odd)) {
      __syncwarp();
      row_from_codes(p, r, k0, nnz, acc64, exps, lane);
    }
  } else {
    for (int kb = 0; kb < nnz; kb += 32) {
      const int k = kb + lane;
      const float2 a = acc[k < nnz ? k : dummy];
      const double v = df_to_double(a.x, a.y);
      if (k < nnz) p.values[k0 + k] = v;
    }
  }
  if (p.rhs != nullptr) {
    if (ns == 1) {
      if (lane == 0) p.rhs[r] = fe;
    } else {
      uint64_t m = 0;
      int ex = 1;
      bool ng = false;
      if (lane < ns) FxTraits<double>::split(fe, m, ex, ng);
      const int emax = __reduce_max_sync(kFull, m != 0 ? ex : 1);
      const int sh = FxTraits<double>::kShift0 - (emax - ex);
      const uint64_t a = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> (-sh)) : 0ull);
      int64_t T = ng ? -int64_t(a) : int64_t(a);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) T += __shfl_xor_sync(kFull, T, off);
      if (lane == 0) p.rhs[r] = fx_to_double(T, emax - FxTraits<double>::kScale);
    }
  }
}

cudaError_t launch_scatter_small(const fe_space* s, ScatterParams p, fe_precision prec, int64_t max_row_nnz,
                                 cudaStream_t st, bool* taken) {
  *taken = false;
  const bool f64 = prec == FE_PREC_FP64;
  // one row per warp; 32-bit offsets
  if (p.n_rows > int64_t(s->n_sm) * kSmallRowsPerSm || int64_t(s->n_cells) * s->nl * s->nlp >= (int64_t(1) << 32))
    return cudaSuccess;
  p.acc_stride = int((max_row_nnz + 3) & ~int64_t(3));
  p.warp_bytes = (p.acc_stride + 32) * (f64 ? 12 : 8);
  const size_t bytes = size_t(p.warp_bytes) * kScatterWarps;
  if (bytes > 48 * 1024) return cudaSuccess;  // (within the default limit: no attribute to set)
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned((p.n_rows + kScatterWarps - 1) / kScatterWarps));
  cfg.blockDim = dim3(kScatterWarps * 32);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  auto rows = [&](auto nl) -> cudaError_t {
    constexpr int NL = decltype(nl)::value;
    *taken = true;
    return f64 ? cudaLaunchKernelEx(&cfg, k_scatter_small<NL, double>, p) : cudaLaunchKernelEx(&cfg, k_scatter_small<NL, float>, p);
  };
  using std::integral_constant;
  switch (s->nl) {
    case 8: return rows(integral_constant<int, 8>());
    case 24: return rows(integral_constant<int, 24>());
    case 27: return rows(integral_constant<int, 27>());
    case 64: return rows(integral_constant<int, 64>());
    case 81: return rows(integral_constant<int, 81>());
    case 89: return rows(integral_constant<int, 89>());
    case 192: return rows(integral_constant<int, 192>());
    default: return cudaSuccess;
  }
}

cudaError_t launch_scatter_slots64(const fe_space* s, ScatterParams p, bool node_rows, int64_t max_row_nnz,
                                   int blocks_needed, cudaStream_t st, bool* taken) {
  *taken = false;
  const bool idx32 = int64_t(s->n_cells) * s->nl * s->nlp < (int64_t(1) << 32);
  const int R = node_rows && s->ncomp == 3 && s->nl == 24 ? 3 : 1;
  p.acc_stride = int((max_row_nnz + 3) & ~int64_t(3));
  p.warp_bytes = R * (p.acc_stride + 32) * 12;  // sums and exponents, each row with one dummy per lane
  const long bytes = long(p.warp_bytes) * kScatterWarps;
  if (bytes > 200 * 1024) return cudaSuccess;
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, s->device);
  auto launch = [&](auto kern) -> cudaError_t {
    *taken = true;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kScatterWarps * 32, size_t(bytes));
    if (e != cudaSuccess) return e;
    const int blocks = std::min(blocks_needed, nsm * std::max(1, per_sm));
    kern<<<blocks, kScatterWarps * 32, size_t(bytes), st>>>(p);
    return cudaGetLastError();
  };
  auto rows = [&](auto nl, auto r) -> cudaError_t {
    constexpr int NL = decltype(nl)::value, RR = decltype(r)::value;
    return idx32 ? launch(k_scatter_slots64<NL, RR, true>) : launch(k_scatter_slots64<NL, RR, false>);
  };
  using std::integral_constant;
  const integral_constant<int, 1> one;
  switch (s->nl) {
    case 8: return rows(integral_constant<int, 8>(), one);
    case 24: return R == 3 ? rows(integral_constant<int, 24>(), integral_constant<int, 3>()) : rows(integral_constant<int, 24>(), one);
    case 27: return rows(integral_constant<int, 27>(), one);
    case 64: return rows(integral_constant<int, 64>(), one);
    case 81: return rows(integral_constant<int, 81>(), one);
    case 89: return rows(integral_constant<int, 89>(), one);  // Stokes Q2/Q1
    case 192: return rows(integral_constant<int, 192>(), one);
    default: return cudaSuccess;
  }
}

}  // namespace feasm
