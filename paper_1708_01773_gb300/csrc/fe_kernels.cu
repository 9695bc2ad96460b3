// CUDA kernels of libfeasm (sm_103a): cell integration (geometry, physical
// gradients, cell-matrix contraction, cell vectors) and the deterministic
// segmented scatter into CSR.
#include "fe_device.cuh"

namespace feasm {


// Shared memory of k_cell: for FP64, vertex coordinates [cpb][24],
// trilinear coefficients [cpb][21], per-point geometry [cpb][nq][11]
// (cofactors, w/det, w*det) and the cofactor gradients [cpb][nq][3][nb]; for
// the FP32/BF16 forms the layout of mixed_layout. -1 if it exceeds an SM.
long cell_smem_bytes(int nb, int nq, fe_precision prec, int cpb) {
  long bytes;
  if (prec == FE_PREC_FP64) {
    bytes = long(cpb) * (24 + 21) * 8 + long(cpb) * nq * 11 * 8 + long(cpb) * nq * 3 * nb * 8;
  } else {
    int n1d = 1;
    while (n1d * n1d * n1d < nq) ++n1d;
    bytes = mixed_layout(cpb, nq, n1d, nb).bytes;
  }
  return bytes <= 227 * 1024 ? bytes : -1;
}

// Cells per block of k_cell: at least one node pair per thread, then doubled
// while the block has fewer than 128 quadrature points (the FP64 geometry
// runs one thread per point: 128 points fill four warps, one per SM
// sub-partition, each with its own share of the FP64 pipe) and the shared
// memory of every precision stays within 64 KB.
int cells_per_block(int nb, int nq) {
  const int pairs = nb * nb;
  int cpb = pairs >= kCellThreads ? 1 : kCellThreads / pairs;
  auto fits = [&](int c) {
    const long a = cell_smem_bytes(nb, nq, FE_PREC_FP64, c), b = cell_smem_bytes(nb, nq, FE_PREC_FP32, c);
    return a >= 0 && b >= 0 && a <= 64 * 1024 && b <= 64 * 1024;
  };
  while (cpb * nq < 128 && fits(2 * cpb)) cpb *= 2;
  return cpb;
}

template <int P, int NC, int PREC>
__global__ void __launch_bounds__(kCellThreads) k_cell(CellParams prm) {
  extern __shared__ __align__(16) double smem[];
  const int64_t e0 = int64_t(blockIdx.x) * prm.cpb;
  const int ncell = int(prm.n_cells - e0 < prm.cpb ? prm.n_cells - e0 : prm.cpb);
  cell_block<P, NC, PREC, true>(prm, e0, ncell, smem);
}

template <int P, int NC, int PREC>
static cudaError_t launch_cell_t(const fe_space* s, CellParams prm, long smem, cudaStream_t st) {
  auto kern = k_cell<P, NC, PREC>;
  int threads = kCellThreads;
  if (PREC == 0 && prm.nq1d == P + 1) {
    // cell_block_fixed needs less shared memory than the general layout, and no fixed block size
    using F = FixedShape<P, NC>;
    static_assert(NC == 3 || F::CELLS * F::TILES <= F::THREADS, "one tile per thread");
    threads = F::THREADS;
    prm.cpb = F::CELLS;
    smem = F::smem(prm.cpb);
  }
  if constexpr (PREC != 0) {
    using W = WideShape<P, NC, PREC>;
    if (W::THREADS && prm.nq1d == P + 1) {
      threads = W::THREADS;
      prm.cpb = W::CELLS;
      const MixedLayout L = mixed_layout(prm.cpb, prm.nq, prm.nq1d, (P + 1) * (P + 1) * (P + 1));
      // Q3 Poisson holds the operands of one slab of points, plain and scaled
      smem = P == 3 && NC == 1 ? L.ga + 2l * 16 * 3 * 64 * 4 : L.bytes;
    }
  }
  if (smem > 48 * 1024) {  // (above the default limit)
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
  }
  const int64_t blocks = (s->n_cells + prm.cpb - 1) / prm.cpb;
  kern<<<dim3(unsigned(blocks)), threads, size_t(smem), st>>>(prm);
  return cudaGetLastError();
}

template <int P, int NC>
static cudaError_t launch_cell_p(const fe_space* s, const CellParams& prm, long smem, fe_precision prec,
                                 cudaStream_t st) {
  switch (prec) {
    case FE_PREC_FP64: return launch_cell_t<P, NC, 0>(s, prm, smem, st);
    case FE_PREC_FP32: return launch_cell_t<P, NC, 1>(s, prm, smem, st);
    default: return launch_cell_t<P, NC, 2>(s, prm, smem, st);
  }
}

CellParams space_cell_params(const fe_space* s) {
  CellParams p;
  p.n_cells = s->n_cells;
  p.nq = s->nq;
  p.cpb = cells_per_block(s->nb, s->nq);
  p.qblock = s->nq1d * s->nq1d;
  p.nq1d = s->nq1d;
  p.xv = s->d_xv;
  p.w = s->d_w;
  p.xq = s->d_xq;
  p.phi = s->d_phi;
  p.phi2 = reinterpret_cast<const float2*>(s->d_phi2);
  p.dphi = s->d_dphi;
  p.dphi32 = s->d_dphi32;
  p.coef = nullptr;
  p.dfix = reinterpret_cast<const int2*>(s->d_dfix);
  p.fix_lm = s->d_fix_lm;
  for (int k = 0; k < 3; ++k) p.f[k] = 0.0;
  p.lam_hat = s->nu / ((1.0 + s->nu) * (1.0 - 2.0 * s->nu));
  p.mu_hat = 1.0 / (2.0 * (1.0 + s->nu));
  p.ke = s->d_ke;
  p.fe = s->d_fe;
  p.err = s->d_err;
  return p;
}

cudaError_t launch_cell_integration(const fe_space* s, const double* coef, const double force[3],
                                    fe_precision prec, cudaStream_t st) {
  if (s->n_cells == 0) return cudaSuccess;
  CellParams prm = space_cell_params(s);
  prm.coef = coef;
  for (int k = 0; k < 3; ++k) prm.f[k] = force[k];
  const long smem = cell_smem_bytes(s->nb, s->nq, prec, prm.cpb);
  if (smem < 0) return cudaErrorInvalidConfiguration;
  const int key = s->order * 10 + s->ncomp;
  switch (key) {
    case 11: return launch_cell_p<1, 1>(s, prm, smem, prec, st);
    case 13: return launch_cell_p<1, 3>(s, prm, smem, prec, st);
    case 21: return launch_cell_p<2, 1>(s, prm, smem, prec, st);
    case 23: return launch_cell_p<2, 3>(s, prm, smem, prec, st);
    case 31: return launch_cell_p<3, 1>(s, prm, smem, prec, st);
    case 33: return launch_cell_p<3, 3>(s, prm, smem, prec, st);
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------------------
// Deterministic scatter (Eq. assembly). One warp assembles one CSR row r at a
// time. The row's contributions are its codes, sorted by destination nonzero
// (columns ascending) and, within a nonzero, by ascending cell; a code
// (head << 15 | s << 8 | m) names entry m of the cell-matrix row of DOF r in
// the row's s-th cell ("slot"), head marking the first contribution of a
// nonzero.
//
// k_scatter_rows copies the row's cell-matrix rows (padded to NLP entries,
// 16-byte vector loads) and its codes (16-byte aligned blocks) into a
// per-warp region of shared memory, finds the segment starts from the head
// flags with one ballot per 32 codes, then gives each lane one nonzero: the
// lane sums its segment from shared memory and stores values[k] (consecutive
// k across the lanes: coalesced). The RHS entry of the row is the exact sum of
// its cells' FP64 cell-vector entries.
//
// k_scatter (one lane per nonzero, direct gathers from global memory, using
// the per-nonzero counts, same arithmetic) serves meshes whose largest row does
// not fit the shared-memory region or that have more than 32 cells around a DOF.
template <typename TK>
__global__ void __launch_bounds__(kScatterWarps * 32) k_scatter(ScatterParams p) {
  __shared__ int64_t sbase[kScatterWarps][kMaxSlots + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const TK* ke = reinterpret_cast<const TK*>(p.ke);
  ItemStream items(p.sched, p.n_rows, 1, lane);
  for (; items.valid(); items.advance(lane)) {
    const int64_t r = items.u;
    const int64_t s0 = p.slot_ptr[r];
    const int ns = int(p.slot_ptr[r + 1] - s0);
    for (int s = lane; s < ns; s += 32) sbase[warp][s] = int64_t(p.slots[s0 + s]) * p.nlp;
    __syncwarp();
    if (p.rhs != nullptr && lane == 0)
      p.rhs[r] = fx_sum<double>(ns, [&](int t) { return p.fe[p.slots[s0 + t]]; });
    const int64_t k0 = p.row_ptr[r], k1 = p.row_ptr[r + 1];
    int64_t c = p.code_ptr[r];
    for (int64_t kb = k0; kb < k1; kb += 32) {
      const int64_t k = kb + lane;
      const int n = k < k1 ? int(p.cnt[k]) : 0;
      int incl = n;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += t;
      }
      const int total = __shfl_sync(kFull, incl, 31);
      const uint16_t* cp = p.codes + c + (incl - n);
      if (k < k1) {
        p.values[k] = fx_sum<TK>(n, [&](int t) {
          const unsigned code = cp[t];
          return ke[sbase[warp][(code >> 8) & 127u] + (code & 255u)];
        });
      }
      c += total;
    }
    __syncwarp();
  }
  items.finish(int64_t(gridDim.x) * kScatterWarps, lane);
}

template <typename TK>
__global__ void __launch_bounds__(kScatterWarps * 32) k_scatter_rows(ScatterParams p) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* region = sm + size_t(warp) * p.warp_bytes;
  TK* ske = reinterpret_cast<TK*>(region);
  uint16_t* scode = reinterpret_cast<uint16_t*>(region + p.ke_bytes);
  uint16_t* sseg = reinterpret_cast<uint16_t*>(region + p.ke_bytes + p.code_bytes);
  const int vper = p.nlp * int(sizeof(TK)) / 16;  // 16-byte vectors per cell-matrix row
  const uint4* ke4 = reinterpret_cast<const uint4*>(p.ke);
  const unsigned lt_mask = (1u << lane) - 1u;
  ItemStream items(p.sched, p.n_rows, 1, lane);
  for (; items.valid(); items.advance(lane)) {
    const int64_t r = items.u;
    const int64_t s0 = p.slot_ptr[r];
    const int ns = int(p.slot_ptr[r + 1] - s0);
    const int64_t k0 = p.row_ptr[r];
    const int64_t c0 = p.code_ptr[r];
    const int nc = p.ncode ? p.ncode[r] : ns * p.nl;
    const int my_slot = lane < ns ? p.slots[s0 + lane] : 0;
    const uint4* c4 = reinterpret_cast<const uint4*>(p.codes + c0);
    const int nc8 = (nc + 7) >> 3;
    for (int i = lane; i < nc8; i += 32) reinterpret_cast<uint4*>(scode)[i] = __ldg(c4 + i);
    const int nv = ns * vper;
    for (int base = 0; base < nv; base += 32) {
      const int i = base + lane;
      const int s = min(i / vper, ns - 1);
      const int sid = __shfl_sync(kFull, my_slot, s);
      if (i < nv) reinterpret_cast<uint4*>(ske)[i] = __ldg(ke4 + int64_t(sid) * vper + (i - s * vper));
    }
    if (p.rhs != nullptr) {
      // the same exact fixed-point sum, the terms spread over the lanes
      uint64_t m = 0;
      int ex = 1;
      bool ng = false;
      if (lane < ns) FxTraits<double>::split(p.fe[my_slot], m, ex, ng);
      const int emax = __reduce_max_sync(kFull, m != 0 ? ex : 1);
      const int sh = FxTraits<double>::kShift0 - (emax - ex);
      const uint64_t a = sh >= 0 ? (m << sh) : (sh > -64 ? (m >> (-sh)) : 0ull);
      int64_t S = ng ? -int64_t(a) : int64_t(a);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) S += __shfl_xor_sync(kFull, S, off);
      if (lane == 0) p.rhs[r] = fx_to_double(S, emax - FxTraits<double>::kScale);
    }
    __syncwarp();
    int heads = 0;
    for (int cb = 0; cb < nc; cb += 32) {
      const int i = cb + lane;
      const bool h = i < nc && (scode[i] & 0x8000u) != 0;
      const unsigned m = __ballot_sync(kFull, h);
      if (h) sseg[heads + __popc(m & lt_mask)] = uint16_t(i);
      heads += __popc(m);
    }
    if (lane == 0) sseg[heads] = uint16_t(nc);
    __syncwarp();
    for (int k = lane; k < heads; k += 32) {
      const int a = sseg[k], b = sseg[k + 1];
      p.values[k0 + k] = fx_sum<TK>(b - a, [&](int t) {
        const unsigned code = scode[a + t];
        return ske[((code >> 8) & 127u) * p.nlp + (code & 255u)];
      });
    }
    __syncwarp();
  }
  items.finish(int64_t(gridDim.x) * kScatterWarps, lane);
}

// Slot-wise scatter for FP32 cell matrices (the FP32 and BF16 forms). One warp
// per work item: a CSR row r (R = 1), or the R = ncomp rows of one node, which
// lie in the same cells at local rows i * nb + a and share their column
// pattern (R = 3). For each cell around the DOF in ascending order ("slot"),
// the lanes read that cell's matrix row(s) (coalesced) and the slot-major
// positions pos[s][m] of the entries among the row's nonzeros (one position
// block serves all R rows). The first contribution of each nonzero (flag bit
// 15 of pos; every entry of slot 0) stores (v, 0) into the row's double-float
// accumulator in shared memory; later ones add with Knuth's TwoSum, whose
// rounding error is kept exactly in the low part. The entries of one cell row
// go to distinct nonzeros, so the lanes never collide; a __syncwarp between
// slots orders the additions, so every nonzero sums its terms in ascending cell
// order. Each accumulator is rounded once to FP64 (df_to_double) and stored
// coalesced. Lanes past the end of a cell row (m >= NL) read padding and touch
// a private dummy accumulator, so the inner loop has no divergent branches
// (the position array and the cell-matrix scratch are allocated with padding
// for those reads). Slots are processed in batches of 4, 2 or 1 (the
// largest that fits the slots left and the register budget), all loads of a
// batch issued before its additions; the item descriptors (pointers, slot ids)
// of the warp's next item are fetched while the current one is reduced. Items
// go to warps on demand, kSlotGrab at a time (ItemStream). The RHS entries are
// formed first, in a static pass of 32 consecutive items per warp, one item per
// lane (exact fixed-point sum of its cells' FP64 cell-vector entries).
constexpr int kSlotGrab = 4;  // items per grab of k_scatter_slots

template <int NL, int R, bool IDX32>
__global__ void __launch_bounds__(kScatterWarps * 32, NL >= 128 ? 4 : 5) k_scatter_slots(ScatterParams p) {
  using S = SlotScatter<NL, R>;
  extern __shared__ __align__(16) unsigned char sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* acc = reinterpret_cast<float2*>(sm + size_t(warp) * p.warp_bytes);
  const int rs = p.acc_stride + 32;       // accumulator row: acc_stride nonzeros, then one dummy per lane
  const int dummy = p.acc_stride + lane;  // within each accumulator row
  const float* ke = reinterpret_cast<const float*>(p.ke) + lane;
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
    int sb = 0;
    while (sb < ns) {
      const int left = ns - sb;
      if (S::SB >= 4 && left >= 4) {
        S::template batch<4, IDX32>(p, ke, pos, my_slot, sb, acc, rs, dummy, lane);
        sb += 4;
      } else if (S::SB >= 2 && left >= 2) {
        S::template batch<2, IDX32>(p, ke, pos, my_slot, sb, acc, rs, dummy, lane);
        sb += 2;
      } else {
        S::template batch<1, IDX32>(p, ke, pos, my_slot, sb, acc, rs, dummy, lane);
        sb += 1;
      }
    }
    // second-level descriptors of the next item (its slot ids)
    const int nsn = int(s1n - s0n);
    const int my_slot_n = (un < n_items && lane < nsn) ? p.slots[s0n + lane] : 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int64_t ki = k0 + int64_t(i) * nnz;  // the rows of one node are consecutive and equally long
      const float2* ai = acc + i * rs;
      for (int kb = 0; kb < nnz; kb += 32) {
        const int k = kb + lane;
        const float2 a = ai[k < nnz ? k : dummy];
        const double v = df_to_double(a.x, a.y);
        if (k < nnz) p.values[ki + k] = v;
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

static int align16(long x) { return int((x + 15) & ~15L); }

ScatterPattern space_pattern(const fe_space* s) {
  ScatterPattern pt;
  pt.n_rows = s->hs.n_dofs;
  pt.nnz = s->hs.nnz;
  pt.max_row_nnz = s->hs.max_row_nnz;
  pt.max_slots = s->hs.max_slots;
  pt.node_rows = s->hs.node_rows;
  pt.pos_ok = s->hs.pos_ok;
  pt.row_ptr = s->d_row_ptr;
  pt.cnt = s->d_cnt;
  pt.code_ptr = s->d_code_ptr;
  pt.codes = s->d_codes;
  pt.pos = s->d_pos;
  pt.slot_ptr = s->d_slot_ptr;
  pt.slots = s->d_slots;
  pt.ncode = nullptr;
  pt.sched = s->d_sched;
  return pt;
}

cudaError_t launch_scatter(const fe_space* s, fe_precision prec, double* values, double* rhs, cudaStream_t st) {
  return launch_scatter_pattern(s, space_pattern(s), prec, values, rhs, st);
}

cudaError_t launch_scatter_rows(const fe_space* s, const ScatterPattern& pt, fe_precision prec, double* values,
                                double* rhs, int64_t r0, int64_t r1, cudaStream_t st) {
  // every row-indexed array is offset to r0; positions within values, codes,
  // slots and cell data are absolute, so the kernels run unchanged
  ScatterPattern q = pt;
  q.n_rows = r1 - r0;
  q.row_ptr = pt.row_ptr + r0;
  q.code_ptr = pt.code_ptr + r0;
  q.slot_ptr = pt.slot_ptr + r0;
  if (pt.ncode) q.ncode = pt.ncode + r0;
  return launch_scatter_pattern(s, q, prec, values, rhs ? rhs + r0 : nullptr, st);
}

cudaError_t launch_scatter_pattern(const fe_space* s, const ScatterPattern& pt, fe_precision prec, double* values,
                                   double* rhs, cudaStream_t st) {
  if (pt.n_rows == 0) return cudaSuccess;
  ScatterParams p;
  p.n_rows = pt.n_rows;
  p.nl = s->nl;
  p.nlp = s->nlp;
  p.row_ptr = pt.row_ptr;
  p.cnt = pt.cnt;
  p.code_ptr = pt.code_ptr;
  p.codes = pt.codes;
  p.pos = pt.pos;
  p.slot_ptr = pt.slot_ptr;
  p.slots = pt.slots;
  p.ncode = pt.ncode;
  p.sched = pt.sched;
  p.ke = s->d_ke;
  p.fe = s->d_fe;
  p.values = values;
  p.rhs = rhs;
  const int tk = prec == FE_PREC_FP64 ? 8 : 4;
  p.ke_bytes = align16(long(pt.max_slots) * s->nlp * tk);
  p.code_bytes = align16(((long(pt.max_slots) * s->nl + 7) & ~7L) * 2);
  const int rows_warp_bytes = p.ke_bytes + p.code_bytes + align16((pt.max_row_nnz + 1) * 2);
  const long smem = long(rows_warp_bytes) * kScatterWarps;
  const int nsm = s->n_sm;
  if (pt.max_slots <= 32 && pt.pos_ok) {
    bool taken;
    const cudaError_t e = launch_scatter_small(s, p, prec, pt.max_row_nnz, st, &taken);
    if (taken || e != cudaSuccess) return e;
  }
  const int64_t need = (p.n_rows + kScatterWarps - 1) / kScatterWarps;
  auto launch = [&](auto kern, long bytes) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kScatterWarps * 32, size_t(bytes));
    if (e != cudaSuccess) return e;
    const int blocks = int(std::min<int64_t>(need, int64_t(nsm) * std::max(1, per_sm)));
    kern<<<blocks, kScatterWarps * 32, size_t(bytes), st>>>(p);
    return cudaGetLastError();
  };
  if (prec != FE_PREC_FP64 && pt.max_slots <= 32 && pt.pos_ok) {
    const bool idx32 = int64_t(s->n_cells) * s->nl * s->nlp < (int64_t(1) << 32);
    p.acc_stride = int((pt.max_row_nnz + 3) & ~int64_t(3));
    // rows of one node together (3-component problems), else one row per warp
    // (measured: pays for Q1, 24-entry cell rows; for wider rows one row per warp is faster)
    const int R = (pt.node_rows && s->ncomp == 3 && s->nl <= 32) ? 3 : 1;  // 3: nl = 24 only
    p.warp_bytes = R * (p.acc_stride + 32) * 8;  // R accumulator rows, each with one dummy per lane
    const long bytes = long(p.warp_bytes) * kScatterWarps;
    if (bytes <= 200 * 1024) {
      switch (s->nl * 4 + (R == 3 ? 2 : 0) + (idx32 ? 1 : 0)) {
        case 32: return launch(k_scatter_slots<8, 1, false>, bytes);
        case 33: return launch(k_scatter_slots<8, 1, true>, bytes);
        case 96: return launch(k_scatter_slots<24, 1, false>, bytes);
        case 97: return launch(k_scatter_slots<24, 1, true>, bytes);
        case 98: return launch(k_scatter_slots<24, 3, false>, bytes);
        case 99: return launch(k_scatter_slots<24, 3, true>, bytes);
        case 108: return launch(k_scatter_slots<27, 1, false>, bytes);
        case 109: return launch(k_scatter_slots<27, 1, true>, bytes);
        case 256: return launch(k_scatter_slots<64, 1, false>, bytes);
        case 257: return launch(k_scatter_slots<64, 1, true>, bytes);
        case 324: return launch(k_scatter_slots<81, 1, false>, bytes);
        case 325: return launch(k_scatter_slots<81, 1, true>, bytes);
        case 356: return launch(k_scatter_slots<89, 1, false>, bytes);   // Stokes Q2/Q1
        case 357: return launch(k_scatter_slots<89, 1, true>, bytes);
        case 768: return launch(k_scatter_slots<192, 1, false>, bytes);
        case 769: return launch(k_scatter_slots<192, 1, true>, bytes);
        default: break;
      }
    }
  }
  if (prec == FE_PREC_FP64 && pt.max_slots <= 32 && pt.pos_ok) {
    bool taken;
    const int all = int(std::min<int64_t>(need, int64_t(1) << 30));
    const cudaError_t e = launch_scatter_slots64(s, p, pt.node_rows, pt.max_row_nnz, all, st, &taken);
    if (taken || e != cudaSuccess) return e;
  }
  p.warp_bytes = rows_warp_bytes;
  if (smem <= 200 * 1024 && pt.max_slots <= 32) {
    return prec == FE_PREC_FP64 ? launch(k_scatter_rows<double>, smem) : launch(k_scatter_rows<float>, smem);
  }
  const int blocks = int(std::min<int64_t>(need, int64_t(nsm) * 8));
  if (prec == FE_PREC_FP64)
    k_scatter<double><<<blocks, kScatterWarps * 32, 0, st>>>(p);
  else
    k_scatter<float><<<blocks, kScatterWarps * 32, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace feasm
