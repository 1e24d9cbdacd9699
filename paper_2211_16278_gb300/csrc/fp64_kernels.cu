// FP64 form of the baryon-block hot path on sm_103a.
//
//   k_phase_table     e^{-i p.x} for integer momenta (Eq. 1/3; the paper precomputes the
//                     phase once per momentum set instead of using an FFT, Sec. 3)
//   k_project_fp64    Eq. (2) as a complex GEMM, q = V^T Phi, one launch for every field
//   k_contract_fp64   fused diquark + colour singlet + momentum projection (Eq. 1/3,
//                     Algorithm 1's diq / singlet / phase-GEMM steps), site-split into slabs
//   k_reduce_slabs    fixed-order sum of the per-slab partial blocks
//
// GB300 runs IEEE double at 1/64 of the FP32 rate (measured: DFMA ~1.19 TFLOP/s, DMMA
// ~1.04 TFLOP/s), so these kernels are bound by the FP64 pipe and are written to
// execute as few FP64 operations as possible:
//   * complex products inside the long sums use the three-multiplication form
//     (re = k1 - k3, im = k1 + k2 with k1 = c(a+b), k2 = a(d-c), k3 = b(c+d));
//     the operand-side sums are formed once when a tile is staged in shared memory;
//   * the spin sum is taken inside the colour singlet, in groups of terms that share a
//     third-quark field, and the momenta along lattice rows (rows_contract.cuh);
//   * the diquark of a (d1,d2) tile is built once per site and reused for every d3 of its tile.
#include "bblock_internal.h"
#include "rows_contract.cuh"

namespace bb {

// ------------------------------------------------------------------ phases

__global__ void k_phase_table(int L, int n_mom, const int* __restrict__ mom,
                              double2* __restrict__ ph, float2* __restrict__ ph_f) {
  const long long X = (long long)L * L * L;
  const long long total = X * n_mom;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int p = (int)(i / X);
    const long long x = i - (long long)p * X;
    const long long x0 = x % L, x1 = (x / L) % L, x2 = x / ((long long)L * L);
    long long k = mom[3 * p] * x0 + mom[3 * p + 1] * x1 + mom[3 * p + 2] * x2;
    k %= L;
    if (k < 0) k += L;
    double s, c;
    sincospi(2.0 * (double)k / (double)L, &s, &c);
    ph[i] = make_double2(c, -s);
    if (ph_f) ph_f[i] = make_float2((float)c, (float)-s);
  }
}

cudaError_t launch_phase_table(int L, int n_mom, const int* d_mom, double2* ph, float2* ph_f,
                               cudaStream_t s) {
  const long long total = (long long)L * L * L * n_mom;
  if (total == 0) return cudaSuccess;
  const int grid = (int)((total + kThreads - 1) / kThreads < 65536 ? (total + kThreads - 1) / kThreads : 65536);
  k_phase_table<<<grid, kThreads, 0, s>>>(L, n_mom, d_mom, ph, ph_f);
  note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------------------ projection (Eq. 2)

// Bound by the FP64 pipe; a padded column or eigenvector costs as much as a real one (a
// predicated-off DFMA still takes the pipe), so the inner loop is instantiated for the 8-column
// blocks of the tile in use and stops at N_ev. 64-row tiles, or 32-row ones where the launch
// would not fill the SMs twice (small lattices: one 64-row CTA of 4 column blocks takes 24 us
// whatever its columns). 4^3, N_ev = 8, N_dil = 8: 36 -> 8 us; the large cases are unchanged.
constexpr int PBN = 32, PBK = 16;

template <int RM>
__global__ void __launch_bounds__(kThreads) k_project_fp64(const ProjField* __restrict__ fields,
                                                           int rows, int n_ev) {
  constexpr int PBM = 32 * RM;
  __shared__ double Ar[PBK][PBM], Ai[PBK][PBM], As[PBK][PBM];
  __shared__ double Bc[PBK][PBN], Bd[PBK][PBN], Be[PBK][PBN];
  const ProjField& F = fields[blockIdx.z];
  const int nd = F.nd;
  const int n0 = blockIdx.y * PBN;
  if (n0 >= nd) return;
  const int m0 = blockIdx.x * PBM;
  const int tid = threadIdx.x, tn = tid % 8, tm = tid / 8;
  const int n_terms = F.n_terms;
  const int act = min(4, (nd - n0 + 7) / 8);   // 8-column blocks in use

  double k1[RM][4], k2[RM][4], k3[RM][4];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) k1[i][j] = k2[i][j] = k3[i][j] = 0.0;
  auto multiply = [&](auto blocks, int kn) {
    constexpr int ACT = decltype(blocks)::value;
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      double ar[RM], ai[RM], as[RM], bc[ACT], bd[ACT], be[ACT];
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        ar[i] = Ar[kk][tm + 32 * i];
        ai[i] = Ai[kk][tm + 32 * i];
        as[i] = As[kk][tm + 32 * i];
      }
#pragma unroll
      for (int j = 0; j < ACT; ++j) {
        bc[j] = Bc[kk][tn + 8 * j];
        bd[j] = Bd[kk][tn + 8 * j];
        be[j] = Be[kk][tn + 8 * j];
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < ACT; ++j) {
          k1[i][j] = fma(bc[j], as[i], k1[i][j]);
          k2[i][j] = fma(ar[i], bd[j], k2[i][j]);
          k3[i][j] = fma(ai[i], be[j], k3[i][j]);
        }
    }
  };

  for (int kb = 0; kb < n_ev; kb += PBK) {
    const int kn = min(PBK, n_ev - kb);
    for (int idx = tid; idx < kn * PBM; idx += kThreads) {
      const int r = idx % PBM, kk = idx / PBM;
      const int l = kb + kk, row = m0 + r;
      double2 v = make_double2(0.0, 0.0);
      if (row < rows) v = F.V[(size_t)l * rows + row];
      Ar[kk][r] = v.x;
      Ai[kk][r] = v.y;
      As[kk][r] = v.x + v.y;
    }
    for (int idx = tid; idx < kn * PBN; idx += kThreads) {
      const int c = idx % PBN, kk = idx / PBN;
      if (c >= 8 * act) continue;
      const int l = kb + kk, col = n0 + c;
      double2 b = make_double2(0.0, 0.0);
      if (col < nd) {
        for (int t = 0; t < n_terms; ++t) {
          const double2 f = F.phi[(size_t)(F.row_off[t] + l) * nd + col];
          const double2 w = F.w[t];
          b.x = fma(w.x, f.x, fma(-w.y, f.y, b.x));
          b.y = fma(w.x, f.y, fma(w.y, f.x, b.y));
        }
      }
      Bc[kk][c] = b.x;
      Bd[kk][c] = b.y - b.x;
      Be[kk][c] = b.x + b.y;
    }
    __syncthreads();
    switch (act) {
      case 1: multiply(std::integral_constant<int, 1>{}, kn); break;
      case 2: multiply(std::integral_constant<int, 2>{}, kn); break;
      case 3: multiply(std::integral_constant<int, 3>{}, kn); break;
      default: multiply(std::integral_constant<int, 4>{}, kn); break;
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int row = m0 + tm + 32 * i;
    if (row >= rows) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = n0 + tn + 8 * j;
      if (col < nd)
        F.q[(size_t)row * nd + col] = make_double2(k1[i][j] - k3[i][j], k1[i][j] + k2[i][j]);
    }
  }
}

cudaError_t launch_project_fp64(const ProjField* d_fields, int n_fields, int rows, int n_ev,
                                int max_nd, cudaStream_t s) {
  if (n_fields == 0 || rows == 0) return cudaSuccess;
  const long long ctas64 = (long long)((rows + 63) / 64) * ((max_nd + PBN - 1) / PBN) * n_fields;
  for (int f0 = 0; f0 < n_fields; f0 += 65535) {  // grid.z limit
    const int nf = n_fields - f0 < 65535 ? n_fields - f0 : 65535;
    const int bm = ctas64 < 2 * kSmHint ? 32 : 64;
    dim3 grid((rows + bm - 1) / bm, (max_nd + PBN - 1) / PBN, nf);
    if (bm == 32) k_project_fp64<1><<<grid, kThreads, 0, s>>>(d_fields + f0, rows, n_ev);
    else k_project_fp64<2><<<grid, kThreads, 0, s>>>(d_fields + f0, rows, n_ev);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ------------------------------------------------------------------ contraction (Eq. 1/3)
//
// The body is rowsc::contract_rows (rows_contract.cuh); here the work units come from the
// context's job table, the fields from the projection (spin coefficients folded) and w^k from
// the cached table. Measured on GB300 (contraction of one time slice or as stated, ms), against
// a singlet per (alpha, beta) pair with a phase product per momentum and site:
//   L = 32, N_dil = 32, 9 momenta, 4 pairs / 2 groups          146.9 -> 55.5
//   L = 24, N_dil = 32, 3 momenta, 3 pairs / 2 groups, 2 slices 66.9 -> 32.1
// i.e. 30.9 (21.3) FP64 instructions per output element and site at 0.95-0.97 of the pipe's
// nominal 1.26 TFLOP/s.

__global__ void k_omega_table(int L, double2* __restrict__ om) {
  for (int k = threadIdx.x; k < L; k += blockDim.x) {
    double s, c;
    sincospi(2.0 * (double)k / (double)L, &s, &c);
    om[k] = make_double2(c, -s);
  }
}

cudaError_t launch_omega_table(int L, double2* om, cudaStream_t s) {
  k_omega_table<<<1, 128, 0, s>>>(L, om);
  note_launch();
  return cudaGetLastError();
}

namespace {

int mod_l(int v, int L) { const int m = v % L; return m < 0 ? m + L : m; }

// The row-factored plans along one axis: classes in order of appearance, kMaxRowCls to a plan;
// the momenta of n0 = 0 join the first plan; a plan that is full of momenta continues in another.
int row_plans(int L, const int32_t* momenta, int n_mom, int axis, RowPlan* out, int max_out) {
  auto cls = [&](int p) {   // |n0| in [0, L / 2]
    const int n = mod_l(momenta[3 * p + axis], L);
    return n < L - n ? n : L - n;
  };
  int order[65], n_order = 0;   // L / 2 <= 64
  for (int p = 0; p < n_mom; ++p) {
    const int k = cls(p);
    bool have = k == 0;
    for (int i = 0; i < n_order; ++i) have = have || order[i] == k;
    if (!have && n_order < 65) order[n_order++] = k;
  }
  const int a1 = axis == 0 ? 1 : 0, a2 = axis == 2 ? 1 : 2;
  int n_plans = 0;
  for (int first = 0; first == 0 || first < n_order; first += kMaxRowCls) {
    RowPlan pl{};
    auto start = [&] {
      pl = RowPlan{};
      pl.axis = axis;
      for (int i = first; i < n_order && i < first + kMaxRowCls; ++i) pl.cls_n0[pl.n_cls++] = order[i];
    };
    auto flush = [&] {
      if (out && n_plans < max_out) out[n_plans] = pl;
      ++n_plans;
    };
    start();
    for (int p = 0; p < n_mom; ++p) {
      const int k = cls(p);
      int sel = 0;
      if (k == 0) {
        if (first != 0) continue;
      } else {
        for (int c = 0; c < pl.n_cls; ++c)
          if (pl.cls_n0[c] == k) sel = mod_l(momenta[3 * p + axis], L) == k ? c + 1 : -(c + 1);
        if (sel == 0) continue;
      }
      if (pl.n_mom == kMaxRowP) { flush(); start(); }
      pl.mom[pl.n_mom++] = RowMom{p, mod_l(momenta[3 * p + a1], L), mod_l(momenta[3 * p + a2], L), sel};
      if (sel == 0) pl.has_zero = 1;
    }
    if (pl.n_mom > 0) flush();
  }
  return n_plans;
}

// The plans with a phase per site, at most cap momenta each, as evenly as possible.
int site_plans(int L, const int32_t* momenta, int n_mom, int cap, RowPlan* out, int max_out) {
  const int parts = (n_mom + cap - 1) / cap, step = (n_mom + parts - 1) / parts;
  int n_plans = 0;
  for (int first = 0; first < n_mom; first += step, ++n_plans) {
    if (!out || n_plans >= max_out) continue;
    RowPlan pl{};
    pl.per_site = 1;
    for (int p = first; p < n_mom && p < first + step; ++p)
      pl.mom[pl.n_mom++] = RowMom{p, mod_l(momenta[3 * p + 1], L), mod_l(momenta[3 * p + 2], L),
                                  mod_l(momenta[3 * p], L)};
    out[n_plans] = pl;
  }
  return n_plans;
}

}  // namespace

// Row-factored along the axis with the fewest classes (the last on a tie), or a phase per site, by
// the operations per output and site (rows_contract.cuh) of all launches: each of them repeats the
// singlet and the diquarks, so lists with more classes than a launch takes, and whose momenta
// hardly share a class, are the second kind's. Beside the operations, as measured (L = 2 to 24,
// N_dil 16 and 32, 1 to 4 pairs): a row's end costs 8 (16 in double-float: the partial block's
// latency) per momentum after the first, and launches of two or three classes, one CTA an SM, a
// tenth more; a phase per site costs a tenth more too (spills, its runs' ends, the shorter
// renormalisation of double-float), so that a single momentum, or lists of one class from L = 4 on,
// go by rows. L = 16, N_dil = 32, one pair, momenta (k, k, k), FP64 / double-float, ms row-factored
// and per site: k < 4  6.83 / 2.17 and 6.70 / 2.13; k < 5  10.7 / 3.34 and 7.96 / 2.51;
// k < 8  16.7 / 5.21 and 10.8 / 3.28; k < 16 in double-float 6.12 and 6.4;
// -3 <= k <= 3  7.06 / 2.39 and 9.6 / 2.6.
int plan_rows(int L, const int32_t* momenta, int n_mom, int groups, int terms, int nd3, bool df,
              RowKind kind, RowPlan* out, int max_out) {
  if (n_mom < 1) return 0;
  int axis = 2, fewest = 1 << 30;
  for (int a = 2; a >= 0; --a) {
    bool seen[65] = {};
    int n = 0;
    for (int p = 0; p < n_mom; ++p) {
      const int n0 = mod_l(momenta[3 * p + a], L), k = n0 < L - n0 ? n0 : L - n0;
      if (k && !seen[k]) { seen[k] = true; ++n; }
    }
    if (n < fewest) { fewest = n; axis = a; }
  }
  const int cap = df ? kMaxSitePDf : kMaxSiteP;
  auto singlet_ops = [&](const RowPlan& shape) {   // of a launch, with the diquarks
    const int tile = 16 * rows_rn_for(&shape, 1, nd3);
    return 9.0 * groups + 24.0 * terms / (tile < nd3 ? tile : nd3);
  };
  RowPlan shape{};
  shape.n_cls = fewest < kMaxRowCls ? fewest : kMaxRowCls;
  const double site_ops = fewest > 0 ? 4.0 : df ? 4.0 : 0.0;   // recombined, and n0 = 0 (ArithF64::kEachSite)
  double by_row = row_plans(L, momenta, n_mom, axis, nullptr, 0) * (singlet_ops(shape) + site_ops) +
                  4.0 * fewest + (df ? 16.0 : 8.0) * (n_mom - 1) / L;
  if (shape.n_cls >= 2) by_row *= 1.1;
  shape = RowPlan{};
  shape.per_site = 1;
  shape.n_mom = n_mom < cap ? n_mom : cap;
  const double by_site = 1.1 * ((n_mom + cap - 1) / cap * (singlet_ops(shape) + 2.0) + 4.0 * n_mom);
  if (kind == ROWS_AUTO && by_site < 0.97 * by_row) return site_plans(L, momenta, n_mom, cap, out, max_out);
  return row_plans(L, momenta, n_mom, axis, out, max_out);
}

template <int NCLS, int NP, int RN>
__global__ void __launch_bounds__(kThreads, RN == 4 || NCLS >= 2 ? 1 : 2)
k_contract_fp64(const __grid_constant__ ContractParams prm) {
  rowsc::contract_rows<rowsc::ArithF64, NCLS, NP, kRowRM, RN>(prm, rowsc::TableSource<rowsc::ArithF64>{&prm});
}

template <int NCLS, int NP, int RN>
struct RowsF64 {
  static cudaError_t launch(const ContractParams& prm, int grid, cudaStream_t s) {
    const size_t smem = rows_smem_bytes(prm.L, prm.rows, RN, prm.n_groups, prm.xc);
    cudaError_t e = cudaFuncSetAttribute(k_contract_fp64<NCLS, NP, RN>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_contract_fp64<NCLS, NP, RN><<<grid, kThreads, smem, s>>>(prm);
    note_launch();
    return cudaGetLastError();
  }
};

cudaError_t launch_contract_fp64(const ContractParams& prm, int rn, int grid, cudaStream_t s) {
  if (prm.total_units == 0 || prm.rows.n_mom == 0) return cudaSuccess;
  return rowsc::launch_plan<RowsF64, kMaxSiteP>(prm, rn, prm, grid, s);
}

// ------------------------------------------------------------------ slab reduction

__global__ void k_reduce_slabs(const ContractJob* __restrict__ jobs, int n_slab, int P_total) {
  const ContractJob& J = jobs[blockIdx.y];
  const long long per = (long long)P_total * job_rows(J) * J.nd3;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < per;
       e += (long long)gridDim.x * blockDim.x) {
    double2 s = J.partial[e];
    // fixed order: the result is run-to-run identical; the loads of 8 slabs are in flight at once
#pragma unroll 8
    for (int sl = 1; sl < n_slab; ++sl) {
      const double2 v = J.partial[(size_t)sl * per + e];
      s.x += v.x;
      s.y += v.y;
    }
    J.B[e] = s;
  }
}

cudaError_t launch_reduce_slabs(const ContractJob* d_jobs, int n_jobs, int n_slab, int P_total,
                                long long max_elems, cudaStream_t s) {
  if (n_jobs == 0 || max_elems == 0) return cudaSuccess;
  long long bx = (max_elems + kThreads - 1) / kThreads;
  if (bx > 4096) bx = 4096;
  dim3 grid((unsigned)bx, n_jobs);
  k_reduce_slabs<<<grid, kThreads, 0, s>>>(d_jobs, n_slab, P_total);
  note_launch();
  return cudaGetLastError();
}

}  // namespace bb
