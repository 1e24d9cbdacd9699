// The FP64 contraction body (fused diquark + colour singlet + momentum projection, Eq. 1/3,
// Algorithm 1's diq / singlet / phase steps) shared by the context path (k_contract_fp64)
// and the allocation-free entry point (bblock_contract_noalloc). The two differ only in
// where a unit's job, a field element and w^k come from, which a source policy supplies:
//   const ContractJob& job(long long u)             the job of work unit u
//   void uv(J, t, x, d1, d2, u[3], v[3])            line-1 and line-2 colour vectors of term t
//   double2 third(J, g, x, c, n)                    third quark of group g
//   double2 omega(int k)                            w^k = e^{-2 pi i k / L}
//
// Bound: the FP64 pipe (2 FMAs a clock and SM on GB300; every other instruction hides behind
// it), so the kernel executes as few FP64 instructions as the sums allow, per output element
// (d1, d2, d3) and site:
//   * 9 G for the colour singlet, G groups of spin terms that share a third-quark field
//     (GroupPlan; three-multiplication complex products, re = k1 - k3, im = k1 + k2 with
//     k1 = c(a+b), k2 = a(d-c), k3 = b(c+d), the operand sums formed when a tile is staged);
//   * 2 to recombine k1..k3, 2 for the momenta whose component n0 along the summed axis is 0
//     and 4 for every +-n0 class: e^{-ip.x} = w^{n0 x0} w^{n1 x1 + n2 x2}, a lattice row is
//     summed over x0 against each class first. With e = c + i s the four real sums c Sr, s Si,
//     c Si, s Sr give both signs: (c Sr -+ s Si) + i (c Si +- s Sr). Without a class
//     (RowPlan picks the axis with the fewest) k1..k3 run on over the whole row, unrecombined;
//   * 4 per momentum and row at the row's end, into the unit's partial block, which stays in
//     L2 (the read-modify-write is below 3 % of the L2 rate).
// (A singlet per spin pair and a phase product per momentum and site take 9 n_pairs + 2 + 4 P:
// 74 instead of 26 at 4 pairs, 2 groups and 9 momenta of n0 = 0, +-1.) Times: k_contract_fp64.
//
// Work unit = (job, slab of lattice rows, 16 RM (d1, d2) pairs, 16 RN d3 columns). Per chunk
// of XC sites of a row the CTA stages A[k][m] = diquark and B[k][n] = third quark with
// k = (site, group, colour); each thread owns RM x RN outputs. A wide d3 tile matters: the
// diquark costs 24 FP64 instructions per term, pair and site for all of the tile's columns.
#pragma once

#include "bblock_internal.h"

namespace bb {
namespace fp64c {

__device__ __forceinline__ int find_job(const ContractJob* jobs, int n_jobs, long long u) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].unit_begin <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// acc += a b - c d, complex
__device__ __forceinline__ void cross_add(double2& acc, double2 a, double2 b, double2 c, double2 d) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, fma(-c.x, d.x, fma(c.y, d.y, acc.x))));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, fma(-c.x, d.y, fma(-c.y, d.x, acc.y))));
}

template <int NCLS, int RM, int RN, class Src>
__device__ __forceinline__ void contract_rows(const ContractParams& prm, const Src& src) {
  constexpr int MT = 16 * RM, NT = 16 * RN;
  constexpr int NC = NCLS > 0 ? NCLS : 1;
  static_assert(kThreads % MT == 0, "a thread stages one row of the diquark tile");
  extern __shared__ __align__(16) double smem[];
  const RowPlan& rp = prm.rows;
  const int G = prm.n_groups, L = prm.L, XC = prm.xc;
  const int KC = XC * G * 3;
  double* __restrict__ Ar = smem;
  double* __restrict__ Ai = Ar + KC * MT;
  double* __restrict__ As = Ai + KC * MT;
  double* __restrict__ Bc = As + KC * MT;
  double* __restrict__ Bd = Bc + KC * NT;
  double* __restrict__ Be = Bd + KC * NT;
  double2* __restrict__ ph = reinterpret_cast<double2*>(Be + KC * NT);
  double2* __restrict__ om = ph + XC * NC;

  const int tid = threadIdx.x, tn = tid % 16, tm = tid / 16;
  const int ml = tid % MT;   // the diquark row this thread stages
  // sites of a row: base + x0 * sx along the summed axis
  const int sx = rp.axis == 0 ? 1 : rp.axis == 1 ? L : L * L;
  for (int k = tid; k < L; k += kThreads) om[k] = src.omega(k);
  __syncthreads();

  for (long long u = blockIdx.x; u < prm.total_units; u += gridDim.x) {
    const ContractJob& J = src.job(u);
    const int nd1 = J.nd1, nd2 = J.nd2, nd3 = J.nd3;
    const int M = nd1 * nd2;
    long long r = u - J.unit_begin;
    const int mt = (int)(r % J.m_tiles);
    r /= J.m_tiles;
    const int nt = (int)(r % J.n_tiles);
    const int slab = (int)(r / J.n_tiles);
    if (slab >= prm.n_slab) {  // inconsistent job table: flag it, skip the unit
      if (tid == 0 && prm.status) atomicOr(prm.status, kStatusBadJob);
      continue;
    }
    const int row_begin = slab * prm.rows_per_slab;
    const int row_end = min(L * L, row_begin + prm.rows_per_slab);
    const int ms = mt * MT + ml;
    const bool m_ok = ms < M;
    const int d1 = m_ok ? ms / nd2 : 0, d2 = m_ok ? ms - d1 * nd2 : 0;
    // 16-row and 16-column blocks of the tile that hold outputs: the others are skipped
    const int act_m = min(RM, (M - mt * MT + 15) / 16);
    const int act_n = min(RN, (nd3 - nt * NT + 15) / 16);
    const int n_cols = act_n * 16;

    for (int row = row_begin; row < row_end; ++row) {
      const int ra = row % L, rb = row / L;   // the other two coordinates, ascending
      const int base = rp.axis == 0 ? L * row : rp.axis == 1 ? ra + L * L * rb : row;
      double k1[RM][RN], k2[RM][RN], k3[RM][RN];
      double zr[RM][RN], zi[RM][RN];                       // n0 = 0
      double cr[RM][RN][NC], si_[RM][RN][NC], ci[RM][RN][NC], sr_[RM][RN][NC];   // +-n0 classes
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          k1[i][j] = k2[i][j] = k3[i][j] = zr[i][j] = zi[i][j] = 0.0;
#pragma unroll
          for (int c = 0; c < NC; ++c) cr[i][j][c] = si_[i][j][c] = ci[i][j][c] = sr_[i][j][c] = 0.0;
        }

      for (int x0 = 0; x0 < L; x0 += XC) {
        const int nx = min(XC, L - x0);
        // --- diquark tile: A[(xc, group, c)][m], the group's terms summed
        for (int xc = tid / MT; xc < nx; xc += kThreads / MT) {
          const int x = base + (x0 + xc) * sx;
          for (int g = 0; g < G; ++g) {
            double2 dq0 = make_double2(0.0, 0.0), dq1 = dq0, dq2 = dq0;
            if (m_ok) {
              for (int t = prm.tbeg[g]; t < prm.tbeg[g + 1]; ++t) {
                double2 uu[3], vv[3];
                src.uv(J, t, x, d1, d2, uu, vv);
                cross_add(dq0, uu[1], vv[2], uu[2], vv[1]);   // eps_{120}, eps_{210}
                cross_add(dq1, uu[2], vv[0], uu[0], vv[2]);   // eps_{201}, eps_{021}
                cross_add(dq2, uu[0], vv[1], uu[1], vv[0]);   // eps_{012}, eps_{102}
              }
            }
            const int k = (xc * G + g) * 3;
            Ar[(k + 0) * MT + ml] = dq0.x; Ai[(k + 0) * MT + ml] = dq0.y; As[(k + 0) * MT + ml] = dq0.x + dq0.y;
            Ar[(k + 1) * MT + ml] = dq1.x; Ai[(k + 1) * MT + ml] = dq1.y; As[(k + 1) * MT + ml] = dq1.x + dq1.y;
            Ar[(k + 2) * MT + ml] = dq2.x; Ai[(k + 2) * MT + ml] = dq2.y; As[(k + 2) * MT + ml] = dq2.x + dq2.y;
          }
        }
        // --- third quark tile: B[(xc, group, c)][n]
        for (int idx = tid; idx < nx * G * 3 * n_cols; idx += kThreads) {
          const int nl = idx % n_cols;
          const int k = idx / n_cols;
          const int c = k % 3, t2 = k / 3;
          const int g = t2 % G, xc = t2 / G;
          const int n = nt * NT + nl;
          double2 b = make_double2(0.0, 0.0);
          if (n < nd3) b = src.third(J, g, base + (x0 + xc) * sx, c, n);
          Bc[k * NT + nl] = b.x;
          Bd[k * NT + nl] = b.y - b.x;
          Be[k * NT + nl] = b.x + b.y;
        }
        if (NCLS > 0)
          for (int idx = tid; idx < nx * NCLS; idx += kThreads) {
            const int c = idx % NC, xc = idx / NC;
            ph[idx] = om[(rp.cls_n0[c] * (x0 + xc)) % L];
          }
        __syncthreads();

        for (int xc = 0; xc < nx; ++xc) {
          const int kbeg = xc * G * 3, kend = kbeg + G * 3;
#pragma unroll 3
          for (int k = kbeg; k < kend; ++k) {
            double ar[RM], ai[RM], as[RM], bc[RN], bd[RN], be[RN];
#pragma unroll
            for (int i = 0; i < RM; ++i) {
              ar[i] = Ar[k * MT + tm + 16 * i];
              ai[i] = Ai[k * MT + tm + 16 * i];
              as[i] = As[k * MT + tm + 16 * i];
            }
#pragma unroll
            for (int j = 0; j < RN; ++j) {
              bc[j] = Bc[k * NT + tn + 16 * j];
              bd[j] = Bd[k * NT + tn + 16 * j];
              be[j] = Be[k * NT + tn + 16 * j];
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < RN; ++j)
                if (i < act_m && j < act_n) {
                  k1[i][j] = fma(bc[j], as[i], k1[i][j]);
                  k2[i][j] = fma(ar[i], bd[j], k2[i][j]);
                  k3[i][j] = fma(ai[i], be[j], k3[i][j]);
                }
          }
          if (NCLS > 0) {
            double2 e[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) e[c] = ph[xc * NC + c];
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < RN; ++j)
                if (i < act_m && j < act_n) {
                  const double sr = k1[i][j] - k3[i][j], si = k1[i][j] + k2[i][j];
                  k1[i][j] = k2[i][j] = k3[i][j] = 0.0;
                  if (rp.has_zero) {
                    zr[i][j] += sr;
                    zi[i][j] += si;
                  }
#pragma unroll
                  for (int c = 0; c < NC; ++c) {
                    cr[i][j][c] = fma(e[c].x, sr, cr[i][j][c]);
                    si_[i][j][c] = fma(e[c].y, si, si_[i][j][c]);
                    ci[i][j][c] = fma(e[c].x, si, ci[i][j][c]);
                    sr_[i][j][c] = fma(e[c].y, sr, sr_[i][j][c]);
                  }
                }
          }
        }
        __syncthreads();
      }

      // --- the row's sums times w^{n1 x1 + n2 x2} into every momentum's partial block
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j)
          if (NCLS == 0) {
            zr[i][j] = k1[i][j] - k3[i][j];
            zi[i][j] = k1[i][j] + k2[i][j];
          }
      for (int q = 0; q < rp.n_mom; ++q) {
        const RowMom mo = rp.mom[q];
        const double2 e = om[(mo.n1 * ra + mo.n2 * rb) % L];
        double2* __restrict__ out = J.partial + ((size_t)slab * prm.P_total + mo.p) * M * nd3;
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          const int m = mt * MT + tm + 16 * i;
#pragma unroll
          for (int j = 0; j < RN; ++j) {
            const int n = nt * NT + tn + 16 * j;
            if (m < M && n < nd3) {
              double tr = zr[i][j], ti = zi[i][j];
#pragma unroll
              for (int c = 0; c < NCLS; ++c) {
                if (mo.sel == c + 1) { tr = cr[i][j][c] - si_[i][j][c]; ti = ci[i][j][c] + sr_[i][j][c]; }
                if (mo.sel == -c - 1) { tr = cr[i][j][c] + si_[i][j][c]; ti = ci[i][j][c] - sr_[i][j][c]; }
              }
              const size_t o = (size_t)m * nd3 + n;
              double2 v = make_double2(0.0, 0.0);
              if (row > row_begin) v = out[o];
              v.x = fma(e.x, tr, fma(-e.y, ti, v.x));
              v.y = fma(e.x, ti, fma(e.y, tr, v.y));
              out[o] = v;
            }
          }
        }
      }
    }
  }
}

}  // namespace fp64c
}  // namespace bb
