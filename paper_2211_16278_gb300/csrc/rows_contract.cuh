// The contraction body (fused diquark + colour singlet + momentum projection, Eq. 1/3,
// Algorithm 1's diq / singlet / phase steps) of the FP64 form (k_contract_fp64), the
// double-float form (k_contract_df) and the allocation-free entry point
// (bblock_contract_noalloc). An arithmetic policy (ArithF64, ArithDf) supplies the numbers, a
// source policy where a unit's job, a field element and w^k come from:
//   const ContractJob& job(long long u)             the job of work unit u
//   void uv(J, t, x, d1, d2, u[3], v[3])            line-1 and line-2 colour vectors of term t
//   Cx third(J, g, x, c, n)                         third quark of group g
//   Cx omega(int k)                                 w^k = e^{-2 pi i k / L}
//
// Bound: the arithmetic pipe (2 FP64 FMAs, or 128 FP32 instructions, a clock and SM on GB300;
// in the FP64 form every other instruction hides behind them), so the kernel executes as few
// operations as the sums allow, per output element (d1, d2, d3) and site:
//   * 9 G for the colour singlet, G groups of spin terms that share a third-quark field
//     (ContractParams::tbeg; three-multiplication complex products, re = k1 - k3,
//     im = k1 + k2 with k1 = c(a+b), k2 = a(d-c), k3 = b(c+d), the operand sums formed when a
//     tile is staged);
//   * 2 to recombine k1..k3, 2 for the momenta whose component n0 along the summed axis is 0
//     and 4 for every +-n0 class: e^{-ip.x} = w^{n0 x0} w^{n1 x1 + n2 x2}, a lattice row is
//     summed over x0 against each class first. With e = c + i s the four real sums c Sr, s Si,
//     c Si, s Sr give both signs: (c Sr -+ s Si) + i (c Si +- s Sr). Without a class
//     (RowPlan picks the axis with the fewest) k1..k3 run on over the whole row, unrecombined
//     (FP64; in double-float the longer sums of the larger k's cost accuracy, 4.2e-14 against
//     2.7e-14 at L = 24, so each site is recombined, 4 operations);
//   * 4 per momentum and row at the row's end, into the unit's partial block, which stays in
//     L2 (the read-modify-write is below 3 % of the L2 rate in the FP64 form);
//   * or, for lists whose momenta hardly share an n0 (plan_rows), a phase per momentum and site
//     (NP of them): 2 to recombine, then 4 for every momentum, into sums that stay in registers
//     over a run of sites; runs meet in the unit's partial block as rows do, which keeps the error
//     at the row-factored one's. (With sums over all 216 sites of a unit at L = 24, 8 momenta, it was
//     1.08 times that in FP64 and 1.3 to 1.5 times in double-float, now 1.00 and 0.99; double-float
//     takes 10 to 16 % longer for it, FP64 2 %.)
// (A singlet per spin pair and a phase product per momentum and site take 9 n_pairs + 2 + 4 P:
// 74 instead of 26 at 4 pairs, 2 groups and 9 momenta of n0 = 0, +-1.) Times: k_contract_fp64,
// k_contract_df.
//
// Work unit = (job, slab of lattice rows or, with a phase per site, of sites, 16 RM (d1, d2) pairs,
// 16 RN d3 columns). Per chunk of XC sites the CTA stages A[k][m] = diquark and B[k][n] = third quark with
// k = (site, group, colour); each thread owns RM x RN outputs. A wide d3 tile matters: the
// diquark costs 24 operations per term, pair and site for all of the tile's columns.
#pragma once

#include <type_traits>

#include "bblock_internal.h"
#include "dfloat.cuh"

namespace bb {
namespace rowsc {

__device__ __forceinline__ int find_job(const ContractJob* jobs, int n_jobs, long long u) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].unit_begin <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// IEEE double on the FP64 pipe. T: a number, Cx: a complex number, Z: its 16 bytes in memory.
struct ArithF64 {
  static constexpr bool kEachSite = false;   // recombine k1..k3 at each site also without a class
  static constexpr bool kExactP = false;     // a site loop of its own for each momentum count (NP)
  static constexpr int kSiteRun = 24;        // a phase per site: sites of a run (whole chunks)
  static constexpr int kNormSites = 1 << 30; // and between renormalisations within a chunk
  using T = double;
  struct Cx { double re, im; };
  using Z = double2;
  __device__ static T zero() { return 0.0; }
  __device__ static void fma_add(T& acc, T a, T b) { acc = fma(a, b, acc); }
  __device__ static void fma_sub(T& acc, T a, T b) { acc = fma(-a, b, acc); }
  __device__ static T add(T a, T b) { return a + b; }
  __device__ static T sub(T a, T b) { return a - b; }
  __device__ static T norm(T a) { return a; }
  __device__ static T norm_site(T a) { return a; }
  __device__ static void site_add(Cx& acc, Cx e, Cx s) {   // acc += e s
    fma_add(acc.re, e.re, s.re);
    fma_sub(acc.re, e.im, s.im);
    fma_add(acc.im, e.re, s.im);
    fma_add(acc.im, e.im, s.re);
  }
  __device__ static Cx load(const Z* p) { const double2 v = *p; return Cx{v.x, v.y}; }
  __device__ static Cx cx(double2 v) { return Cx{v.x, v.y}; }
  __device__ static void store(Z* p, Cx v) { *p = make_double2(v.re, v.im); }
  __device__ static double2 to_double2(Cx v) { return make_double2(v.re, v.im); }
};

// Double-float pairs on the FP32 pipe (12 instructions per multiply-add), low parts collected
// lazily: norm() brings them back below ulp(h) / 2.
struct ArithDf {
  static constexpr bool kEachSite = true;
  static constexpr bool kExactP = true;
  static constexpr int kSiteRun = 64;
  static constexpr int kNormSites = 2;
  using T = dfloat;
  using Cx = dcomplex;
  using Z = float4;
  __device__ static T zero() { return df_zero(); }
  __device__ static void fma_add(T& acc, T a, T b) { df_fma(acc, a, b); }
  __device__ static void fma_sub(T& acc, T a, T b) { df_fms(acc, a, b); }
  __device__ static T add(T a, T b) { return df_add(a, b); }
  __device__ static T sub(T a, T b) { return df_sub(a, b); }
  __device__ static T norm(T a) { return df_norm(a); }
  __device__ static T norm_site(T a) { return df_norm_quick(a); }
  // The product first: as many instructions as two multiply-adds into the sum, which then takes
  // one rounding of its low part instead of two.
  __device__ static void site_add(Cx& acc, Cx e, Cx s) {
    Cx t{df_mul(e.re, s.re), df_mul(e.re, s.im)};
    df_fms(t.re, e.im, s.im);
    df_fma(t.im, e.im, s.re);
    acc.re = df_add(acc.re, t.re);
    acc.im = df_add(acc.im, t.im);
  }
  __device__ static Cx load(const Z* p) {
    const float4 v = *p;
    return Cx{dfloat{v.x, v.y}, dfloat{v.z, v.w}};
  }
  __device__ static Cx cx(double2 v) { return dc_from_double2(v); }
  __device__ static void store(Z* p, Cx v) { *p = make_float4(v.re.h, v.re.l, v.im.h, v.im.l); }
  __device__ static double2 to_double2(Cx v) {
    return make_double2(df_to_double(v.re), df_to_double(v.im));
  }
};

// acc += a b (complex)
template <class A> __device__ __forceinline__ void cmul_add(typename A::Cx& acc, typename A::Cx a, typename A::Cx b) {
  A::fma_add(acc.re, a.re, b.re);
  A::fma_sub(acc.re, a.im, b.im);
  A::fma_add(acc.im, a.re, b.im);
  A::fma_add(acc.im, a.im, b.re);
}
// acc += a b - c d (complex)
template <class A>
__device__ __forceinline__ void cross_add(typename A::Cx& acc, typename A::Cx a, typename A::Cx b,
                                          typename A::Cx c, typename A::Cx d) {
  A::fma_add(acc.re, c.im, d.im);
  A::fma_sub(acc.re, c.re, d.re);
  A::fma_sub(acc.re, a.im, b.im);
  A::fma_add(acc.re, a.re, b.re);
  A::fma_sub(acc.im, c.im, d.re);
  A::fma_sub(acc.im, c.re, d.im);
  A::fma_add(acc.im, a.im, b.re);
  A::fma_add(acc.im, a.re, b.im);
}

// The context's job table, projected fields and cached w^k.
template <class A> struct TableSource {
  using Cx = typename A::Cx;
  using Z = typename A::Z;
  static constexpr bool kRowParts = false;   // slabs are whole rows
  const ContractParams* prm;
  __device__ const ContractJob& job(long long u) const {
    return prm->jobs[find_job(prm->jobs, prm->n_jobs, u)];
  }
  __device__ void uv(const ContractJob& J, int t, int x, int d1, int d2, Cx (&u)[3],
                     Cx (&v)[3]) const {
    const Z* a = reinterpret_cast<const Z*>(J.q1[prm->a_slot[t]]) + (size_t)x * 3 * J.nd1 + d1;
    const Z* b = reinterpret_cast<const Z*>(J.q2[prm->b_slot[t]]) + (size_t)x * 3 * J.nd2 + d2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = A::load(a + c * J.nd1);
      v[c] = A::load(b + c * J.nd2);
    }
  }
  __device__ Cx third(const ContractJob& J, int g, int x, int c, int n) const {
    return A::load(reinterpret_cast<const Z*>(J.q3[g]) + ((size_t)x * 3 + c) * J.nd3 + n);
  }
  __device__ Cx omega(int k) const { return A::cx(prm->phase[k]); }
};

// f(integral_constant n), n in [LO, HI]
template <int LO, int HI, class F> __device__ __forceinline__ void with_count(int n, F&& f) {
  if constexpr (LO < HI) {
    if (n <= LO) f(std::integral_constant<int, LO>{});
    else with_count<LO + 1, HI>(n, f);
  } else {
    f(std::integral_constant<int, HI>{});
  }
}

template <class A, int NCLS, int NP, int RM, int RN, class Src>
__device__ __forceinline__ void contract_rows(const ContractParams& prm, const Src& src) {
  static_assert(NCLS == 0 || NP == 0, "row-factored or a phase per site");
  constexpr int MT = 16 * RM, NT = 16 * RN;
  constexpr int NC = NCLS > 0 ? NCLS : 1;
  constexpr int NPS = NP > 0 ? NP : 1;
  constexpr int NPH = NCLS + NP > 0 ? NCLS + NP : 1;   // phases of a site
  using T = typename A::T;
  using Cx = typename A::Cx;
  using Z = typename A::Z;
  static_assert(sizeof(T) == 8 && sizeof(Z) == 16, "tiles and partial blocks of every arithmetic");
  static_assert(kThreads % MT == 0, "a thread stages one row of the diquark tile");
  extern __shared__ __align__(16) double2 smem_rows[];
  const RowPlan& rp = prm.rows;
  const int G = prm.n_groups, L = prm.L, XC = prm.xc;
  const int KC = XC * G * 3;
  T* __restrict__ Ar = reinterpret_cast<T*>(smem_rows);
  T* __restrict__ Ai = Ar + KC * MT;
  T* __restrict__ As = Ai + KC * MT;
  T* __restrict__ Bc = As + KC * MT;
  T* __restrict__ Bd = Bc + KC * NT;
  T* __restrict__ Be = Bd + KC * NT;
  Z* __restrict__ ph = reinterpret_cast<Z*>(Be + KC * NT);
  Z* __restrict__ om = ph + XC * (NP > kSitePNarrow ? kMaxSiteP : NPH);

  const int tid = threadIdx.x, tn = tid % 16, tm = tid / 16;
  const int ml = tid % MT;   // the diquark row this thread stages
  // sites of a row: base + x0 * sx along the summed axis
  const int run = max(1, A::kSiteRun / XC) * XC;   // sites of a run (a phase per site)
  const int sx = NP > 0 || rp.axis == 0 ? 1 : rp.axis == 1 ? L : L * L;
  for (int k = tid; k < L; k += kThreads) A::store(om + k, src.omega(k));
  __syncthreads();

  for (long long u = blockIdx.x; u < prm.total_units; u += gridDim.x) {
    const ContractJob& J = src.job(u);
    const int nd2 = J.nd2, nd3 = J.nd3;
    const int M = job_rows(J);
    long long r = u - J.unit_begin;
    const int mt = (int)(r % J.m_tiles);
    r /= J.m_tiles;
    const int nt = (int)(r % J.n_tiles);
    const int slab = (int)(r / J.n_tiles);
    if (slab >= prm.n_slab) {  // inconsistent job table: flag it, skip the unit
      if (tid == 0 && prm.status) atomicOr(prm.status, kStatusBadJob);
      continue;
    }
    // the tile's first column: with triangular rows (m = (l1, l2), l1 < l2, ordered by l2) only
    // the 16-column blocks that hold an l3 > l2 of the tile's first row are needed
    const int col0 = (J.tri ? (tri_l2(mt * MT) + 1) / 16 * 16 : 0) + nt * NT;
    if (col0 >= nd3) continue;
    // a slab of rows, or, of small lattices, one run of sites of a row
    int row_begin = slab * prm.rows_per_slab, row_end = min(L * L, row_begin + prm.rows_per_slab);
    int x_begin = 0, x_end = L;
    if (NP > 0) {   // a phase per site: a slab of sites, in the lattice's own order
      row_begin = 0;
      row_end = 1;
      x_begin = slab * prm.sites_per_slab;
      x_end = min(prm.X, x_begin + prm.sites_per_slab);
    } else if (Src::kRowParts && prm.row_parts > 1) {
      const int len = (L + prm.row_parts - 1) / prm.row_parts;
      row_begin = slab / prm.row_parts;
      row_end = row_begin + 1;
      x_begin = min(L, (slab - row_begin * prm.row_parts) * len);
      x_end = min(L, x_begin + len);
    }
    const int ms = mt * MT + ml;
    const bool m_ok = ms < M;
    int d1 = 0, d2 = 0;
    if (m_ok && J.tri) {
      d2 = tri_l2(ms);
      d1 = ms - d2 * (d2 - 1) / 2;
    } else if (m_ok) {
      d1 = ms / nd2;
      d2 = ms - d1 * nd2;
    }
    // 16-column blocks of the tile that hold outputs
    const int act_n = min(RN, (nd3 - col0 + 15) / 16);
    const int n_cols = act_n * 16;

    T wr[RM][RN][NPS], wi[RM][RN][NPS];   // the run's sums of each momentum (a phase per site)
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j)
#pragma unroll
        for (int c = 0; c < NPS; ++c) wr[i][j][c] = wi[i][j][c] = A::zero();

    for (int row = row_begin; row < row_end; ++row) {
      const int ra = row % L, rb = row / L;   // the other two coordinates, ascending
      const int base = NP > 0 ? 0 : rp.axis == 0 ? L * row : rp.axis == 1 ? ra + L * L * rb : row;
      T k1[RM][RN], k2[RM][RN], k3[RM][RN];
      T zr[RM][RN], zi[RM][RN];                                          // n0 = 0
      T cr[RM][RN][NC], si_[RM][RN][NC], ci[RM][RN][NC], sr_[RM][RN][NC];   // +-n0 classes
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          k1[i][j] = k2[i][j] = k3[i][j] = zr[i][j] = zi[i][j] = A::zero();
#pragma unroll
          for (int c = 0; c < NC; ++c) cr[i][j][c] = si_[i][j][c] = ci[i][j][c] = sr_[i][j][c] = A::zero();
        }

      auto add_sites = [&](auto act, auto n_site, int nx) {
        constexpr int ACT = decltype(act)::value, NS = decltype(n_site)::value;   // NS: of NP
        for (int xc = 0; xc < nx; ++xc) {
          const int kbeg = xc * G * 3, kend = kbeg + G * 3;
#pragma unroll 3
          for (int k = kbeg; k < kend; ++k) {
            T ar[RM], ai[RM], as[RM], bc[RN], bd[RN], be[RN];
#pragma unroll
            for (int i = 0; i < RM; ++i) {
              ar[i] = Ar[k * MT + tm + 16 * i];
              ai[i] = Ai[k * MT + tm + 16 * i];
              as[i] = As[k * MT + tm + 16 * i];
            }
#pragma unroll
            for (int j = 0; j < ACT; ++j) {
              bc[j] = Bc[k * NT + tn + 16 * j];
              bd[j] = Bd[k * NT + tn + 16 * j];
              be[j] = Be[k * NT + tn + 16 * j];
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < ACT; ++j) {
                A::fma_add(k1[i][j], bc[j], as[i]);
                A::fma_add(k2[i][j], ar[i], bd[j]);
                A::fma_add(k3[i][j], ai[i], be[j]);
              }
          }
          if (NCLS == 0 && NP == 0 && A::kEachSite) {
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < ACT; ++j) {
                zr[i][j] = A::add(zr[i][j], A::sub(k1[i][j], k3[i][j]));
                zi[i][j] = A::add(zi[i][j], A::add(k1[i][j], k2[i][j]));
                k1[i][j] = k2[i][j] = k3[i][j] = A::zero();
              }
          }
          if (NP > 0) {
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < ACT; ++j) {
                const T sr = A::sub(k1[i][j], k3[i][j]);
                k2[i][j] = A::add(k1[i][j], k2[i][j]);
                k1[i][j] = sr;
              }
#pragma unroll
            for (int c = 0; c < NS; ++c) {
              if (!A::kExactP && c >= rp.n_mom) break;
              const Cx e = A::load(ph + xc * NPH + c);
#pragma unroll
              for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < ACT; ++j) {
                  Cx w{wr[i][j][c], wi[i][j][c]};
                  A::site_add(w, e, Cx{k1[i][j], k2[i][j]});
                  wr[i][j][c] = w.re;
                  wi[i][j][c] = w.im;
                }
            }
            if (xc % A::kNormSites == A::kNormSites - 1) {
#pragma unroll
              for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < ACT; ++j)
#pragma unroll
                  for (int c = 0; c < NS; ++c) {
                    wr[i][j][c] = A::norm_site(wr[i][j][c]);
                    wi[i][j][c] = A::norm_site(wi[i][j][c]);
                  }
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < ACT; ++j) k1[i][j] = k2[i][j] = k3[i][j] = A::zero();
          }
          if (NCLS > 0) {
            Cx e[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) e[c] = A::load(ph + xc * NC + c);
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < ACT; ++j) {
                  const T sr = A::sub(k1[i][j], k3[i][j]), si = A::add(k1[i][j], k2[i][j]);
                  k1[i][j] = k2[i][j] = k3[i][j] = A::zero();
                  if (rp.has_zero) {
                    zr[i][j] = A::add(zr[i][j], sr);
                    zi[i][j] = A::add(zi[i][j], si);
                  }
#pragma unroll
                  for (int c = 0; c < NC; ++c) {
                    A::fma_add(cr[i][j][c], e[c].re, sr);
                    A::fma_add(si_[i][j][c], e[c].im, si);
                    A::fma_add(ci[i][j][c], e[c].re, si);
                    A::fma_add(sr_[i][j][c], e[c].im, sr);
                  }
                }
          }
        }
      };

      for (int x0 = x_begin; x0 < x_end; x0 += XC) {   // a row: [0, L) without parts
        const int nx = min(XC, x_end - x0);
        // --- diquark tile: A[(xc, group, c)][m], the group's terms summed
        for (int xc = tid / MT; xc < nx; xc += kThreads / MT) {
          const int x = base + (x0 + xc) * sx;
          for (int g = 0; g < G; ++g) {
            Cx dq[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) dq[c] = Cx{A::zero(), A::zero()};
            if (m_ok) {
              for (int t = prm.tbeg[g]; t < prm.tbeg[g + 1]; ++t) {
                Cx uu[3], vv[3];
                src.uv(J, t, x, d1, d2, uu, vv);
                cross_add<A>(dq[0], uu[1], vv[2], uu[2], vv[1]);   // eps_{120}, eps_{210}
                cross_add<A>(dq[1], uu[2], vv[0], uu[0], vv[2]);   // eps_{201}, eps_{021}
                cross_add<A>(dq[2], uu[0], vv[1], uu[1], vv[0]);   // eps_{012}, eps_{102}
              }
            }
            const int k = (xc * G + g) * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const T re = A::norm(dq[c].re), im = A::norm(dq[c].im);
              Ar[(k + c) * MT + ml] = re;
              Ai[(k + c) * MT + ml] = im;
              As[(k + c) * MT + ml] = A::norm(A::add(re, im));
            }
          }
        }
        // --- third quark tile: B[(xc, group, c)][n]
        for (int idx = tid; idx < nx * G * 3 * n_cols; idx += kThreads) {
          const int nl = idx % n_cols;
          const int k = idx / n_cols;
          const int c = k % 3, t2 = k / 3;
          const int g = t2 % G, xc = t2 / G;
          const int n = col0 + nl;
          Cx b{A::zero(), A::zero()};
          if (n < nd3) b = src.third(J, g, base + (x0 + xc) * sx, c, n);
          Bc[k * NT + nl] = b.re;
          Bd[k * NT + nl] = A::norm(A::sub(b.im, b.re));
          Be[k * NT + nl] = A::norm(A::add(b.re, b.im));
        }
        if (NCLS > 0)
          for (int idx = tid; idx < nx * NCLS; idx += kThreads) {
            const int c = idx % NC, xc = idx / NC;
            ph[idx] = om[(rp.cls_n0[c] * (x0 + xc)) % L];
          }
        if (NP > 0)
          for (int idx = tid; idx < nx * NP; idx += kThreads) {
            const int c = idx % NPS, xc = idx / NPS;
            if (c >= rp.n_mom) continue;
            const RowMom mo = rp.mom[c];
            const int x = x0 + xc, xr = x / L;
            ph[idx] = om[(mo.sel * (x - xr * L) + mo.n1 * (xr % L) + mo.n2 * (xr / L)) % L];
          }
        __syncthreads();

        // the staged sites into the sums, by the tile's 16-column blocks in use: a block that is
        // only predicated off still takes the FP64 pipe (measured: 96 columns cost 128)
        with_count<1, RN>(act_n, [&](auto act) {
          if constexpr (NP > 0 && A::kExactP)
            with_count<(NP > kSitePNarrow ? kSitePNarrow + 1 : 1), NP>(rp.n_mom, [&](auto n) { add_sites(act, n, nx); });
          else
            add_sites(act, std::integral_constant<int, NP>{}, nx);
        });
        // renormalise once per chunk of sites
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
          for (int j = 0; j < RN; ++j) {
            zr[i][j] = A::norm(zr[i][j]);
            zi[i][j] = A::norm(zi[i][j]);
#pragma unroll
            for (int c = 0; c < NCLS; ++c) {
              cr[i][j][c] = A::norm(cr[i][j][c]);
              si_[i][j][c] = A::norm(si_[i][j][c]);
              ci[i][j][c] = A::norm(ci[i][j][c]);
              sr_[i][j][c] = A::norm(sr_[i][j][c]);
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) {
              wr[i][j][c] = A::norm(wr[i][j][c]);
              wi[i][j][c] = A::norm(wi[i][j][c]);
            }
          }
        __syncthreads();
        // --- a phase per site: the run's sums into the partial blocks, in FP64 after the last
        if (NP > 0 && ((x0 + nx - x_begin) % run == 0 || x0 + nx >= x_end)) {
#pragma unroll
          for (int c = 0; c < NP; ++c) {
            if (c >= rp.n_mom) break;
            Z* __restrict__ out =
                reinterpret_cast<Z*>(J.partial) + ((size_t)slab * prm.P_total + rp.mom[c].p) * M * nd3;
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
              for (int j = 0; j < RN; ++j) {
                const int m = mt * MT + tm + 16 * i, n = col0 + tn + 16 * j;
                if (m < M && n < nd3) {
                  const size_t o = (size_t)m * nd3 + n;
                  Cx v{wr[i][j][c], wi[i][j][c]};
                  if (x0 - x_begin >= run) {
                    const Cx t = A::load(out + o);
                    v = Cx{A::norm(A::add(t.re, v.re)), A::norm(A::add(t.im, v.im))};
                  }
                  if (x0 + nx < x_end) A::store(out + o, v);
                  else reinterpret_cast<double2*>(out)[o] = A::to_double2(v);
                }
                wr[i][j][c] = wi[i][j][c] = A::zero();
              }
          }
        }
      }

      // --- the row's sums times w^{n1 x1 + n2 x2} into every momentum's partial block
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j)
          if (NCLS == 0 && NP == 0 && !A::kEachSite) {
            zr[i][j] = A::norm(A::sub(k1[i][j], k3[i][j]));
            zi[i][j] = A::norm(A::add(k1[i][j], k2[i][j]));
          }
      for (int q = 0; NP == 0 && q < rp.n_mom; ++q) {
        const RowMom mo = rp.mom[q];
        const Cx e = A::load(om + (mo.n1 * ra + mo.n2 * rb) % L);
        // the unit's own sums until its last row, which leaves them in FP64
        Z* __restrict__ out =
            reinterpret_cast<Z*>(J.partial) + ((size_t)slab * prm.P_total + mo.p) * M * nd3;
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          const int m = mt * MT + tm + 16 * i;
#pragma unroll
          for (int j = 0; j < RN; ++j) {
            const int n = col0 + tn + 16 * j;
            if (m < M && n < nd3) {
              Cx t{zr[i][j], zi[i][j]};
#pragma unroll
              for (int c = 0; c < NCLS; ++c) {
                if (mo.sel == c + 1)
                  t = Cx{A::sub(cr[i][j][c], si_[i][j][c]), A::add(ci[i][j][c], sr_[i][j][c])};
                if (mo.sel == -c - 1)
                  t = Cx{A::add(cr[i][j][c], si_[i][j][c]), A::sub(ci[i][j][c], sr_[i][j][c])};
              }
              t.re = A::norm(t.re);
              t.im = A::norm(t.im);
              const size_t o = (size_t)m * nd3 + n;
              Cx v{A::zero(), A::zero()};
              if (row > row_begin) v = A::load(out + o);
              cmul_add<A>(v, e, t);
              if (row + 1 < row_end) {
                v.re = A::norm(v.re);
                v.im = A::norm(v.im);
                A::store(out + o, v);
              } else {
                reinterpret_cast<double2*>(out)[o] = A::to_double2(v);
              }
            }
          }
        }
      }
    }
  }
}

// The launch of Kernel<NCLS, NP, RN> for a plan; WIDE: momenta of the widest per-site launch.
template <template <int, int, int> class Kernel, int WIDE, class Params>
cudaError_t launch_plan(const ContractParams& c, int rn, const Params& prm, int grid, cudaStream_t s) {
  const RowPlan& r = c.rows;
  // a chunk and a slab of the plan's kind, and tiles that it has
  if (c.xc < 1 || (r.per_site ? c.sites_per_slab : c.rows_per_slab) < 1 || rn > rows_max_rn(r))
    return cudaErrorInvalidValue;
  if (r.per_site) {
    if (r.n_mom > WIDE) return cudaErrorInvalidValue;
    if (r.n_mom > kSitePNarrow) return Kernel<0, WIDE, 1>::launch(prm, grid, s);
    return rn == 1 ? Kernel<0, kSitePNarrow, 1>::launch(prm, grid, s)
                   : Kernel<0, kSitePNarrow, 2>::launch(prm, grid, s);
  }
  switch (r.n_cls * 8 + rn) {
    case 0 + 1: return Kernel<0, 0, 1>::launch(prm, grid, s);
    case 0 + 2: return Kernel<0, 0, 2>::launch(prm, grid, s);
    case 0 + 4: return Kernel<0, 0, 4>::launch(prm, grid, s);
    case 8 + 1: return Kernel<1, 0, 1>::launch(prm, grid, s);
    case 8 + 2: return Kernel<1, 0, 2>::launch(prm, grid, s);
    case 8 + 4: return Kernel<1, 0, 4>::launch(prm, grid, s);
    case 16 + 1: return Kernel<2, 0, 1>::launch(prm, grid, s);
    case 16 + 2: return Kernel<2, 0, 2>::launch(prm, grid, s);
    case 24 + 1: return Kernel<3, 0, 1>::launch(prm, grid, s);
    case 24 + 2: return Kernel<3, 0, 2>::launch(prm, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rowsc
}  // namespace bb
