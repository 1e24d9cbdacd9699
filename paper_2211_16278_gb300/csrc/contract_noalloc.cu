// bblock_contract_noalloc: the FP64 contraction (fused diquark + colour singlet + momentum
// projection, then the fixed-order slab reduction) for callers that cannot allocate device
// memory. Its per-slab partial sums live in one file-scope __device__ array instead of a
// context workspace, so the entry point needs no context and calls no allocator.
#include <cstdio>
#include <mutex>

#include "../../include/bblock.h"
#include "bblock_internal.h"
#include "rows_contract.cuh"

namespace bb {
namespace {

// Fixed scratch for the per-slab partial blocks. Every device that loads the library
// holds this array for the life of the process.
constexpr size_t kNoallocScratchBytes = (size_t)BBLOCK_NOALLOC_SCRATCH_BYTES;
static __device__ __align__(256) double2 g_noalloc_scratch[kNoallocScratchBytes / sizeof(double2)];

constexpr int kNaMaxP = 8;
constexpr int kNaMaxDevices = 64;

// One folded field element: sum_t w[t] f[spin[t]], by the launch's spin coefficients.
struct NaFold {
  int n;
  int spin[kMaxTerms];
  double2 w[kMaxTerms];
};

// The launch: the shared FP64 contraction body's parameters (one job, embedded below; no
// status word) plus what this entry point takes instead of a context's tables. The spin sum is
// grouped as in the context (ContractParams::tbeg); a_slot is the line-1 spin, and the folds
// that the context's projection applies are taken while a tile is staged.
struct NoallocParams {
  ContractParams base;    // jobs = nullptr, status = nullptr, P_total = P
  ContractJob job;        // q1 slots = spins 0..3 of the caller's array; partial = scratch
  const double2* q2;      // [4][X][3][nd2]
  const double2* q3;      // [4][X][3][nd3]
  NaFold f2[kMaxPairs];   // line-2 element of term t
  NaFold f3[kMaxPairs];   // line-3 element of group g
};

// Where the shared body's inputs come from without a context: the single job of the launch,
// the spin coefficients folded while the tile is staged, and w^k by sincospi.
struct NoallocSource {
  using Cx = rowsc::ArithF64::Cx;
  static constexpr bool kRowParts = true;
  const NoallocParams* np;
  __device__ const ContractJob& job(long long) const { return np->job; }
  __device__ static double2 fold(const NaFold& f, const double2* q, size_t spin_stride, size_t at) {
    if (f.n == 1 && f.w[0].x == 1.0 && f.w[0].y == 0.0) return q[f.spin[0] * spin_stride + at];
    double2 b = make_double2(0.0, 0.0);
    for (int t = 0; t < f.n; ++t) {
      const double2 v = q[f.spin[t] * spin_stride + at];
      const double2 w = f.w[t];
      b.x = fma(w.x, v.x, fma(-w.y, v.y, b.x));
      b.y = fma(w.x, v.y, fma(w.y, v.x, b.y));
    }
    return b;
  }
  __device__ void uv(const ContractJob& J, int t, int x, int d1, int d2, Cx (&u)[3],
                     Cx (&v)[3]) const {
    const double2* a = J.q1[np->base.a_slot[t]] + (size_t)x * 3 * J.nd1 + d1;
    const size_t b = (size_t)x * 3 * J.nd2 + d2, st = (size_t)np->base.X * 3 * J.nd2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = rowsc::ArithF64::load(a + c * J.nd1);
      v[c] = rowsc::ArithF64::cx(fold(np->f2[t], np->q2, st, b + c * J.nd2));
    }
  }
  __device__ Cx third(const ContractJob& J, int g, int x, int c, int n) const {
    return rowsc::ArithF64::cx(fold(np->f3[g], np->q3, (size_t)np->base.X * 3 * J.nd3,
                                    ((size_t)x * 3 + c) * J.nd3 + n));
  }
  __device__ Cx omega(int k) const {
    double sn, cs;
    sincospi(2.0 * (double)k / (double)np->base.L, &sn, &cs);
    return Cx{cs, -sn};
  }
};

template <int NCLS, int NP, int RN>
__global__ void __launch_bounds__(kThreads, RN == 4 || NCLS >= 2 ? 1 : 2)
k_contract_fp64_noalloc(const __grid_constant__ NoallocParams prm) {
  rowsc::contract_rows<rowsc::ArithF64, NCLS, NP, kRowRM, RN>(prm.base, NoallocSource{&prm});
}

// B[e] = sum over slabs of partial[slab][e]: LANES threads per element take runs of the slabs, in
// index order, with the loads of 8 in flight, then their sums in order. A small call has many slabs
// of few elements, one long chain of loads at one thread per element (L = 6, N_dil 14, 11, 9, 5
// momenta, 72 slabs: the call takes 72.3 us with 1 thread, 62.6 with 8).
template <int LANES>
__global__ void k_reduce_noalloc(const double2* __restrict__ partial, double2* __restrict__ B,
                                 long long per, int n_slab) {
  constexpr int E = kThreads / LANES;   // elements of a block at a time
  __shared__ double2 sums[LANES][E];
  const int le = threadIdx.x % E, lane = threadIdx.x / E;
  const int run = (n_slab + LANES - 1) / LANES;
  const int s0 = min(n_slab, lane * run), s1 = min(n_slab, s0 + run);
  for (long long e0 = blockIdx.x * (long long)E; e0 < per; e0 += (long long)gridDim.x * E) {
    const long long e = e0 + le;
    double2 s = make_double2(0.0, 0.0);
    if (e < per) {
#pragma unroll 8
      for (int sl = s0; sl < s1; ++sl) {
        const double2 v = partial[(size_t)sl * per + e];
        s.x += v.x;
        s.y += v.y;
      }
    }
    if (LANES > 1) {
      sums[lane][le] = s;
      __syncthreads();
      if (lane == 0) {
#pragma unroll
        for (int k = 1; k < LANES; ++k) {
          s.x += sums[k][le].x;
          s.y += sums[k][le].y;
        }
      }
      __syncthreads();
    }
    if (lane == 0 && e < per) B[e] = s;
  }
}

template <int NCLS, int NP, int RN>
struct RowsNoalloc {
  static cudaError_t launch(const NoallocParams& prm, int grid, cudaStream_t s) {
    const size_t smem = rows_smem_bytes(prm.base.L, prm.base.rows, RN, prm.base.n_groups, prm.base.xc);
    cudaError_t e = cudaFuncSetAttribute(k_contract_fp64_noalloc<NCLS, NP, RN>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_contract_fp64_noalloc<NCLS, NP, RN><<<grid, kThreads, smem, s>>>(prm);
    note_launch();
    return cudaGetLastError();
  }
};

// Per-device device address of g_noalloc_scratch. In host code the array's name stands
// for a host-side shadow, not device memory, so the address must be looked up with
// cudaGetSymbolAddress once per device while that device is current.
std::mutex g_na_mu;
void* g_na_addr[kNaMaxDevices] = {};
void* g_na_ctx[kNaMaxDevices] = {};   // the CUDA context each address was looked up in

// The calling thread's current CUDA context (driver API, reached through the runtime's
// entry-point query so that the library needs no link against libcuda), or nullptr.
void* na_current_context() {
  typedef int (*CtxGetCurrentFn)(void**);
  static CtxGetCurrentFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<CtxGetCurrentFn>(f);
    else
      cudaGetLastError();
  }
  void* ctx = nullptr;
  if (fn && fn(&ctx) != 0) ctx = nullptr;
  return ctx;
}

int na_fail(char* err, size_t err_len, int code, const char* msg) {
  if (err && err_len) snprintf(err, err_len, "%s", msg);
  return code;
}

bool na_device_ptr(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == dev);
}

}  // namespace
}  // namespace bb

using namespace bb;

extern "C" int bblock_contract_noalloc(int L, const void* q1, const void* q2, const void* q3,
                                       int nd1, int nd2, int nd3, const int32_t* momenta,
                                       int n_mom, const int32_t* spin_idx,
                                       const double* spin_coeffs, int n_spin, void* B_out,
                                       void* stream, char* err, size_t err_len) {
  if (err && err_len) err[0] = '\0';
  if (L < 1 || L > 128) return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "L outside 1..128");
  if (nd1 < 1 || nd2 < 1 || nd3 < 1 || nd1 > 256 || nd2 > 256 || nd3 > 256)
    return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "dilution sizes must be 1..256");
  if (n_mom < 0 || n_mom > kNaMaxP)
    return na_fail(err, err_len, BBLOCK_ERR_TOO_LARGE, "n_mom must be 0..8 for this entry point");
  if (n_spin < 1 || n_spin > 64 || !spin_idx || !spin_coeffs || (n_mom > 0 && !momenta))
    return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "bad momentum or spin arguments");
  if (n_mom == 0) return BBLOCK_OK;
  if (!q1 || !q2 || !q3 || !B_out)
    return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "a data pointer is NULL");
  const void* ptrs[4] = {q1, q2, q3, B_out};
  for (const void* p : ptrs)
    if ((reinterpret_cast<uintptr_t>(p) & 15u) != 0)
      return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "a data pointer is not 16-byte aligned");

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) {
    cudaGetLastError();
    return na_fail(err, err_len, BBLOCK_ERR_CUDA, "no usable current CUDA device");
  }
  for (const void* p : ptrs)
    if (!na_device_ptr(p, dev))
      return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG,
                     "q1, q2, q3 and B_out must be device memory of the current device");

  NoallocParams prm{};
  ContractParams& base = prm.base;
  ContractJob& job = prm.job;
  const int X = L * L * L;
  // the q1 slots are the four spins of the caller's array
  for (int a = 0; a < 4; ++a)
    job.q1[a] = static_cast<const double2*>(q1) + (size_t)a * X * 3 * nd1;
  job.nd1 = nd1; job.nd2 = nd2; job.nd3 = nd3;
  job.unit_begin = 0;
  prm.q2 = static_cast<const double2*>(q2);
  prm.q3 = static_cast<const double2*>(q3);
  base.L = L;
  base.X = X;
  base.n_jobs = 1;
  base.P_total = n_mom;
  // spin triples -> coefficients by (alpha, beta, gamma), then the groups: one per
  // (alpha, beta) pair with the coefficients in its third quark, or, where that makes fewer,
  // one per gamma with a term per alpha and the coefficients in its line-2 element
  double2 coef[4][4][4] = {};
  bool have[4][4][4] = {};
  for (int s = 0; s < n_spin; ++s) {
    const int al = spin_idx[3 * s], be = spin_idx[3 * s + 1], ga = spin_idx[3 * s + 2];
    if (al < 0 || al > 3 || be < 0 || be > 3 || ga < 0 || ga > 3)
      return na_fail(err, err_len, BBLOCK_ERR_INVALID_ARG, "spin index outside 0..3");
    have[al][be][ga] = true;
    coef[al][be][ga].x += spin_coeffs[2 * s];
    coef[al][be][ga].y += spin_coeffs[2 * s + 1];
  }
  const double2 one = make_double2(1.0, 0.0);
  auto push = [](NaFold& f, int spin, double2 w) { f.spin[f.n] = spin; f.w[f.n++] = w; };
  int n_pairs = 0, n_gamma = 0;
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) {
      bool any = false, g_any = false;
      for (int g = 0; g < 4; ++g) any = any || have[a][b][g];
      for (int i = 0; i < 16; ++i) g_any = g_any || have[i / 4][i % 4][b];
      n_pairs += any;
      if (a == 0) n_gamma += g_any;
    }
  if (n_gamma < n_pairs) {
    for (int g = 0; g < 4; ++g) {
      const int t0 = base.n_terms;
      for (int a = 0; a < 4; ++a) {
        NaFold f{};
        for (int b = 0; b < 4; ++b)
          if (have[a][b][g]) push(f, b, coef[a][b][g]);
        if (f.n == 0) continue;
        base.a_slot[base.n_terms] = a;
        prm.f2[base.n_terms++] = f;
      }
      if (base.n_terms == t0) continue;
      push(prm.f3[base.n_groups], g, one);
      base.tbeg[++base.n_groups] = base.n_terms;
    }
  } else {
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b) {
        NaFold f{};
        for (int g = 0; g < 4; ++g)
          if (have[a][b][g]) push(f, g, coef[a][b][g]);
        if (f.n == 0) continue;
        base.a_slot[base.n_terms] = a;
        push(prm.f2[base.n_terms++], b, one);
        prm.f3[base.n_groups] = f;
        base.tbeg[++base.n_groups] = base.n_terms;
      }
  }

  RowPlan plans[kNaMaxP];
  const int n_plans = plan_rows(L, momenta, n_mom, base.n_groups, base.n_terms, nd3, false, ROWS_AUTO, plans, kNaMaxP);
  const int rn = rows_rn_for(plans, n_plans, nd3);
  job.m_tiles = (nd1 * nd2 + 16 * kRowRM - 1) / (16 * kRowRM);
  job.n_tiles = (nd3 + 16 * rn - 1) / (16 * rn);
  const size_t per = (size_t)n_mom * nd1 * nd2 * nd3;
  const size_t max_slabs_fit = kNoallocScratchBytes / (per * sizeof(double2));
  if (max_slabs_fit < 1)
    return na_fail(err, err_len, BBLOCK_ERR_TOO_LARGE,
                   "n_mom*nd1*nd2*nd3*16 bytes exceeds the static scratch of this entry point");

  // set-up once per device and CUDA context: the device address of the static scratch
  // (looked up again if the device's context was reset and recreated since)
  {
    std::lock_guard<std::mutex> lock(g_na_mu);
    void* ctx = na_current_context();
    if (!g_na_addr[dev] || ctx != g_na_ctx[dev]) {
      void* addr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
      if (e != cudaSuccess || !addr) {
        cudaGetLastError();
        return na_fail(err, err_len, BBLOCK_ERR_CUDA, "cudaGetSymbolAddress of the scratch failed");
      }
      g_na_addr[dev] = addr;
      g_na_ctx[dev] = ctx;
    }
    job.partial = static_cast<double2*>(g_na_addr[dev]);
  }

  int num_sms = 0;
  if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return na_fail(err, err_len, BBLOCK_ERR_CUDA, "device query failed");
  }
  const long long tiles = (long long)job.m_tiles * job.n_tiles;
  // Slabs of lattice rows, at most what the scratch holds: the count with the least work on the
  // busiest SM (the FP64 pipe is shared by an SM's CTAs, so only its units count), in operations
  // of the contraction per output: 9 per group and 4 per class of a site, 6 per momentum of a
  // row's end. With 12 slabs allowed and 32 tiles (L = 16, N_dil = 32, 5 momenta) 12 would put 3
  // units of 22 rows on some SMs, 9 put 2 of 29: 9.64 -> 8.36 ms. Where single rows are too coarse
  // for the SMs, rows are divided into runs of sites, each with a row's end of its own (L = 6,
  // N_dil 14, 11, 9, 5 momenta: contraction 63.5 -> 57.8 us).
  // Among equals, the count with the least work one after another: an SM's resident CTAs take the
  // latencies side by side.
  const int n_rows = L * L;
  const long long resident = (long long)rows_ctas_per_sm(plans[0], rn) * num_sms;
  const int per_mom = plans[0].per_site ? plans[0].n_mom : plans[0].n_cls;
  const long long site_ops = 9 * base.n_groups + 4 + 4 * per_mom, row_ops = 6 * n_mom;
  long long best = -1, best_chain = 0;
  auto consider = [&](long long slabs, long long cost, long long work, int rps, int parts, int sites) {
    const long long chain = (tiles * slabs + resident - 1) / resident * work;
    if (best < 0 || cost < best || (cost == best && chain < best_chain)) {
      best = cost;
      best_chain = chain;
      base.rows_per_slab = rps;
      base.row_parts = parts;
      base.sites_per_slab = sites;
      base.n_slab = (int)slabs;
    }
    return slabs * tiles < 8LL * num_sms;   // finer slabs gain nothing more
  };
  auto on_busiest = [&](long long slabs) { return (tiles * slabs + num_sms - 1) / num_sms; };
  const long long most = (long long)max_slabs_fit;
  bool finer = true;
  const int xc = site_chunk(L, base.n_groups, tiles, resident);
  if (plans[0].per_site) {
    // slabs of staged chunks of sites; a unit's start and end cost about 4 sites, and an uneven last
    // round leaves some SMs with a unit more than others (measured: L = 12, N_dil = 32, 6 momenta,
    // one pair, 448 units on 304 CTAs 11 % slower than 576)
    const int chunks = (X + xc - 1) / xc;
    for (long long n = 1; finer && n <= most && n <= chunks; ++n) {
      const int sites = (int)((chunks + n - 1) / n) * xc;
      const long long slabs = (X + sites - 1) / sites, work = (sites + 4) * site_ops;
      const long long rounds = (tiles * slabs + resident - 1) / resident;
      finer = consider(slabs, (3 * on_busiest(slabs) + resident / num_sms * rounds) * work, work, 0, 1, sites);
    }
  } else {
    for (long long n = 1; finer && n <= most && n <= n_rows; ++n) {
      const int rps = (int)((n_rows + n - 1) / n);
      const long long slabs = (n_rows + rps - 1) / rps, work = rps * (L * site_ops + row_ops);
      finer = consider(slabs, on_busiest(slabs) * work, work, rps, 1, rps * L);
    }
    for (int parts = 2; finer && parts <= L && (long long)n_rows * parts <= most; ++parts) {
      const long long slabs = (long long)n_rows * parts, work = (L + parts - 1) / parts * site_ops + row_ops;
      finer = consider(slabs, on_busiest(slabs) * work, work, 1, parts, L);
    }
  }
  base.total_units = tiles * base.n_slab;

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < n_plans && e == cudaSuccess; ++k) {
    base.rows = plans[k];
    base.xc = plans[k].per_site ? xc : rows_sites_per_chunk(L, plans[k], rn, base.n_groups);
    const long long cap = (long long)rows_ctas_per_sm(plans[k], rn) * num_sms;
    e = rowsc::launch_plan<RowsNoalloc, kNaMaxP>(base, rn, prm, (int)(base.total_units < cap ? base.total_units : cap), s);
  }
  if (e == cudaSuccess) {
    const int lanes = base.n_slab >= 16 ? 8 : 1;
    long long bx = ((long long)per * lanes + kThreads - 1) / kThreads;
    if (bx > 4096) bx = 4096;
    (lanes == 8 ? k_reduce_noalloc<8> : k_reduce_noalloc<1>)<<<(unsigned)bx, kThreads, 0, s>>>(
        job.partial, static_cast<double2*>(B_out), (long long)per, base.n_slab);
    note_launch();
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    if (err && err_len) snprintf(err, err_len, "launch failed: %s", cudaGetErrorString(e));
    return BBLOCK_ERR_CUDA;
  }
  return BBLOCK_OK;
}
