// Mode-triplet ordering of Eq. (3) (Sec. 2, Eq. 4): the baryon block as
//   B[p][d1][d2][d3] = sum_s c_s sum_{l1 l2 l3} T[p][l1][l2][l3]
//                      phi1[alpha_s N_ev + l1][d1] phi2[beta_s N_ev + l2][d2] phi3[gamma_s N_ev + l3][d3]
// with the eigenvector mode triplet
//   T[p][l1][l2][l3] = sum_x e^{-ip.x} eps_abc V[l1][x][a] V[l2][x][b] V[l3][x][c].
//
// T is the contraction of Eq. (1) with q_i = V, i.e. with identity coefficients
// (phi = [I; 0; 0; 0]) and the single spin triple (0, 0, 0): the host computes it with the
// contraction kernels of the context's form. T is totally antisymmetric in (l1, l2, l3), so the
// FP64 and double-float forms sum only the elements l1 < l2 < l3 (in tiles of 16 columns: about
// a fifth of all) and copy them with their signs:
//   k_tri_field       the fields q[r][l] = V[l][r] of the identity coefficients, a transposition
//   k_tri_fill        all n^3 elements of T from the ordered ones
// L = 24, N_ev = 96, 3 momenta, FP64: contraction 286 -> 51.2 ms (the ordered elements are a
// sixth), projection 5.9 -> 0.03 ms, k_tri_fill and the slab reduction 0.07 ms.
// For the second step:
//   k_fill_identity   the identity coefficient matrix [4 N_ev][N_ev]
//   k_fold_phi        phi' = sum_t w_t phi[spin_t N_ev + l][d]  (the spin coefficients of a group's
//                     third line or of a term's second line, as in the projection's fold)
//   k_zgemm           batched complex GEMM with arbitrary strides, FP64, for the three mode
//                     products T x3 phi3' (one per group of spin terms, the dominant one),
//                     x2 phi2' (one per term) and x1 phi1 (summed over the terms)
#include "bblock_internal.h"
#include "dfloat.cuh"

namespace bb {
namespace {

__global__ void k_fill_identity(double2* __restrict__ id, int n_ev) {
  const long long total = 4LL * n_ev * n_ev;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / n_ev, c = i - r * n_ev;
    id[i] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
}

__global__ void k_fold_phi(const __grid_constant__ FoldBatch fb) {
  const FoldTerms& terms = fb.fold[blockIdx.y];
  const int nd = terms.nd;
  const long long total = (long long)fb.n_ev * nd;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long l = i / nd, d = i - l * nd;
    double re = 0.0, im = 0.0;
    for (int t = 0; t < terms.n; ++t) {
      const double2 f = terms.phi[((long long)terms.row[t] * fb.n_ev + l) * nd + d];
      const double2 w = terms.w[t];
      re = fma(w.x, f.x, fma(-w.y, f.y, re));
      im = fma(w.x, f.y, fma(w.y, f.x, im));
    }
    terms.out[i] = make_double2(re, im);
  }
}

// field[r][l] = V[l][r] by 32 x 32 tiles through shared memory (both sides 512-byte runs): one
// read and one write of V, bound by HBM.
template <bool DF>
__global__ void __launch_bounds__(256) k_tri_field(const TriSlice* __restrict__ slices, int n,
                                                   int rows) {
  __shared__ double2 tile[32][33];
  const TriSlice S = slices[blockIdx.z];
  const int r0 = blockIdx.x * 32, l0 = blockIdx.y * 32;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int i = ty; i < 32; i += 8) {
    const int l = l0 + i, r = r0 + tx;
    double2 v = make_double2(0.0, 0.0);
    if (l < n && r < rows) v = S.V[(size_t)l * rows + r];
    tile[i][tx] = v;
    if (!isfinite(v.x) || !isfinite(v.y)) S.bad[l] = 1;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int r = r0 + i, l = l0 + tx;
    if (r >= rows || l >= n) continue;
    const double2 v = tile[tx][i];
    if (DF) {
      const dcomplex z = dc_from_double2(v);
      reinterpret_cast<float4*>(S.field)[(size_t)r * n + l] = make_float4(z.re.h, z.re.l, z.im.h, z.im.l);
    } else {
      S.field[(size_t)r * n + l] = v;
    }
  }
}

// One thread per element (p, l1, l2, l3), l3 fastest: the ordered element with the sign of the
// permutation; zero on repeated indices (not a number where a vector is not finite, as the
// products of the sum itself are).
__global__ void k_tri_fill(const TriSlice* __restrict__ slices, int n, int n_mom) {
  const TriSlice S = slices[blockIdx.y];
  const long long total = (long long)n_mom * n * n * n;
  const long long M = (long long)n * (n - 1) / 2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int l3 = (int)(e % n);
    long long q = e / n;
    const int l2 = (int)(q % n);
    q /= n;
    const int l1 = (int)(q % n), p = (int)(q / n);
    double2 v;
    if (l1 == l2 || l2 == l3 || l1 == l3) {
      const double z = S.bad[l1] | S.bad[l2] | S.bad[l3] ? nan("") : 0.0;
      v = make_double2(z, z);
    } else {
      int a = l1, b = l2, c = l3;
      double sgn = 1.0;
      if (a > b) { const int t = a; a = b; b = t; sgn = -sgn; }
      if (b > c) { const int t = b; b = c; c = t; sgn = -sgn; }
      if (a > b) { const int t = a; a = b; b = t; sgn = -sgn; }
      const double2 w = S.compact[((size_t)p * M + (size_t)b * (b - 1) / 2 + a) * n + c];
      v = make_double2(sgn * w.x, sgn * w.y);
    }
    S.T[e] = v;
  }
}

// Complex GEMMs of the three mode products, FP64, bound by the FP64 pipe. Four multiplications to a
// complex one: the form with three (re = k1 - k3, im = k1 + k2) takes 1.74 instead of 2.12 ms for the
// case below, but leaves each part accurate to the modulus only, and over three products in a row
// the error grew from 1.13e-15 to 1.32e-15. The products of a list are summed from zero each and
// then added, 9.8e-16 (in one chain 1.18e-15). The row tile is the one that wastes fewer rows:
// 64 (T x3 phi3, thousands of rows), or 32 (the products over N_dil rows, half of a 64-row tile
// idle at N_dil = 32). L = 24, N_ev = 96, N_dil = 32, 3 momenta, 3 pairs / 2 gammas, all products of
// one time slice: 3.63 ms with a product per pair, 2.12 with one per group (1.8 of FP64 operations).
constexpr int ZBK = 16, ZRN = 4, ZBN = 8 * ZRN;

template <int RM, bool SUM>
__global__ void __launch_bounds__(kThreads) k_zgemm(const __grid_constant__ ZgemmParams p) {
  constexpr int BM = 32 * RM;
  __shared__ double2 As[ZBK][BM], Bs[ZBK][ZBN];
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * ZBN;
  const long long bt = blockIdx.z % p.batch;
  const int l0 = SUM ? 0 : (int)(blockIdx.z / p.batch), l1 = SUM ? p.n_list : l0 + 1;
  double2* __restrict__ C = p.C[l0] + bt * p.c_b;
  const int tid = threadIdx.x, tn = tid % 8, tm = tid / 8;
  double re[RM][ZRN], im[RM][ZRN];
  double sr[RM][ZRN], si[RM][ZRN];   // SUM: of the list's products, each summed from zero
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < ZRN; ++j) re[i][j] = im[i][j] = sr[i][j] = si[i][j] = 0.0;

  for (int l = l0; l < l1; ++l) {
    const double2* __restrict__ A = p.A[l] + bt * p.a_b;
    const double2* __restrict__ B = p.B[l] + bt * p.b_b;
    for (int k0 = 0; k0 < p.K; k0 += ZBK) {
      for (int idx = tid; idx < ZBK * BM; idx += kThreads) {
        // neighbouring threads along A's unit stride
        const int r = p.a_k == 1 ? idx / ZBK : idx % BM, kk = p.a_k == 1 ? idx % ZBK : idx / BM;
        const int m = m0 + r, k = k0 + kk;
        double2 v = make_double2(0.0, 0.0);
        if (m < p.M && k < p.K) v = A[(long long)m * p.a_m + (long long)k * p.a_k];
        As[kk][r] = v;
      }
      for (int idx = tid; idx < ZBK * ZBN; idx += kThreads) {
        const int c = idx % ZBN, kk = idx / ZBN;
        const int n = n0 + c, k = k0 + kk;
        double2 v = make_double2(0.0, 0.0);
        if (n < p.N && k < p.K) v = B[(long long)k * p.b_k + (long long)n * p.b_n];
        Bs[kk][c] = v;
      }
      __syncthreads();
      const int kn = min(ZBK, p.K - k0);
#pragma unroll 4
      for (int kk = 0; kk < kn; ++kk) {
        double2 a[RM], b[ZRN];
#pragma unroll
        for (int i = 0; i < RM; ++i) a[i] = As[kk][tm + 32 * i];
#pragma unroll
        for (int j = 0; j < ZRN; ++j) b[j] = Bs[kk][tn + 8 * j];
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
          for (int j = 0; j < ZRN; ++j) {
            re[i][j] = fma(a[i].x, b[j].x, fma(-a[i].y, b[j].y, re[i][j]));
            im[i][j] = fma(a[i].x, b[j].y, fma(a[i].y, b[j].x, im[i][j]));
          }
      }
      __syncthreads();
    }
    if (SUM) {
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < ZRN; ++j) {
          sr[i][j] += re[i][j];
          si[i][j] += im[i][j];
          re[i][j] = im[i][j] = 0.0;
        }
    }
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int m = m0 + tm + 32 * i;
    if (m >= p.M) continue;
#pragma unroll
    for (int j = 0; j < ZRN; ++j) {
      const int n = n0 + tn + 8 * j;
      if (n >= p.N) continue;
      double2& c = C[(long long)m * p.c_m + (long long)n * p.c_n];
      double2 r = SUM ? make_double2(sr[i][j], si[i][j]) : make_double2(re[i][j], im[i][j]);
      if (p.accumulate) { r.x += c.x; r.y += c.y; }
      c = r;
    }
  }
}

int grid_for(long long total) {
  long long g = (total + kThreads - 1) / kThreads;
  return (int)(g < 1 ? 1 : (g > 65536 ? 65536 : g));
}

}  // namespace

cudaError_t launch_fill_identity(double2* id, int n_ev, cudaStream_t s) {
  k_fill_identity<<<grid_for(4LL * n_ev * n_ev), kThreads, 0, s>>>(id, n_ev);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_tri_field(const TriSlice* d_slices, int n_slices, int n, int rows, bool df,
                             cudaStream_t s) {
  for (int z0 = 0; z0 < n_slices; z0 += 65535) {  // grid.z limit
    const dim3 grid((rows + 31) / 32, (n + 31) / 32, n_slices - z0 < 65535 ? n_slices - z0 : 65535);
    if (df) k_tri_field<true><<<grid, 256, 0, s>>>(d_slices + z0, n, rows);
    else k_tri_field<false><<<grid, 256, 0, s>>>(d_slices + z0, n, rows);
    note_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_tri_fill(const TriSlice* d_slices, int n_slices, int n, int n_mom,
                            cudaStream_t s) {
  const int bx = grid_for((long long)n_mom * n * n * n);
  for (int y0 = 0; y0 < n_slices; y0 += 65535) {  // grid.y limit
    const dim3 grid(bx, n_slices - y0 < 65535 ? n_slices - y0 : 65535);
    k_tri_fill<<<grid, kThreads, 0, s>>>(d_slices + y0, n, n_mom);
    note_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_fold_phi(const FoldBatch& fb, cudaStream_t s) {
  if (fb.n == 0) return cudaSuccess;
  int nd = 1;
  for (int k = 0; k < fb.n; ++k) nd = fb.fold[k].nd > nd ? fb.fold[k].nd : nd;
  k_fold_phi<<<dim3(grid_for((long long)fb.n_ev * nd), fb.n), kThreads, 0, s>>>(fb);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_zgemm(const ZgemmParams& p, cudaStream_t s) {
  if (p.M <= 0 || p.N <= 0 || p.batch <= 0 || p.n_list <= 0) return cudaSuccess;
  const int per = p.sum_list ? 1 : p.n_list;
  const long long step = 65535 / per;            // grid.z limit
  const bool half = (p.M + 31) / 32 % 2 == 1 && p.M < 1024;
  for (long long b0 = 0; b0 < p.batch; b0 += step) {
    ZgemmParams q = p;
    for (int l = 0; l < p.n_list; ++l) {
      q.A[l] += b0 * p.a_b;
      q.B[l] += b0 * p.b_b;
    }
    for (int l = 0; l < per; ++l) q.C[l] += b0 * p.c_b;
    q.batch = (int)(p.batch - b0 < step ? p.batch - b0 : step);
    const int bm = half ? 32 : 64;
    const dim3 grid((p.M + bm - 1) / bm, (p.N + ZBN - 1) / ZBN, q.batch * per);
    (p.sum_list ? half ? k_zgemm<1, true> : k_zgemm<2, true>
                : half ? k_zgemm<1, false> : k_zgemm<2, false>)<<<grid, kThreads, 0, s>>>(q);
    note_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace bb
