// Double-float form of the fused diquark + colour singlet + momentum projection (Eq. 1/3).
//
// GB300 executes IEEE double at 1/64 of the FP32 rate, and the FP64 contraction already
// runs at that pipe's roofline. This kernel computes the same sums in double-float
// arithmetic (dfloat.cuh: h + l, FP32 pairs, error-free products and sums, about 48
// significant bits) on the FP32 pipe, and converts to FP64 only the per-slab partial blocks a
// unit leaves, which the FP64 slab reduction sums in a fixed order.
//
// The body is rowsc::contract_rows (rows_contract.cuh) with each double replaced by a
// double-float of the same 8 bytes. Accumulators are renormalised once per chunk of sites, so
// their low parts never grow beyond a few ulp of the high parts.
#include "bblock_internal.h"
#include "rows_contract.cuh"

namespace bb {
namespace {

template <int NCLS, int NP, int RN>
__global__ void __launch_bounds__(kThreads, RN == 4 || NCLS >= 2 ? 1 : 2)
k_contract_df(const __grid_constant__ ContractParams prm) {
  rowsc::contract_rows<rowsc::ArithDf, NCLS, NP, kRowRM, RN>(prm, rowsc::TableSource<rowsc::ArithDf>{&prm});
}

template <int NCLS, int NP, int RN>
struct RowsDf {
  static cudaError_t launch(const ContractParams& prm, int grid, cudaStream_t s) {
    const size_t smem = rows_smem_bytes(prm.L, prm.rows, RN, prm.n_groups, prm.xc);
    cudaError_t e = cudaFuncSetAttribute(k_contract_df<NCLS, NP, RN>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_contract_df<NCLS, NP, RN><<<grid, kThreads, smem, s>>>(prm);
    note_launch();
    return cudaGetLastError();
  }
};

}  // namespace

cudaError_t launch_contract_df(const ContractParams& prm, int rn, int grid, cudaStream_t s) {
  if (prm.total_units == 0 || prm.rows.n_mom == 0) return cudaSuccess;
  return rowsc::launch_plan<RowsDf, kMaxSitePDf>(prm, rn, prm, grid, s);
}

}  // namespace bb
