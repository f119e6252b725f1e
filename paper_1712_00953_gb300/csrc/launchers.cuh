// Definitions of the per-cell kernel launches declared in device.cuh.  Only
// the k_*.cu translation units include this header, each explicitly
// instantiating its share, so every heavy kernel is compiled exactly once.
#pragma once
#include "device.cuh"

namespace rk {

// Persistent ROK4E launch: as many cells per block as shared memory allows
// (or a.cells_per_block), one wave of blocks sized to the device.
template <int G, bool MIXED, bool TC, int THREADS>
int launch_rok4e_kernel(const IntegrateLaunch& a) {
  IntegrateParams& P = *a.P;
  LaunchPlan plan;
  const int rc =
      plan_for<G>(rok4e_integrate_kernel<G, MIXED, TC, THREADS>, a.mech, P.S, a.cells_per_block, a.ncell, true, &plan,
                  a.blocks_per_sm, a.static_bins, P.mech_copy + P.fx_copy + P.tc_bytes, THREADS);
  if (rc) return rc;
  if (a.static_bins) P.subq = plan.cells_per_block % 4 == 0 ? 4 : (plan.cells_per_block % 2 == 0 ? 2 : 1);
  rok4e_integrate_kernel<G, MIXED, TC, THREADS>
      <<<plan.blocks, plan.cells_per_block * G, plan.smem, a.stream>>>(P);
  return RK_OK;
}
template <int THREADS>
int launch_rok4e_wide(const IntegrateLaunch& a) {
  return launch_rok4e_kernel<32, false, false, THREADS>(a);
}

extern template int launch_rok4e_wide<384>(const IntegrateLaunch&);
extern template int launch_rok4e_wide<512>(const IntegrateLaunch&);

// FP64 cells one to a warp: an attempt is a chain of dependent instructions that
// leaves its sub-partition idle a third of the time with two warps on it, so more
// cells to an SM finish more of them, each with fewer registers (168 with up to
// twelve warps, 128 with sixteen; 0 and 400 bytes of spills).  How many fit is the
// mechanism's size: ten at 53 species / 325 reactions (12288 cells, two steps: 177
// ms with eight, 165 with ten), sixteen at 10 / 24 (20001 cells: 287 and 210 ms).  With few cells for each SM the step lasts as long as its
// slowest cells, which run fastest on eight warps.
inline int rok4e_threads(const IntegrateLaunch& a) {
  const IntegrateParams& P = *a.P;
  int n_sm = 0;
  size_t smem_max = 0;
  if (device_props(&n_sm, &smem_max) != RK_OK) return MAX_BLOCK_THREADS;
  const int64_t room = (int64_t)smem_max - 64 - EXP_TAB_BYTES - P.mech_copy - P.fx_copy;
  int64_t cells = room / ((int64_t)P.S.stride * 8);
  if (a.cells_per_block > 0 && a.cells_per_block < cells) cells = a.cells_per_block;
  if (cells <= 8 || a.ncell < (int64_t)WIDE_MIN_CELLS_PER_SM * n_sm) return MAX_BLOCK_THREADS;
  return cells <= 12 ? 384 : 512;
}

template <int G, bool MIXED, bool TC>
int launch_rok4e(const IntegrateLaunch& a) {
  if constexpr (G == 32 && !MIXED && !TC) {
    const int threads = rok4e_threads(a);
    if (threads == 384) return launch_rok4e_wide<384>(a);
    if (threads == 512) return launch_rok4e_wide<512>(a);
  }
  return launch_rok4e_kernel<G, MIXED, TC, MAX_BLOCK_THREADS>(a);
}

// Persistent explicit Dormand-Prince launch, planned like ROK4E's.
template <int G>
int launch_rkdp(const IntegrateLaunch& a) {
  IntegrateParams& P = *a.P;
  LaunchPlan plan;
  const int rc = plan_for<G>(rkdp_integrate_kernel<G>, a.mech, P.S, a.cells_per_block, a.ncell, true, &plan,
                             a.blocks_per_sm, a.static_bins, P.mech_copy + P.fx_copy, rkdp_threads(G));
  if (rc) return rc;
  if (a.static_bins) P.subq = plan.cells_per_block % 4 == 0 ? 4 : (plan.cells_per_block % 2 == 0 ? 2 : 1);
  rkdp_integrate_kernel<G><<<plan.blocks, plan.cells_per_block * G, plan.smem, a.stream>>>(P);
  return RK_OK;
}

// The adjoint: 128-thread blocks of 128 / G cell slots, the mechanism in
// shared memory; enough blocks for one slot per cell, at most as many as the
// device holds at once (the cells are then dealt over them in turn).  Filling
// every resident slot instead, with some warps holding one or two cells,
// measured 28 % slower on 4096 cells at 8 lanes.
template <int G>
int launch_adjoint(const AdjointParams& P, size_t smem, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(rok4e_adjoint_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute");
  int n_sm = 0;
  size_t smem_max = 0;
  const int rc = device_props(&n_sm, &smem_max);
  if (rc) return rc;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rok4e_adjoint_kernel<G>, 128, smem);
  if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  if (per_sm < 1) return set_error(RK_E_UNSUPPORTED, "adjoint kernel cannot be resident on an SM");
  const int64_t resident = (int64_t)per_sm * n_sm;
  const int64_t need = (P.ncell * G + 127) / 128;
  const int64_t blocks = need < resident ? need : resident;
  rok4e_adjoint_kernel<G><<<(unsigned)blocks, 128, smem, st>>>(P);
  return RK_OK;
}

}  // namespace rk
