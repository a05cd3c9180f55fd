// Kernel instantiations for PrecF32.
#include "lbm_launch_impl.cuh"

namespace lbm {
// Whether two steps per launch take less time than two launches.  They do not
// below 2^22 nodes, whose populations are not far from fitting L2 (2048 x 1024,
// three species: 79 us per step with one step per launch, 89 with two; 1000 x
// 900: 48 and 47), nor for one species (4096 x 2048: 113 and 127), and the kernel
// numbers the populations of all species with 32 bits.  Beyond that the kernel
// pays for whole strips and waves of runs, the one-step kernel for nodes, so the
// line lies at a cost of the plan per node: 1.99e-5 for three species, 1.88e-5
// for two, a tenth more where the one-step kernel has 64-thread blocks (padding),
// which take longer per node.  us per step of three species with one step per
// launch and two, and the cost in 1e-5:
//   16384 x 4096  2327  1690  1.49    2048 x 2048   159  167  2.09
//   8192 x 8192   2342  1718  1.51    224 x 19000   203  209  2.11
//   16384 x 1024   592   516  1.60    430 x 10000   192  213  2.18
//   4096 x 2048    300   287  1.80    1280 x 3300   166  184  2.20
//   140000 x 32    156   131  1.69    1020 x 4200   170  194  2.28
//   2032 x 2100    163   152  1.90    510 x 8300    177  234  2.66
//   508 x 8300     177   191  1.90    256 x 16500   200  293  3.40
//   3000 x 1500    169   175  1.91   and with 64-thread blocks
//   1020 x 16000   613   623  1.94    600 x 14000   393  362  2.11
//   4096 x 1100    167   159  1.97    350 x 24000   398  423  2.38
// (two species: 4096 x 2048 203 and 196, 2048 x 4096 203 and 213, 1.89).  On 58
// such lattices, some with thin fibers everywhere or periodic, the form taken is
// the slower one by at most 8% (508 x 8300), 0.2% in the mean.
bool two_step_pays(int prec, int ns, int nx, int ny) {
  const long long plane = pad32(nx) * ny;
  if (prec != LBM_F32 || ns < 2 || plane < (1ll << 22) || 9 * ns * plane >= (1ll << 32))
    return false;
  const double per_node =
      two_step_plan(nx, ny, TwoStep<2>::kOwned, TwoStep<2>::kBlocks).cost / ((double)nx * ny);
  const int nx_pad = static_cast<int>(pad32(nx));
  const double line = ns == 2 ? 1.88e-5 : 1.99e-5;
  return per_node < (adr_block_x(prec, nx_pad, ny) == 64 ? 1.1 * line : line);
}

template <int NS>
static cudaError_t two_step_ns(const AdrArgs &a, cudaStream_t st) {
  using K = TwoStep<NS>;
  cudaError_t e = cudaFuncSetAttribute(adr_two_step_kernel<NS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, K::kShared);
  if (e != cudaSuccess) return e;
  const int rows = two_step_plan(a.nx, a.ny, K::kOwned, K::kBlocks).rows;
  const dim3 grid((a.nx + K::kOwned - 1) / K::kOwned, (a.ny + rows - 1) / rows);
  adr_two_step_kernel<NS><<<grid, K::kBX, K::kShared, st>>>(a, rows);
  return cudaGetLastError();
}
cudaError_t launch_adr_two_step(int ns, const AdrArgs &a, cudaStream_t st) {
  switch (ns) {
    case 2: return two_step_ns<2>(a, st);
    case 3: return two_step_ns<3>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_adr<PrecF32>(int, int, const AdrArgs &,
                                            cudaStream_t, bool);
template cudaError_t launch_adr_flux<PrecF32>(int, const void *, const RefT *,
                                                 const uint32_t *, long long,
                                                 int, int, int, double *,
                                                 cudaStream_t);
template cudaError_t launch_flow<PrecF32>(int, const FlowArgs &, cudaStream_t,
                                          bool);
template cudaError_t launch_adjoint<PrecF32>(int, int, const AdjArgs &,
                                                cudaStream_t, bool);
template cudaError_t launch_adjoint_grad<PrecF32>(
    int, const AdjArgs &, const BoundaryNode *, long long, const void *, double *,
    double *, const int32_t *, double *, double, double, cudaStream_t);
}  // namespace lbm
