// Kernel instantiations for PrecF32.
#include "lbm_launch_impl.cuh"

namespace lbm {
// Whether two steps per launch take less time than two launches.  They do not
// below 2^22 nodes, whose populations are not far from fitting L2 (2048 x 1024,
// three species: 79 us per step with one step per launch, 89 with two; 1000 x
// 900: 48 and 47), nor for one species (4096 x 2048: 130 and 127), and the kernel
// numbers the populations of all species with 32 bits.  Beyond that the kernel
// pays for whole strips and waves of runs, the one-step kernel for nodes, so the
// line lies at a cost of the plan per node; about 40% higher where the one-step
// kernel has 64-thread blocks (padding), which take that much longer per node.
// us per step of three species, one step per launch (unchained: 2% less in a
// run of them) and two (cost / line):
//   16384 x 4096  2326  1680 (0.74)    2048 x 2048   158  166 (1.03)
//   8192 x 8192   2342  1705 (0.75)    224 x 19000   221  209 (1.04)
//   4096 x 2048    309   286 (0.89)    430 x 10000   199  213 (1.08)
//   2048 x 4096    317   306 (0.93)    1020 x 4200   169  193 (1.13)
//   140000 x 32    160   131 (0.93)    510 x 8300    180  234 (1.32)
//   2032 x 2100    162   151 (0.94)    256 x 16500   213  292 (1.68)
//   508 x 8300     180   190 (0.94)   and where the one-step kernel has 64-
//   3000 x 1500    169   173 (0.95)   thread blocks
//   1020 x 16000   659   621 (0.96)    300 x 60000  1100  979 (0.89)
//   4096 x 1100    167   158 (0.97)    160 x 27000   309  269 (0.96)
//                                      300 x 14500   264  275 (1.02)
// Of 47 such lattices, two and three species, the form taken is the slower one
// by at most 8% (10% with chained steps, 508 x 8300) and by 0.3% in the mean.
bool two_step_pays(int prec, int ns, int nx, int ny) {
  const long long plane = pad32(nx) * ny;
  if (prec != LBM_F32 || ns < 2 || plane < (1ll << 22) || 9 * ns * plane >= (1ll << 32))
    return false;
  const int nx_pad = static_cast<int>(pad32(nx));
  const double per_node =
      two_step_plan(nx, ny, TwoStep<2>::kOwned, TwoStep<2>::kBlocks).cost / ((double)nx * ny);
  return per_node < (adr_block_x(prec, nx_pad, ny) == 64 ? 2.9e-5 : 2.02e-5);
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
