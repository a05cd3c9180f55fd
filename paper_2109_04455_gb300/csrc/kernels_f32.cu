// Kernel instantiations for PrecF32.
#include "lbm_launch_impl.cuh"

namespace lbm {
// From 2^22 nodes the populations of two or three species are far from
// fitting L2, and reading them half as often pays: 3000 x 1500 nodes of three
// species took 161 us per step with one step per launch and 150 with two,
// 4096 x 2048 306 and 262 (two species 216 and 170), 16384 x 4096 2310 and
// 1660.  Below it does not (2048 x 1024: 79 and 89 us; 1000 x 900: 48 and
// 47), nor for one species (4096 x 2048: 130 and 127).  The kernel numbers
// the populations of all species with 32 bits.
bool two_step_pays(int prec, int ns, long long plane) {
  return prec == LBM_F32 && ns >= 2 && plane >= (1ll << 22) && 9 * ns * plane < (1ll << 32);
}

template <int NS>
static cudaError_t two_step_ns(const AdrArgs &a, cudaStream_t st) {
  using K = TwoStep<NS>;
  cudaError_t e = cudaFuncSetAttribute(adr_two_step_kernel<NS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, K::kShared);
  if (e != cudaSuccess) return e;
  const int rows = two_step_rows(a.nx, a.ny, K::kOwned, K::kBlocks);
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
