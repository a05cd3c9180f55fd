// Definitions of the kernel launchers declared in lbm_kernels.cuh.  Each
// precision's translation unit includes this file and instantiates them, so
// the kernel variants compile in parallel.
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

template <class P, int NS, int MODE>
static cudaError_t launch_step(AdrArgs a, cudaStream_t st, bool chained) {
  if constexpr (P::kDev) {
    constexpr int kThreads = MODE == kAdrCheck ? kPairThreads : kQuadThreads;
    const AdrGrid g = adr_grid(a.nx_pad, a.ny, a.nbnd, kBlockX, kThreads);
    set_grid(a, g, kThreads);
    if constexpr (MODE == kAdrCheck)
      return launch_chained(chained, adr_check_pair_kernel<NS>, g.dim(), kThreads, st, a);
    else
      return launch_chained(chained, adr_step_quad_kernel<NS>, g.dim(), kThreads, st, a);
  } else {
    const int bx = adr_block_x(sizeof(typename P::S) == 8 ? LBM_F64 : LBM_F32,
                               a.nx_pad, a.ny);
    const AdrGrid g = adr_grid(a.nx_pad, a.ny, a.nbnd, bx, bx);
    set_grid(a, g, bx);
    return launch_chained(chained, bx == 64 ? adr_step_kernel<P, NS, MODE, 64>
                                            : adr_step_kernel<P, NS, MODE, 256>,
                          g.dim(), bx, st, a);
  }
}

template <class P, int NS>
static cudaError_t launch_adr_ns(int mode, const AdrArgs &a, cudaStream_t st,
                                 bool chained) {
  if (mode == kAdrStep) return launch_step<P, NS, kAdrStep>(a, st, chained);
  if (mode == kAdrCheck) return launch_step<P, NS, kAdrCheck>(a, st, chained);
  adr_init_kernel<P, NS><<<adr_node_grid(a.nx_pad, a.ny), kBlockX, 0, st>>>(a);
  return cudaGetLastError();
}

template <class P>
cudaError_t launch_adr(int ns, int mode, const AdrArgs &a, cudaStream_t st,
                       bool chained) {
  switch (ns) {
    case 1: return launch_adr_ns<P, 1>(mode, a, st, chained);
    case 2: return launch_adr_ns<P, 2>(mode, a, st, chained);
    case 3: return launch_adr_ns<P, 3>(mode, a, st, chained);
    default: return cudaErrorInvalidValue;
  }
}

template <class P>
cudaError_t launch_adr_flux(int ns, const void *g, const RefT *ref,
                            const uint32_t *links, long long plane, int nx_pad,
                            int ny, int xp, double *out, cudaStream_t st) {
  const dim3 block(kReduceThreads);
  if (ns == 1)
    adr_flux_kernel<P, 1><<<1, block, 0, st>>>(g, ref, links, plane, nx_pad, ny, xp, out);
  else if (ns == 2)
    adr_flux_kernel<P, 2><<<1, block, 0, st>>>(g, ref, links, plane, nx_pad, ny, xp, out);
  else if (ns == 3)
    adr_flux_kernel<P, 3><<<1, block, 0, st>>>(g, ref, links, plane, nx_pad, ny, xp, out);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <class P, int BX, int BLOCKS>
static cudaError_t launch_flow_bx(int mode, const FlowArgs &a, cudaStream_t st,
                                  bool chained) {
  const auto kernel = mode == kFlowStep ? flow_kernel<P, kFlowStep, BX, BLOCKS>
                      : mode == kFlowU  ? flow_kernel<P, kFlowU, BX, BLOCKS>
                      : mode == kFlowCheck ? flow_kernel<P, kFlowCheck, BX, BLOCKS>
                                           : flow_kernel<P, kFlowInit, BX, BLOCKS>;
  return launch_chained(chained, kernel, flow_grid(a.nx_pad, a.ny), BX, st, a);
}

template <class P>
cudaError_t launch_flow(int mode, const FlowArgs &a, cudaStream_t st, bool chained) {
  constexpr int kPrec = sizeof(typename P::T) == 8 ? LBM_F64 : LBM_F32;
  if (flow_block_x(a.nx_pad, a.ny) == 64) return launch_flow_bx<P, 64, 0>(mode, a, st, chained);
  if constexpr (kPrec == LBM_F32) {
    if (flow_blocks_per_sm(kPrec, a.nx_pad, a.ny) == 8)
      return launch_flow_bx<P, 256, 8>(mode, a, st, chained);
  }
  return launch_flow_bx<P, 256, 0>(mode, a, st, chained);
}

template <class P, int NS, int BX>
static cudaError_t launch_adjoint_bx(int mode, const AdjArgs &a, cudaStream_t st,
                                     bool chained) {
  using T = typename P::T;
  const auto kernel = mode == kAdjCheck ? (a.periodic ? adj_kernel<T, NS, kAdjCheck, true, BX>
                                                      : adj_kernel<T, NS, kAdjCheck, false, BX>)
                                        : (a.periodic ? adj_kernel<T, NS, kAdjStep, true, BX>
                                                      : adj_kernel<T, NS, kAdjStep, false, BX>);
  return launch_chained(chained, kernel, adj_grid(sizeof(T) == 8 ? LBM_F64 : LBM_F32, a.nx_pad, a.ny),
                        BX, st, a);
}
template <class P, int NS>
static cudaError_t launch_adjoint_ns(int mode, const AdjArgs &a, cudaStream_t st,
                                     bool chained) {
  const int bx = adr_block_x(sizeof(typename P::T) == 8 ? LBM_F64 : LBM_F32, a.nx_pad, a.ny);
  return bx == 64 ? launch_adjoint_bx<P, NS, 64>(mode, a, st, chained)
                  : launch_adjoint_bx<P, NS, 256>(mode, a, st, chained);
}

template <class P>
cudaError_t launch_adjoint(int ns, int mode, const AdjArgs &a, cudaStream_t st,
                           bool chained) {
  switch (ns) {
    case 1: return launch_adjoint_ns<P, 1>(mode, a, st, chained);
    case 2: return launch_adjoint_ns<P, 2>(mode, a, st, chained);
    case 3: return launch_adjoint_ns<P, 3>(mode, a, st, chained);
    default: return cudaErrorInvalidValue;
  }
}

template <class P>
cudaError_t launch_adjoint_grad(int ns, const AdjArgs &a, const BoundaryNode *bnodes,
                                long long nbnd, const void *conc, double *dkab,
                                double *dkbc, const int32_t *fiber, double *dw,
                                double k1, double k2, cudaStream_t st) {
  using T = typename P::T;
  if (nbnd == 0) return cudaSuccess;
  const dim3 block(kBlockX);
  const unsigned nb = static_cast<unsigned>((nbnd + kBlockX - 1) / kBlockX);
  const T *c = static_cast<const T *>(conc);
  switch (ns) {
    case 1: adj_grad_kernel<T, 1><<<nb, block, 0, st>>>(a, bnodes, nbnd, c, dkab, dkbc, fiber, dw, k1, k2); break;
    case 2: adj_grad_kernel<T, 2><<<nb, block, 0, st>>>(a, bnodes, nbnd, c, dkab, dkbc, fiber, dw, k1, k2); break;
    case 3: adj_grad_kernel<T, 3><<<nb, block, 0, st>>>(a, bnodes, nbnd, c, dkab, dkbc, fiber, dw, k1, k2); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace lbm
