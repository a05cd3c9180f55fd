// sm_103a kernels of liblbm: fused pull stream-collide for the flow lattice
// and for all ADR species at once, plus the outflux and residual reductions.
//
// Data layout in HBM (structure of arrays, x contiguous):
//   populations  [species][q][ny][nx_pad]   (two buffers, ping-pong)
//   link words   [ny][nx_pad]  uint32, nibble j-1 = type of neighbour x+c_j
//   rates        k_AB, k_BC [ny][nx_pad] double (read on catalytic links only)
//   velocity     [2][ny][nx_pad]
// One thread owns one node (two or four with half storage); a block covers
// consecutive nodes of one row, so every population plane is read and written
// with coalesced accesses (the pull of a plane is a pure shift: each element
// of the source plane is read exactly once per step).
//
// There are no contractions here (about 1 flop per byte in float).  What
// bounds a step: bytes in float and half on large lattices, the FP64 pipe in
// double, and the latency of one launch on small lattices.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "lbm_internal.h"

namespace lbm {

// SMs of the part, for the rules on launch shapes and waves of blocks (a host
// without a GPU evaluates them too, for the workspace sizes).
constexpr int kSMs = 152;
// Threads per block of the initial-state and gradient kernels, and nodes of a
// row segment of half storage.  (The flow, step and adjoint kernels take 64 or
// 256 threads, see adr_block_x.)
#ifndef LBM_BLOCK_X
#define LBM_BLOCK_X 256
#endif
constexpr int kBlockX = LBM_BLOCK_X;
constexpr int kReduceThreads = 256;

// ---------------------------------------------------------------------------
// precision traits: storage type S, compute type T
// ---------------------------------------------------------------------------
struct PrecF64 {
  using S = double;
  using T = double;
  static constexpr bool kDev = false;
  static constexpr int kMinBlocks = 4;   // <= 64 registers
  static __device__ __forceinline__ T load(S v) { return v; }
  static __device__ __forceinline__ S store(T v) { return v; }
};
struct PrecF32 {
  using S = float;
  using T = float;
  static constexpr bool kDev = false;
  static constexpr int kMinBlocks = 4;   // <= 64 registers
  static __device__ __forceinline__ T load(S v) { return v; }
  static __device__ __forceinline__ S store(T v) { return v; }
};
// half storage of the deviation g - w_i R from a per-node reference R (the
// node's concentration when the value was stored, kept in half beside the
// populations), scaled by 2^14 (exact) so that the deviations of dilute
// species stay in half's normal range (|value| <= 0.45 * 2^14 < 65504);
// rounded to nearest even.  The deviation is the advective and
// non-equilibrium part of g, a few percent of it, so half's 11 bits resolve
// g to ~1e-5 instead of ~5e-4.
struct PrecF16Dev {
  using S = __half;
  using T = float;
  static constexpr bool kDev = true;
  static __device__ __forceinline__ T load(S v) {
    return __half2float(v) * (1.0f / 16384.0f);
  }
  static __device__ __forceinline__ S store(T v) {
    return __float2half_rn(v * 16384.0f);
  }
};

template <typename T>
struct Lattice {
  static __device__ __forceinline__ T w(int i) {
    return i == 0 ? T(4) / T(9) : (i < 5 ? T(1) / T(9) : T(1) / T(36));
  }
};

__device__ __forceinline__ constexpr int cx(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__device__ __forceinline__ constexpr int cy(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
__device__ __forceinline__ constexpr int opp(int i) {
  return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4 + 1) : ((i - 5 + 2) % 4 + 5));
}
__device__ __forceinline__ uint32_t nib(uint32_t word, int j) {
  return (word >> (4 * (j - 1))) & 0xFu;
}
// Index of the neighbour x + c_j of the node (x, y) (plane index
// y * np + x), wrapped around a periodic edge; for a neighbour inside the
// lattice it is the plain shift.  Used on boundary nodes only (kPeriodic
// pulls, rates of catalytic links).
__device__ __forceinline__ long long neighbour(int x, int y, int j, int nx,
                                               int ny, long long np) {
  int tx = x + cx(j), ty = y + cy(j);
  tx = tx < 0 ? tx + nx : (tx >= nx ? tx - nx : tx);
  ty = ty < 0 ? ty + ny : (ty >= ny ? ty - ny : ty);
  return (long long)ty * np + tx;
}

__device__ __forceinline__ float absT(float x) { return fabsf(x); }
__device__ __forceinline__ double absT(double x) { return fabs(x); }

// Steps follow one another on a stream, each a launch of a few microseconds on
// a small lattice.  A step launched by launch_chained may start while the one
// before it is running (programmatic dependent launch): it reads what no step
// writes (link words, velocity, rates), waits for the one before it to finish,
// lets its own follower start, and goes on to the populations.  Launched
// otherwise the wait is none.  Per step it took a 200 x 100 FP64 flow from 8.5
// to 6.4 us and ADR lattice from 10.6 to 8.6, 300 x 300 FP32 from 8.6 to 4.9,
// 1000 x 300 from 18.9 to 15.3, the 2048 x 512 FP32 adjoint from 47.0 to 43.9;
// the largest lattices are within 1%.  (Letting the follower start before the wait
// fills the SMs with waiting blocks of several steps: a 200 x 100 FP64 flow
// took 23 us per step that way, and 8.5 without overlap.  Pointers to what the
// step before writes are not __restrict__: its data are not read-only during
// this kernel's lifetime.)
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// chained: the work before this launch on the stream is a step of the same
// solver, so that what steps only read was complete before that one started
template <class... P, class... A>
inline cudaError_t launch_chained(bool chained, void (*kernel)(P...), dim3 grid,
                                  unsigned threads, cudaStream_t st, A... args) {
  cudaLaunchAttribute overlap;
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.stream = st;
  c.attrs = &overlap;
  c.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

// ---------------------------------------------------------------------------
// deterministic block sum of K values in the value type A, stored by threads
// 0..K-1 (one component each) to dst[0..K): used in double for the outflux, and
// in the run's precision for the adjoint's convergence measure.  (The forward
// check steps use block_partials_store below, which sums in double whatever
// the precision.)
// ---------------------------------------------------------------------------
template <int K, typename A>
__device__ __forceinline__ void block_sum_store(const A (&v)[K], double *dst) {
  __shared__ A red[32][K];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  A w[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    w[k] = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w[k] += __shfl_down_sync(0xffffffffu, w[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) red[warp][k] = w[k];
  }
  __syncthreads();
  if (threadIdx.x < K) {
    const int nw = (blockDim.x + 31) >> 5;
    A s = A(0);
    for (int i = 0; i < nw; ++i) s += red[i][threadIdx.x];
    dst[threadIdx.x] = double(s);
  }
}

// Check-step partials of one block, accumulated in double.  Each of the BX
// threads passes the values of NPER nodes, v[NPER][KS + KM] (zeros for a
// thread or node without a fluid node): the first KS components are summed,
// the last KM reduced by minimum (a minimum starts at 0, so it is that of
// min(value, 0)).  The values are staged in shared memory, one row per
// component; warp w then reduces components w, w + BX/32, ...: its lanes add
// the component's values at a stride of 32 in double, and the 32 lane sums
// are folded by double shuffles.  Every per-node value enters a double sum,
// so a block partial carries no single-precision rounding; the fixed order
// makes it deterministic.
template <int KS, int KM, int NPER, int BX, typename A>
__device__ __forceinline__ void block_partials_store(const A (&v)[NPER][KS + KM],
                                                     double *dst) {
  constexpr int K = KS + KM;
  constexpr int NV = BX * NPER;
  static_assert(BX % 32 == 0, "whole warps");
  __shared__ A stage[K][NV];
  const int t = threadIdx.x;
#pragma unroll
  for (int p = 0; p < NPER; ++p) {
#pragma unroll
    for (int k = 0; k < K; ++k) stage[k][p * BX + t] = v[p][k];
  }
  __syncthreads();
  const int lane = t & 31, warp = t >> 5;
  for (int k = warp; k < K; k += BX / 32) {
    double r = 0.0;
    if (k < KS) {
#pragma unroll 4
      for (int j = lane; j < NV; j += 32) r += double(stage[k][j]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    } else {
      A m = A(0);
#pragma unroll 4
      for (int j = lane; j < NV; j += 32) m = stage[k][j] < m ? stage[k][j] : m;
      r = double(m);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) r = fmin(r, __shfl_down_sync(0xffffffffu, r, o));
    }
    if (lane == 0) dst[k] = r;
  }
}

// Per-node contribution of species s to a check step's partials (layout
// [2 NS sums | NS minima]): |C(t) - C(t-1)|, |C(t)|, and C(t) for the most
// negative concentration.
template <int NS, typename T>
__device__ __forceinline__ void check_add(T (&acc)[3 * NS], int s, T c, T prev) {
  acc[2 * s] += absT(c - prev);
  acc[2 * s + 1] += absT(c);
  acc[2 * NS + s] = c < acc[2 * NS + s] ? c : acc[2 * NS + s];
}

// Reference concentrations of the half path are themselves stored in half:
// any reference works as long as the writer and every reader use the same
// value, so the writer subtracts the rounded reference it stores.
using RefT = __half;
__device__ __forceinline__ float ref_get(const RefT *r, long long k) {
  return __half2float(r[k]);
}
__device__ __forceinline__ float ref_round(float c) {
  return __half2float(__float2half_rn(c));
}

// Kernel parameters come in double and in float; the float paths read the
// float copy, so no thread converts a double (this part's FP64 pipe is
// narrow enough for per-thread conversions to show up in a step's time).
template <typename T>
__device__ __forceinline__ T pick(double d, float f);
template <>
__device__ __forceinline__ double pick<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float pick<float>(double, float f) { return f; }


// Every operation of the update is written with an explicit rounding (no
// contraction is left to the compiler): the two-step kernel, the one-step
// kernel, the boundary nodes, the batch kernel and the FP64 table must get
// the same bits for the same node, so that a run's result depends neither on
// how its steps are grouped into launches nor on the batch it is part of.
__device__ __forceinline__ float fma_rn(float x, float y, float z) { return __fmaf_rn(x, y, z); }
__device__ __forceinline__ double fma_rn(double x, double y, double z) { return __fma_rn(x, y, z); }
__device__ __forceinline__ float mul_rn(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double mul_rn(double x, double y) { return __dmul_rn(x, y); }
__device__ __forceinline__ float add_rn(float x, float y) { return __fadd_rn(x, y); }
__device__ __forceinline__ double add_rn(double x, double y) { return __dadd_rn(x, y); }
// sum of a node's nine populations
template <typename T>
__device__ __forceinline__ T sum_in_order(const T (&g)[9]) {
  T c = g[0];
#pragma unroll
  for (int i = 1; i < 9; ++i) c = add_rn(c, g[i]);
  return c;
}
__device__ __forceinline__ float sum_rn(const float (&g)[9]) { return sum_in_order(g); }
// In double the sum is taken in integers: the FP64 pipe (two lanes per clock
// and SM, against 128 for integers) bounds the step, and eight of a species'
// 26 double operations were this sum.  The mantissas are aligned to the
// largest exponent with six bits to spare, added exactly and rounded once: off
// by at most half an ulp of the sum and 9/64 ulp of the largest term, against
// up to eight roundings one after the other (over random populations the
// largest error was 5.4e-16 of the largest term, 2.0e-15 in order).  Terms too
// small or too large for that (the largest below 2^-943 or from 2^1016,
// infinite, NaN) are added in order.  That holds for one sum; after a run both
// forms are equally far off, by the rounding of the weights (300 to 1600 steps
// of six lattices, one to three species: 1.5e-14 to 9.7e-14 off an 80-bit run,
// within 1% of each other).  2048 x 512, three species: 163 us per step in order,
// 113 in integers and with the species' loads one by one (adr_interior_node),
// which were not timed apart.
__device__ __forceinline__ double sum_rn(const double (&g)[9]) {
  unsigned top = 0u;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    top = max(top, static_cast<unsigned>(__double2hiint(g[i])) & 0x7FFFFFFFu);
  const unsigned e = top >> 20;
  if (top == 0u) return 0.0;
  if (e - 80u >= 0x7F7u - 80u) return sum_in_order(g);
  long long sum = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const unsigned hi = __double2hiint(g[i]), lo = __double2loint(g[i]);
    const unsigned shift = min(e - ((hi >> 20) & 0x7FFu), 63u);
    const unsigned long long m =
        ((static_cast<unsigned long long>((hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << 6) >> shift;
    // minus m for a negative term: (m ^ -1) + 1
    const long long sign = static_cast<int>(hi) >> 31;
    sum += (static_cast<long long>(m) ^ sign) - sign;
  }
  if (sum == 0) return 0.0;
  // to a double by hand (the conversion instruction takes as long as five
  // FP64 operations): the leading one to bit 62, rounded to 53 bits (to
  // nearest, ties to even; a carry moves into the exponent), times
  // 2^(e - 1023 - 52 - 6)
  unsigned long long u = sum < 0 ? -static_cast<unsigned long long>(sum) : sum;
  const int z = __clzll(u) - 1;
  u <<= z;
  u = (u + 0x1FFu + (u >> 10 & 1u)) >> 10;
  u += static_cast<unsigned long long>(e + 3u - static_cast<unsigned>(z)) << 52;
  u |= static_cast<unsigned long long>(sum) & (1ull << 63);
  return __longlong_as_double(static_cast<long long>(u));
}
// BGK relaxation of a population g towards c E
template <typename T>
__device__ __forceinline__ T relax(T om, T c, T E, T g) {
  return fma_rn(om, fma_rn(c, E, -g), g);
}

// ---------------------------------------------------------------------------
// ADR
// ---------------------------------------------------------------------------
struct AdrArgs {
  const void *src;          // S [ns][9][plane]  post-collision at time t
  void *dst;                // S [ns][9][plane]  post-collision at time t+1
  const uint32_t *links;    // [plane]
  const double *kab, *kbc;  // [plane]
  const void *u;            // T [2][plane]
  void *cprev;              // T [ns][plane]     (check steps)
  double *partials;         // [rows][3*ns]      (check steps)
  const BoundaryNode *bnodes;  // boundary fluid nodes (link word != 0)
  long long nbnd;           // number of boundary nodes
  long long plane;          // ny * nx_pad
  int nx, ny, nx_pad;
  int nxb;                  // row segments per row of a step's grid
  unsigned chunks;          // its boundary chunks, spread over the blocks at
  unsigned share;           // this density, times 2^32 (step_block)
  unsigned rowmul;          // division by nxb of an interior block's number
  int rowshift;
  int abb_all;              // anti-bounce-back inlet for every species
  int nodewise;             // every population of a reactive node reacts
  unsigned step;            // steps done before this one (rounding seed)
  int xp;                   // flux plane
  double omega[3];          // 1/tau per species
  double cin[3];            // inlet concentration per species
  float fomega[3], fcin[3]; // the same in float
  // half storage: reference concentrations [ns][plane] of the src and dst
  // populations (the stored value is g - w_i R of its node)
  const RefT *rsrc;
  RefT *rdst;
  // FP64: equilibrium factors E_i(u) [9][plane] of the frozen velocity,
  // filled once by eq_table_kernel (nullptr: computed per node and step;
  // the FP64 step is bound by this part's FP64 pipe, and the table takes
  // about a third of its double operations away)
  const double *etab;
};

enum AdrMode { kAdrStep = 0, kAdrCheck = 1, kAdrInit = 2 };


// equilibrium factors E_i(u), shared by every species:
// g_i^eq = C * E_i, E_i = w_i (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u.u)
__device__ __forceinline__ void eq_factors(float ux, float uy, float (&E)[9]) {
  const float uu = fma_rn(ux, ux, mul_rn(uy, uy));
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const float cu = add_rn(float(cx(i)) * ux, float(cy(i)) * uy);
    E[i] = mul_rn(Lattice<float>::w(i),
                  fma_rn(-1.5f, uu, fma_rn(mul_rn(4.5f, cu), cu, fma_rn(3.0f, cu, 1.0f))));
  }
}
__device__ __forceinline__ void eq_factors(double ux, double uy, double (&E)[9]) {
  const double base = fma_rn(-1.5, fma_rn(ux, ux, mul_rn(uy, uy)), 1.0);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const double cu = add_rn(double(cx(i)) * ux, double(cy(i)) * uy);
    E[i] = mul_rn(Lattice<double>::w(i),
                  fma_rn(mul_rn(4.5, cu), cu, fma_rn(3.0, cu, base)));
  }
}

// equilibrium factors of node n: from the FP64 table when there is one
template <class P>
__device__ __forceinline__ void adr_eq(const AdrArgs &a, long long n,
                                       typename P::T (&E)[9]) {
  using T = typename P::T;
  if constexpr (sizeof(T) == 8) {
    if (a.etab != nullptr) {
#pragma unroll
      for (int i = 0; i < 9; ++i) E[i] = a.etab[(long long)i * a.plane + n];
      return;
    }
  }
  const T *__restrict__ U = static_cast<const T *>(a.u);
  eq_factors(U[n], U[a.plane + n], E);
}

// E_i(u) of every node of the lattice into etab [9][plane] (FP64 only)
template <typename T>
__global__ void __launch_bounds__(256)
    eq_table_kernel(const T *u, long long plane, T *etab) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= plane) return;
  T E[9];
  eq_factors(u[n], u[plane + n], E);
#pragma unroll
  for (int i = 0; i < 9; ++i) etab[(long long)i * plane + n] = E[i];
}

// The species are updated one after the other (A, then B, then C): the
// sources are triangular (A's depends on C_A, B's on C_A and C_B, C's on
// C_B), so every source term is known when its species is collided, and only
// one species' nine populations need to be live at a time.

// Where the update of a boundary node (x, y), plane index n, reads the old
// populations: the global planes.  at(i, j, t) is the place of population i of
// the neighbour x + c_j (j = 0: the node itself) across a link of type t (kFluid
// or kPeriodic), get(s, place) its value for species s.
template <class P>
struct OldState {
  using T = typename P::T;
  struct Place {
    long long plane, node;   // i * plane, node index
    int i;
  };
  const AdrArgs &a;
  long long n;
  int x, y;
  __device__ __forceinline__ Place at(int i, int j, uint32_t t) const {
    const long long np = a.nx_pad;
    return {i * a.plane,
            t == kPeriodic ? neighbour(x, y, j, a.nx, a.ny, np) : n + cy(j) * np + cx(j),
            i};
  }
  __device__ __forceinline__ T get(int s, const Place &k) const {
    const typename P::S *src = static_cast<const typename P::S *>(a.src);
    const typename P::S v = src[s * 9 * a.plane + k.plane + k.node];
    if constexpr (P::kDev) {   // plus w_i times the node's reference
      const T w = k.i == 0 ? Lattice<T>::w(0) : k.i < 5 ? Lattice<T>::w(1) : Lattice<T>::w(5);
      return fma_rn(__half2float(v), 1.0f / 16384.0f,
                    mul_rn(w, ref_get(a.rsrc, s * a.plane + k.node)));
    } else {
      return P::load(v);
    }
  }
};

// Source of species s on a population of weight w at rates ka, kb:
//   Q_A = -k_AB w C_A,  Q_B = +k_AB w C_A - k_BC w C_B,  Q_C = +k_BC w C_B.
template <int NS, typename T>
__device__ __forceinline__ T react(int s, T ka, T kb, T w, const T (&C)[NS], T g) {
  if (s == 0) return fma_rn(-mul_rn(ka, w), C[0], g);
  const T cb = C[NS >= 2 ? 1 : 0];
  if (s == 2) return fma_rn(mul_rn(kb, w), cb, g);
  if (NS == 2) return fma_rn(mul_rn(ka, w), C[0], g);
  return add_rn(g, fma_rn(mul_rn(ka, w), C[0], -mul_rn(mul_rn(kb, w), cb)));
}

// The source of species s of a node with catalytic links: rates ka, kb of
// the links, concentrations C of species 0..s.
template <int NS, typename T>
__device__ __forceinline__ void add_source(const AdrArgs &a, int s, uint32_t lw,
                                           const T (&ka)[9], const T (&kb)[9],
                                           const T (&C)[NS], T (&g)[9]) {
  if (a.nodewise) {
    T sa = T(0), sb = T(0);
    int ncat = 0;
#pragma unroll
    for (int j = 1; j < 9; ++j) {
      if (nib(lw, j) != kCat) continue;
      sa = add_rn(sa, ka[j]);
      sb = add_rn(sb, kb[j]);
      ++ncat;
    }
    const T ma = sa / T(ncat), mb = sb / T(ncat);
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = react<NS>(s, ma, mb, Lattice<T>::w(i), C, g[i]);
  } else {
#pragma unroll
    for (int j = 1; j < 9; ++j)
      if (nib(lw, j) == kCat) g[j] = react<NS>(s, ka[j], kb[j], Lattice<T>::w(j), C, g[j]);
  }
}

// The old populations that the update of node (link word lw) reads, into g:
// the pulls from x - c_i, or, where the source is not a fluid node, the
// node's own opposite population, to which update_node then applies the rule
// of the link's type (Eq. BC and bounce-back).
//
// There is one load per population whatever the link types, from a selected
// place, and all are issued before any arithmetic: the boundary nodes'
// latency bounds the step of a small lattice (a 200 x 100 one took 23 us per
// step with each load behind its link's branch, species after species).
//
// (The two-step kernel gathers from global planes and from its ring by code of
// its own, and has edge_rules over masks; both forms must stay alike, which the
// tests of equal bits hold them to.)
template <int NS, class P, typename T>
__device__ __forceinline__ void gather_node(const OldState<P> &src, uint32_t lw,
                                            T (&g)[NS][9]) {
  // Any fluid node.  (The boundary list holds none of link word 0, yet without
  // this branch the allocator spills 28 bytes a thread more in the FP32 batch
  // step, whose 16 lattices then take 69.5 ms instead of 68.3.)
  if (lw == 0u) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const auto from = src.at(i, opp(i), kFluid);
#pragma unroll
      for (int s = 0; s < NS; ++s) g[s][i] = src.get(s, from);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const uint32_t t = i == 0 ? (uint32_t)kFluid : nib(lw, opp(i));
    const bool pulled = t == kFluid || t == kPeriodic;
    const auto from = pulled ? src.at(i, opp(i), t) : src.at(opp(i), 0, kFluid);
#pragma unroll
    for (int s = 0; s < NS; ++s) g[s][i] = src.get(s, from);
  }
}

// The inlet and outlet rules of a node of the first or last column (link
// word lw), species s: g holds the node's own opposite populations there.
// cb: the node's own concentration (outlet).
template <typename T>
__device__ __forceinline__ void edge_rules(const AdrArgs &a, int s, uint32_t lw,
                                           T cb, T (&g)[9]) {
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const uint32_t t = nib(lw, opp(i));
    const T w2 = T(2) * Lattice<T>::w(i);
    if (t == kInlet && (s == 0 || a.abb_all))
      g[i] = fma_rn(w2, pick<T>(a.cin[s], a.fcin[s]), -g[i]);
    else if (t == kOutlet)
      g[i] = fma_rn(w2, cb, -g[i]);
  }
}

// BGK of species s towards C E_i; returns C.
template <typename T>
__device__ __forceinline__ T collide(const AdrArgs &a, int s, const T (&E)[9], T (&g)[9]) {
  const T c = sum_rn(g), om = pick<T>(a.omega[s], a.fomega[s]);
#pragma unroll
  for (int i = 0; i < 9; ++i) g[i] = relax(om, c, E[i], g[i]);
  return c;
}

// Whether node (x, y), link word lw, has catalytic links, and their rates, all
// loaded at once.
template <typename T>
__device__ __forceinline__ bool link_rates(const AdrArgs &a, uint32_t lw, int x, int y,
                                           T (&ka)[9], T (&kb)[9]) {
  bool cat = false;
#pragma unroll
  for (int j = 1; j < 9; ++j) cat = cat || nib(lw, j) == kCat;
  if (cat) {
    double da[9], db[9];
#pragma unroll
    for (int j = 1; j < 9; ++j) {
      const bool on = nib(lw, j) == kCat;
      const long long m = on ? neighbour(x, y, j, a.nx, a.ny, a.nx_pad) : 0;
      da[j] = on ? a.kab[m] : 0.0;
      db[j] = on ? a.kbc[m] : 0.0;
    }
#pragma unroll
    for (int j = 1; j < 9; ++j) {
      ka[j] = T(da[j]);
      kb[j] = T(db[j]);
    }
  }
  return cat;
}

// Update of boundary node (x, y) of the global planes from its gathered
// populations g: the rules of its links, BGK towards C E_i, then the Dawson
// source on links into catalytic fiber nodes (Eq. source_lbm), or, with
// a.nodewise, on all nine populations with the mean rates of those links (ka,
// kb, cat: link_rates).  put(s, g, c) stores the new populations of species s,
// whose concentration is c.
template <int NS, class P, typename T, class Put>
__device__ __forceinline__ void update_node(const AdrArgs &a, const OldState<P> &src,
                                            uint32_t lw, bool cat, const T (&ka)[9],
                                            const T (&kb)[9], const T (&E)[9],
                                            T (&g)[NS][9], Put &&put) {
  bool inlet = false, outlet = false;
#pragma unroll
  for (int j = 1; j < 9; ++j) {
    const uint32_t t = nib(lw, j);
    inlet = inlet || t == kInlet;
    outlet = outlet || t == kOutlet;
  }
  if (inlet || outlet) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      T cb = T(0);
      if (outlet) {   // C_w = the node's own concentration
        T own[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) own[j] = src.get(s, src.at(j, 0, kFluid));
        cb = sum_rn(own);
      }
      edge_rules(a, s, lw, cb, g[s]);
    }
  }
  T C[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    C[s] = collide(a, s, E, g[s]);
    if (cat) add_source<NS>(a, s, lw, ka, kb, C, g[s]);
    put(s, g[s], C[s]);
  }
}

// Store of the new populations of species s of node n, whose concentration
// is c, in the global planes (half storage: less w_i times the reference,
// which is stored beside them).
template <class P, typename T>
__device__ __forceinline__ void put_node(const AdrArgs &a, int s, long long n,
                                         const T (&g)[9], T c) {
  typename P::S *__restrict__ dst = static_cast<typename P::S *>(a.dst);
  T cq = c;
  if constexpr (P::kDev) {
    cq = ref_round(c);
    a.rdst[s * a.plane + n] = __float2half_rn(c);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i)
    dst[(long long)(s * 9 + i) * a.plane + n] =
        P::store(P::kDev ? fma_rn(-Lattice<T>::w(i), cq, g[i]) : g[i]);
}

// A boundary node of the global planes, link word lw.
template <class P, int NS, int MODE>
__device__ __forceinline__ void adr_boundary_node(const AdrArgs &a, long long n,
                                                  uint32_t lw,
                                                  typename P::T (&acc)[3 * NS]) {
  using T = typename P::T;
  const int y = static_cast<int>(n / a.nx_pad);
  const int x = static_cast<int>(n - (long long)y * a.nx_pad);
  const OldState<P> src{a, n, x, y};
  T g[NS][9], E[9], ka[9], kb[9], prev[NS];
  adr_eq<P>(a, n, E);
  const bool cat = link_rates(a, lw, x, y, ka, kb);
  wait_for_previous();
  gather_node<NS>(src, lw, g);
  T *cp = static_cast<T *>(a.cprev);
  if (MODE == kAdrCheck) {
#pragma unroll
    for (int s = 0; s < NS; ++s) prev[s] = cp[s * a.plane + n];
  }
  update_node<NS>(a, src, lw, cat, ka, kb, E, g, [&](int s, const T (&g)[9], T c) {
    put_node<P>(a, s, n, g, c);
    if (MODE == kAdrCheck) {
      check_add<NS, T>(acc, s, c, prev[s]);
      cp[s * a.plane + n] = c;
    }
  });
}

// L2 prefetch ahead of the FP16 steps.  With D = LBM_PREFETCH_ROWS_F16 > 0
// each block asks L2 for the row segments that the block D rows further down
// will read: one bulk prefetch per plane (the 9 NS population rows y + D -
// c_iy, the NS reference rows, u and the link words of row y + D).  Blocks
// start in row order, so those lines are on their way from HBM about D rows
// of blocks before their loads are issued, and they are in flight without
// holding registers.
#ifndef LBM_PREFETCH_ROWS_F16
#define LBM_PREFETCH_ROWS_F16 6
#endif
// [p, p + bytes) into L2, nothing to wait for; p 16-byte aligned and bytes
// a multiple of 16
__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
               :: "l"(p), "r"(bytes) : "memory");
}
// Nodes [xb, xb + width) of row yp, xb and width multiples of 32, by a block
// of THREADS threads; rows outside the lattice are skipped.  ANYU: u may start
// at any float (its segment is then taken from the 16-byte boundary before).
template <int NS, int THREADS, bool ANYU>
__device__ __forceinline__ void prefetch_rows_f16(const AdrArgs &a, int yp, int xb, int width) {
  constexpr int kPop = 9 * NS, kAll = kPop + NS + 3;
  if (yp >= a.ny) return;
  const long long np = a.nx_pad, plane = a.plane;
  // nx_pad is a multiple of 32, so every segment starts 64-byte aligned
  // (buffers are 256-byte aligned) and is a multiple of 64 bytes long
  const unsigned cnt = static_cast<unsigned>(min(width, a.nx_pad - xb));
#pragma unroll
  for (int k = 0; k < kAll; k += THREADS) {
    const int t = k + threadIdx.x;
    if (t < kPop) {
      const int row = yp - cy(t % 9);
      if (row >= 0 && row < a.ny)
        prefetch_l2(static_cast<const __half *>(a.src) + t * plane + row * np + xb, 2u * cnt);
    } else if (t < kPop + NS) {
      prefetch_l2(a.rsrc + (t - kPop) * plane + yp * np + xb, 2u * cnt);
    } else if (t < kPop + NS + 2) {
      const float *p = static_cast<const float *>(a.u) + (t - kPop - NS) * plane + yp * np + xb;
      if (ANYU) p = reinterpret_cast<const float *>(reinterpret_cast<uintptr_t>(p) & ~uintptr_t{15});
      prefetch_l2(p, 4u * cnt);
    } else if (t < kAll) {
      prefetch_l2(a.links + yp * np + xb, 4u * cnt);
    }
  }
}

// What a block of a step's grid works on.  A step is one launch: most blocks
// update the interior nodes (link word 0) of one row segment each, in the order
// of the rows, and the others chunks of BX entries of the boundary-node list
// with every link rule in place (both read only the old populations and write
// disjoint nodes).  Two launches on two streams, forked and joined by events
// every step, cost a 1000 x 300 lattice 34 us per step, almost all of it host
// time.  (With a column of blocks for the chunks beside the segments, mostly
// empty blocks on high lattices and a chunk from elsewhere in the list on each
// row, a step of 100 x 20000 FP32 took 167 us, 123 in this form, of 20000 x 50
// half 40 and 30, and of 700 x 400 FP32 with thin fibers everywhere 15.3 and 12.2.)
struct StepBlock {
  long long chunk;   // of the boundary-node list, -1: a row segment
  int xb, y;         // the segment
};
__device__ __forceinline__ StepBlock step_block(const AdrArgs &a) {
  const unsigned b = blockIdx.x;
  const unsigned before = min(__umulhi(b, a.share), a.chunks);
  if (min(__umulhi(b + 1u, a.share), a.chunks) != before) return {before, 0, 0};
  const unsigned i = b - before;
  const unsigned y = a.nxb == 1 ? i : __umulhi(i, a.rowmul) >> a.rowshift;
  return {-1, static_cast<int>(i - y * a.nxb), static_cast<int>(y)};
}
template <class P, int NS, int MODE, int BX>
__device__ __forceinline__ void boundary_nodes(const AdrArgs &a, long long chunk,
                                               typename P::T (&acc)[3 * NS]) {
  const long long t = chunk * BX + threadIdx.x;
  if (t >= a.nbnd) return;
  const BoundaryNode b = a.bnodes[t];
  adr_boundary_node<P, NS, MODE>(a, b.n, b.links, acc);
}
// check-step partial row of a block: the segments row by row, then the chunks
__device__ __forceinline__ long long partial_row(const AdrArgs &a, const StepBlock &k) {
  return k.chunk < 0 ? (long long)k.y * a.nxb + k.xb : (long long)a.ny * a.nxb + k.chunk;
}

}  // namespace lbm
// FP16-deviation storage: interior update (two and four nodes per thread)
#include "lbm_f16.cuh"
namespace lbm {

// Update of one interior node (link word 0: every neighbour is fluid), FP32
// and FP64: the interior formula (pull from x - c_i, BGK, no source).
// EARLY (small lattices): the equilibrium factors are read before waiting for
// the step before this one; on large lattices they would only take registers.
// All populations of all species are loaded before any arithmetic, so that a
// thread keeps NS * 9 independent loads in flight; not so in double on large
// lattices, where the FP64 pipe is the bound and 32 warps per SM with one
// species' loads each keep it busier (2048 x 512: 113 us per step, 137 us with
// 16 warps and all loads first, 115 with 24).
template <class P, int NS, int MODE, bool EARLY>
__device__ __forceinline__ void adr_interior_node(const AdrArgs &a, long long n,
                                                  typename P::T (&acc)[3 * NS]) {
  using S = typename P::S;
  using T = typename P::T;
  constexpr bool kTogether = EARLY || sizeof(T) == 4;
  const long long np = a.nx_pad, plane = a.plane;
  const S *src = static_cast<const S *>(a.src);
  S *__restrict__ dst = static_cast<S *>(a.dst);
  T g[NS][9], E[9];
  auto load = [&](int s) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const long long m = n - (cy(i) * np + cx(i));
      g[s][i] = P::load(src[(long long)(s * 9 + i) * plane + m]);
    }
  };
  if (EARLY) adr_eq<P>(a, n, E);
  wait_for_previous();
  if (kTogether) {
#pragma unroll
    for (int s = 0; s < NS; ++s) load(s);
  }
  // the previous concentrations are loaded with the populations, so the
  // check step waits on memory once, like the plain step
  T *__restrict__ cp = static_cast<T *>(a.cprev);
  T prev[NS];
  if (MODE == kAdrCheck) {
#pragma unroll
    for (int s = 0; s < NS; ++s) prev[s] = cp[s * plane + n];
  }
  if (!EARLY) adr_eq<P>(a, n, E);
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    if (!kTogether) load(s);
    const T c = sum_rn(g[s]);
    const T om = pick<T>(a.omega[s], a.fomega[s]);
#pragma unroll
    for (int i = 0; i < 9; ++i)
      dst[(long long)(s * 9 + i) * plane + n] = P::store(relax(om, c, E[i], g[s][i]));
    if (MODE == kAdrCheck) {
      check_add<NS, T>(acc, s, c, prev[s]);
      cp[s * plane + n] = c;
    }
  }
}

// Initial state g* of every node: C_A = 1, the others 0, at equilibrium, with
// the source of step 0 on catalytic links.  Bound by its stores: registers for
// 1024 threads per SM (512 in double), and the rates loaded once for all species.
template <class P, int NS>
__global__ void __launch_bounds__(kBlockX, sizeof(typename P::T) == 8 ? 2 : 4)
    adr_init_kernel(const AdrArgs a) {
  using T = typename P::T;
  const int x = blockIdx.x * kBlockX + threadIdx.x, y = blockIdx.y;
  const long long n = (long long)y * a.nx_pad + x;
  const uint32_t lw = (x < a.nx_pad) ? a.links[n] : kSolidNode;
  if (lw == kSolidNode) return;
  T E[9], C[NS], ka[9], kb[9];
  adr_eq<P>(a, n, E);
  const bool cat = lw != 0u && link_rates(a, lw, x, y, ka, kb);
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    T g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = mul_rn(s == 0 ? T(1) : T(0), E[i]);
    const T c = sum_rn(g), om = pick<T>(a.omega[s], a.fomega[s]);
    C[s] = c;
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = relax(om, c, E[i], g[i]);
    if (cat) add_source<NS>(a, s, lw, ka, kb, C, g);
    put_node<P>(a, s, n, g, c);
  }
}

// 256-thread blocks per SM that the step bounds its registers by.  FP32 with one
// species has nine loads a thread in flight, so it needs more threads than
// with three: 4096 x 2048 took 130 us per step at four blocks, 113 at six, 2048 x
// 512 12.3 and 10.4.
template <class P, int NS>
constexpr int step_blocks() {
  return sizeof(typename P::T) == 4 && NS == 1 ? 6 : P::kMinBlocks;
}
// One step (or check step), one node per thread.  On large lattices (BX =
// 256) the interior update needs its warps in flight, so the registers that
// the boundary update would like are bounded: with three species its 27 values
// and 16 rates spill (1192 bytes of stores per thread in double, 92 in float),
// which only boundary nodes pay for.
template <class P, int NS, int MODE, int BX>
__global__ void __launch_bounds__(BX, BX == 256 ? step_blocks<P, NS>() : 1)
    adr_step_kernel(const AdrArgs a) {
  using T = typename P::T;
  T acc[1][3 * NS];
#pragma unroll
  for (int k = 0; k < 3 * NS; ++k) acc[0][k] = T(0);
  const StepBlock k = step_block(a);
  if (k.chunk >= 0) {
    boundary_nodes<P, NS, MODE, BX>(a, k.chunk, acc[0]);
  } else {
    const int x = k.xb * BX + threadIdx.x;
    const long long n = (long long)k.y * a.nx_pad + x;
    const uint32_t lw = (x < a.nx_pad) ? a.links[n] : kSolidNode;
    if (lw == 0u) adr_interior_node<P, NS, MODE, BX == 64>(a, n, acc[0]);
  }
  if constexpr (MODE == kAdrCheck) {
    wait_for_previous();   // the partial sums are one buffer
    block_partials_store<2 * NS, NS, 1, BX, T>(acc, a.partials + partial_row(a, k) * (3 * NS));
  }
}

}  // namespace lbm
// two FP32 steps in one pass over memory
#include "lbm_twostep.cuh"
namespace lbm {

// Outflux on the plane x = xp from the stored post-collision populations:
// out[s] = (1/ny) sum_y sum_i c_ix g*_{s,i}(xp, y).  One block.
template <class P, int NS>
__global__ void __launch_bounds__(kReduceThreads)
    adr_flux_kernel(const void *g, const RefT *ref, const uint32_t *links,
                    long long plane, int nx_pad, int ny, int xp, double *out) {
  using S = typename P::S;
  const S *src = static_cast<const S *>(g);
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.0;
  for (int y = threadIdx.x; y < ny; y += blockDim.x) {
    const long long n = (long long)y * nx_pad + xp;
    if (links[n] == kSolidNode) continue;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double v = 0.0;
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        if (cx(i) == 0) continue;
        double gi = double(P::load(src[(long long)(s * 9 + i) * plane + n]));
        if (P::kDev) gi += double(Lattice<float>::w(i)) * double(ref_get(ref, s * plane + n));
        v += cx(i) > 0 ? gi : -gi;
      }
      acc[s] += v;
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] /= double(ny);
  block_sum_store<NS, double>(acc, out);
}

// Fold rows of KS + KM partials in a fixed order (sums of the first KS
// components, minima of the last KM).  Block b of the grid folds the rows
// [b*chunk, (b+1)*chunk) into out[b*K + k]; a second launch with one block
// folds those.  Deterministic for a fixed grid.
template <int KS, int KM>
__global__ void __launch_bounds__(kReduceThreads)
    reduce_partials_kernel(const double *partials, long long nb, long long chunk,
                           double *out) {
  constexpr int K = KS + KM;
  double acc[1][K];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[0][k] = 0.0;
  const long long lo = (long long)blockIdx.x * chunk;
  long long hi = lo + chunk;
  if (hi > nb) hi = nb;
  for (long long b = lo + threadIdx.x; b < hi; b += blockDim.x) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      acc[0][k] = k < KS ? acc[0][k] + partials[b * K + k]
                         : fmin(acc[0][k], partials[b * K + k]);
  }
  block_partials_store<KS, KM, 1, kReduceThreads, double>(
      acc, out + (long long)blockIdx.x * K);
}

}  // namespace lbm
// discrete adjoint of the ADR step: arguments and kernels
#include "lbm_adjoint.cuh"
namespace lbm {

// ---------------------------------------------------------------------------
// flow
// ---------------------------------------------------------------------------
struct FlowArgs {
  const void *src;        // S [9][plane]
  void *dst;              // S [9][plane]
  const uint32_t *links;  // [plane]
  void *u;                // T [2][plane]  (written on u / check steps)
  double *partials;       // [nblocks][2]  (check steps)
  long long plane;
  int nx, ny, nx_pad;
  double keep, kh;        // 1 - 1/tau, and half of it
  double k1, k3, k45;     // k1 = 1/(9 tau), 3 k1, 4.5 k1
  double u0;              // inflow centreline velocity
  float fomega, fu0;      // 1/tau and u0 in float
};

enum FlowMode { kFlowStep = 0, kFlowU = 1, kFlowCheck = 2, kFlowInit = 3 };

// 1 / v.  In double, a float estimate is refined by two Newton steps
// r <- r + r (1 - v r): four FMAs of the narrow double pipe in place of a
// division's, to within an ulp of it.  The conversions to float and back are
// shifts of the bit patterns (they would be FP64 operations too).  Values
// outside 2^-60 .. 2^60 (a lattice that diverges) are divided.
__device__ __forceinline__ double reciprocal(double v) {
  const unsigned hi = __double2hiint(v), lo = __double2loint(v);
  const unsigned sign = hi & 0x80000000u, mag = hi & 0x7FFFFFFFu;
  if (mag - ((1023u - 60u) << 20) >= (120u << 20)) return 1.0 / v;
  constexpr unsigned kBias = (1023u - 127u) << 20;
  const float f = __uint_as_float(((mag - kBias) << 3) | (lo >> 29));
  const unsigned e = __float_as_uint(__fdividef(1.0f, f));
  double r = __hiloint2double(static_cast<int>(sign | ((e >> 3) + kBias)),
                              static_cast<int>(e << 29));
  r = fma(r, fma(-v, r, 1.0), r);
  return fma(r, fma(-v, r, 1.0), r);
}

// One flow step.  The double step is bound by this part's FP64 pipe (two
// lanes per clock and SM; HBM is busy to a tenth).  Two divisions and nine
// equilibria took about 140 double operations a node and 235 us per step of a
// 2048 x 512 lattice; by opposite pairs it takes about 60 and 130 us.  (A 200 x
// 100 lattice: 14.6 and 8.5 us, with 64-thread blocks that reach every SM.)
// With constants that conserve mass (lbm_flow_solve) its velocities are 2e-15
// to 7e-15 off an 80-bit run of the same scheme after 400 steps, over tau 0.56
// to 1.3 and six lattices; the former step's, whose rounded weights lose mass,
// were 1.2e-13 to 2.8e-13 off.
// BLOCKS: per SM, to bound the registers by (see flow_blocks_per_sm).
template <class P, int MODE, int BX, int BLOCKS>
__global__ void __launch_bounds__(BX, BLOCKS) flow_kernel(const FlowArgs a) {
  using S = typename P::S;
  using T = typename P::T;
  const int x = blockIdx.x * BX + threadIdx.x;
  const int y = blockIdx.y;
  const long long n = (long long)y * a.nx_pad + x;
  const long long plane = a.plane;
  const uint32_t lw = (x < a.nx_pad) ? a.links[n] : kSolidNode;
  T acc[1][2] = {{T(0), T(0)}};
  T *U = static_cast<T *>(a.u);

  if (lw != kSolidNode) {
    const S *src = static_cast<const S *>(a.src);
    S *__restrict__ dst = static_cast<S *>(a.dst);
    const long long np = (long long)a.nx_pad;
    auto ld = [&](int i, long long m) -> T {
      return P::load(src[(long long)i * plane + m]);
    };
    // inflow parabola at this row, zeros half a node outside the walls
    // (evaluated only where it is used: the initial state and inlet links;
    // its division is a sizeable share of an FP64 node update)
    auto inflow = [&]() -> T {
      const T yy = T(y);
      return T(4) * pick<T>(a.u0, a.fu0) * (yy + T(0.5)) * (T(a.ny) - T(0.5) - yy) /
             (T(a.ny) * T(a.ny));
    };

    T f[9];
    const T uw = x == 0 ? inflow() : T(0);   // inlet links
    wait_for_previous();
    if (MODE == kFlowInit) {
      const T uin = inflow();
      const T uu = uin * uin;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const T cu = T(cx(i)) * uin;
        f[i] = Lattice<T>::w(i) *
               (T(1) + T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu);
      }
    } else if (lw == 0u) {
#pragma unroll
      for (int i = 0; i < 9; ++i) f[i] = ld(i, n - (cy(i) * np + cx(i)));
    } else {
      // one load per population from a selected place, as in the ADR step:
      // the neighbour's where it is a fluid node, else the node's own
      // opposite population, to which the link's rule is then applied
      bool outlet = false;
      f[0] = ld(0, n);
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const uint32_t t = nib(lw, opp(i));
        const bool pulled = t == kFluid || t == kPeriodic;
        outlet = outlet || t == kOutlet;
        const long long m = t == kPeriodic ? neighbour(x, y, opp(i), a.nx, a.ny, np)
                                           : n - (cy(i) * np + cx(i));
        f[i] = ld(pulled ? i : opp(i), pulled ? m : n);
      }
      T uwx = T(0), uwy = T(0);
      if (outlet) {   // velocity of the boundary node at time t
        T own[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) own[j] = ld(j, n);
        T r = T(0), jx = T(0), jy = T(0);
#pragma unroll
        for (int j = 0; j < 9; ++j) {
          r += own[j];
          jx += T(cx(j)) * own[j];
          jy += T(cy(j)) * own[j];
        }
        if constexpr (sizeof(T) == 8) {
          const T q = reciprocal(r);
          uwx = jx * q;
          uwy = jy * q;
        } else {
          uwx = jx / r;
          uwy = jy / r;
        }
      }
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const uint32_t t = nib(lw, opp(i));
        if (t == kInlet) {
          // velocity bounce-back, rho_w = 1, u_w = (u_in(y), 0)
          f[i] += T(6) * Lattice<T>::w(i) * T(cx(i)) * uw;
        } else if (t == kOutlet) {
          // pressure anti-bounce-back, rho_w = 1, u_w = u(x_b, t)
          const T cu = T(cx(i)) * uwx + T(cy(i)) * uwy;
          const T uu = uwx * uwx + uwy * uwy;
          f[i] = T(2) * Lattice<T>::w(i) * (T(1) + T(4.5) * cu * cu - T(1.5) * uu) - f[i];
        }
      }
    }

    T ux, uy;
    if constexpr (sizeof(T) == 8) {
      // BGK by opposite pairs (i, j): sum s = f_i + f_j, difference d.  The
      // equilibrium's even part depends on rho and the products of j = rho u,
      // its odd part on j alone, so one reciprocal of rho serves all nine, and
      //   f_i', f_j' = h +- e,  h = (1 - om)/2 s + om even, e = (1 - om)/2 d + om odd.
      const T s1 = f[1] + f[3], d1 = f[1] - f[3], s2 = f[2] + f[4], d2 = f[2] - f[4];
      const T s5 = f[5] + f[7], d5 = f[5] - f[7], s6 = f[6] + f[8], d6 = f[6] - f[8];
      const T rho = f[0] + ((s1 + s2) + (s5 + s6));
      const T jx = d1 + (d5 - d6), jy = d2 + (d5 + d6);
      const T q = reciprocal(rho);
      const T keep = a.keep, kh = a.kh;
      const T k1 = a.k1, k3 = a.k3;
      // 4.5 k1 (jx jx, jy jy, jx jy) / rho and k1 rho
      const T q1 = a.k45 * q;
      const T vx = jx * q1, vy = jy * q1;
      const T X = vx * jx, Y = vy * jy, Z = vx * jy;
      const T Q = X + Y;
      const T t = k1 * rho - T(1) / T(3) * Q;   // om even of f_1 less X
      const T t5 = Q + t;                       // 4 om even of f_5 less 2 Z
      const T bx = k3 * jx, by = k3 * jy;
      S *__restrict__ o = dst + n;
      o[0] = P::store(keep * f[0] + T(4) * t);
      auto put = [&](int i, int j, T h, T e) {
        o[(long long)i * plane] = P::store(h + e);
        o[(long long)j * plane] = P::store(h - e);
      };
      put(1, 3, kh * s1 + (X + t), kh * d1 + bx);
      put(2, 4, kh * s2 + (Y + t), kh * d2 + by);
      put(5, 7, T(0.25) * (T(2) * Z + t5) + kh * s5, T(0.25) * (bx + by) + kh * d5);
      put(6, 8, T(0.25) * (T(-2) * Z + t5) + kh * s6, T(0.25) * (by - bx) + kh * d6);
      ux = jx * q;
      uy = jy * q;
    } else {
      // single precision is bound by HBM, and its constants, rounded one by
      // one, would let the pairs' density drift by 1e-8 a step
      T rho = T(0), jx = T(0), jy = T(0);
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        rho += f[i];
        jx += T(cx(i)) * f[i];
        jy += T(cy(i)) * f[i];
      }
      ux = jx / rho;
      uy = jy / rho;
      const T uu = ux * ux + uy * uy;
      const T om = a.fomega;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const T cu = T(cx(i)) * ux + T(cy(i)) * uy;
        const T feq = Lattice<T>::w(i) * rho *
                      (T(1) + T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu);
        dst[(long long)i * plane + n] = P::store(f[i] + om * (feq - f[i]));
      }
    }
    if (MODE == kFlowU || MODE == kFlowCheck) {
      if (MODE == kFlowCheck) {
        acc[0][0] = absT(ux - U[n]) + absT(uy - U[plane + n]);
        acc[0][1] = absT(ux) + absT(uy);
      }
      U[n] = ux;
      U[plane + n] = uy;
    }
  } else if ((MODE == kFlowU || MODE == kFlowCheck) && x < a.nx_pad) {
    wait_for_previous();
    U[n] = T(0);
    U[plane + n] = T(0);
  }

  if constexpr (MODE == kFlowCheck) {
    wait_for_previous();
    const long long b = (long long)blockIdx.y * gridDim.x + blockIdx.x;
    block_partials_store<2, 0, 1, BX, T>(acc, a.partials + b * 2);
  }
}

// ---------------------------------------------------------------------------
// launchers (one translation unit per precision instantiates them)
// ---------------------------------------------------------------------------
// Threads per block of a step (= nodes of a row segment, and entries of a
// boundary chunk).  FP32 and FP64: 256 on large lattices, whose kernels bound
// their registers to keep warps in flight, else 64, without that bound and
// reaching every SM.  The line is where 256-thread blocks are sixteen per SM
// for FP32 (1000 x 300, three species: 15.5 us per step with 256 threads and
// 9.3 with 64; 700 x 400, two species: 7.7 and 6.5; 2048 x 512: 42 and 50),
// four for FP64 (700 x 400, two species: 25 and 29 us; 200 x 100 has 100 such
// blocks), and where they would cover a quarter more than the row.  FP16
// storage: 256-node segments throughout, which its kernels cover with 64
// (plain) and 128 (check) threads.
inline int adr_block_x(int prec, int nx_pad, int ny) {
  if (prec == LBM_F16DEV) return kBlockX;
  const long long seg = (nx_pad + 255) / 256, few = (prec == LBM_F64 ? 4 : 16) * kSMs;
  return seg * ny < few || seg * 256 * 4 > 5LL * nx_pad ? 64 : 256;
}
// Grid of a step: nxb row segments per row and the boundary chunks of bthreads
// nodes, in one dimension (step_block).
struct AdrGrid {
  int nxb;            // row segments per row
  long long chunks;   // boundary chunks
  int ny;
  long long blocks() const { return static_cast<long long>(nxb) * ny + chunks; }
  dim3 dim() const { return dim3(static_cast<unsigned>(blocks())); }
};
inline AdrGrid adr_grid(int nx_pad, int ny, long long nbnd, int bx, int bthreads) {
  return {(nx_pad + bx - 1) / bx, (nbnd + bthreads - 1) / bthreads, ny};
}
// The grid's numbers for step_block.  Where the chunks go: every other block from
// the start, so that none of them, which take longest, starts late (evenly over
// the grid 1000 x 300 FP32, three species, took 11.7 us per step instead of
// 9.3, 2048 x 512 FP64 121 instead of 113); from twelve waves of blocks evenly,
// so that the latency of their scattered loads hides behind the segments'
// streams and they run near the segments whose lines they share (the list goes
// by rows too), up to two waves from the end, or to the end where they are a
// sixth of the blocks (4096 x 2048 half, one species and thin fibers everywhere:
// 209 us per step up to two waves, 192 to the end).
//
// share is rounded up, so that after `span` blocks all chunks have been passed
// (step_block takes no more).  i / nxb for i < 2^31 is i ceil(2^(31 + s) / nxb) /
// 2^(31 + s), s the bits of nxb - 1: the product is off by less than i 2^s <
// 2^(31 + s).
inline void set_grid(AdrArgs &a, const AdrGrid &g, int bx) {
  const long long wave = kSMs * (bx == 64 ? 8 : 4), blocks = g.blocks();
  long long span = 2 * g.chunks + 1;
  if (blocks >= 12 * wave)
    span = 6 * g.chunks >= blocks ? blocks : std::max(span, blocks - 2 * wave);
  span = std::min(span, blocks);
  a.nxb = g.nxb;
  a.chunks = static_cast<unsigned>(g.chunks);
  a.share = static_cast<unsigned>(
      ((static_cast<unsigned long long>(g.chunks) << 32) + span - 1) / span);
  int s = 1;
  while ((1ll << s) < g.nxb) ++s;
  a.rowshift = s - 1;
  a.rowmul = static_cast<unsigned>(((1ull << (31 + s)) + g.nxb - 1) / g.nxb);
}
inline int flow_block_x(int nx_pad, int ny) {
  return adr_block_x(LBM_F32, nx_pad, ny);
}
// 256-thread blocks per SM that the flow step bounds its registers by (0: none).
// FP32 lattices whose populations don't fit L2 need the eight that 32 registers
// allow, though their boundary nodes spill a little: 4096 x 2048 108 us per step
// without a bound, 100 with; 2048 x 700 19.2 and 18.8; but 2048 x 512 11.5 and
// 12.1.
inline int flow_blocks_per_sm(int prec, int nx_pad, int ny) {
  return prec == LBM_F32 && flow_block_x(nx_pad, ny) == 256 &&
                 static_cast<long long>(nx_pad) * ny >= 5ll << 18
             ? 8
             : 0;
}
inline dim3 flow_grid(int nx_pad, int ny) {
  const int bx = flow_block_x(nx_pad, ny);
  return dim3(static_cast<unsigned>((nx_pad + bx - 1) / bx),
              static_cast<unsigned>(ny));
}
inline dim3 adr_node_grid(int nx_pad, int ny) {
  return dim3(static_cast<unsigned>((nx_pad + kBlockX - 1) / kBlockX),
              static_cast<unsigned>(ny));
}
// of the adjoint: one node per thread
inline dim3 adj_grid(int prec, int nx_pad, int ny) {
  const int bx = adr_block_x(prec, nx_pad, ny);
  return dim3(static_cast<unsigned>((nx_pad + bx - 1) / bx), static_cast<unsigned>(ny));
}
// boundary entries per chunk of a check step
inline int adr_check_threads(int prec, int nx_pad, int ny) {
  return prec == LBM_F16DEV ? kPairThreads : adr_block_x(prec, nx_pad, ny);
}
// partial-sum rows written by one check step
inline long long adr_partial_rows(int prec, int nx_pad, int ny, long long nbnd) {
  const AdrGrid g = adr_grid(nx_pad, ny, nbnd, adr_block_x(prec, nx_pad, ny),
                             adr_check_threads(prec, nx_pad, ny));
  return g.blocks();
}

template <class P>
cudaError_t launch_adr(int ns, int mode, const AdrArgs &a, cudaStream_t st,
                       bool chained = false);
// two plain steps in one launch (FP32), and whether they are worth it
bool two_step_pays(int prec, int ns, int nx, int ny);
cudaError_t launch_adr_two_step(int ns, const AdrArgs &a, cudaStream_t st);
template <class P>
cudaError_t launch_adr_flux(int ns, const void *g, const RefT *ref,
                            const uint32_t *links, long long plane, int nx_pad,
                            int ny, int xp, double *out, cudaStream_t st);
template <class P>
cudaError_t launch_flow(int mode, const FlowArgs &a, cudaStream_t st, bool chained);
template <class P>
cudaError_t launch_adjoint(int ns, int mode, const AdjArgs &a, cudaStream_t st,
                           bool chained);
// FP64 equilibrium-factor table of a velocity field (defined with the FP64
// kernels)
cudaError_t launch_eq_table(const double *u, long long plane, double *etab,
                            cudaStream_t st);
template <class P>
cudaError_t launch_adjoint_grad(int ns, const AdjArgs &a, const BoundaryNode *bnodes,
                                long long nbnd, const void *conc, double *dkab,
                                double *dkbc, const int32_t *fiber, double *dw,
                                double k1, double k2, cudaStream_t st);

// Two-level deterministic fold of nb rows of ks + km partials (ks sums, km
// minima) into out[0..ks+km); scratch holds kReduceGrid * (ks + km)
// doubles.  (ks, km) is (2, 0) (flow and adjoint residuals) or
// (2 ns, ns) (ADR check steps).
constexpr int kReduceGrid = 256;
cudaError_t launch_reduce(int ks, int km, const double *partials, long long nb,
                          double *scratch, double *out, cudaStream_t st);

// Slots of a solver's result buffer: the folded check partials
// [2 ns sums | ns minima] from 0, the outfluxes from kResFlux.
constexpr int kResFlux = 16;
constexpr int kResSlots = 24;

}  // namespace lbm
