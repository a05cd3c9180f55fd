// Two plain FP32 steps in one pass over memory.  Included by lbm_kernels.cuh.
#pragma once

namespace lbm {

// A block owns a strip of BX - 2 columns and a run of rows, one column per
// thread (the first and the last thread are the neighbouring strips').  It
// walks down the rows: iteration r updates row r once from the global planes
// (t -> t+1) into a ring of four rows in shared memory, and then row r - 1 a
// second time (t+1 -> t+2) from the ring rows r - 2 .. r, which it writes to
// the global planes.  So memory is read and written once per two steps; the
// nodes around a strip are updated by its neighbours too (2 columns of BX,
// 2 rows of each run of rows + 2).
//
// The ring's fourth row lets one barrier per iteration do: what iteration
// r + 1 overwrites was last read in iteration r - 1.  The loads of row r + 1
// are issued before that barrier and the second update of row r - 1, their
// lines prefetched into L2 two rows earlier, its link word and velocity a row
// earlier.
//
// A node's update costs as much as in the one-step kernel, and 16 warps per
// SM (128 registers; 2 x 108 KB of ring) do not hide all of its latency, so
// the step is not at HBM's rate any more: 1.68 ms per step of the 16384 x
// 4096 lattice of three species, against 2.31 ms for the one-step kernel at
// 95% of the copy bandwidth.  Runs of at most 32 rows keep what all blocks
// touch at a time within a few pages of every plane: with 128 rows a 4096 x
// 2048 lattice took twice as long.  Strips of 126 columns (4 blocks per SM)
// took 1.75 ms; two columns per thread, with packed arithmetic, 1.89 ms; a
// warp per strip with the rows in registers and shuffles instead of shared
// memory 1.96 ms; the link rates loaded link by link 1.91 ms.
template <int NS>
struct TwoStep {
  static constexpr int kBX = 256;
  static constexpr int kOwned = kBX - 2;
  static constexpr int kBlocks = 2;           // per SM
  static constexpr int kRow = 9 * NS * kBX;   // floats of a ring row
  static constexpr int kShared = 4 * kRow * sizeof(float);
  static constexpr int kPrefetch = 2;         // rows ahead of the loads
};

// which populations i of a node are pulled across a link that is not to a
// fluid node (bit i): the node's own opposite population is read instead
__device__ __forceinline__ uint32_t bounce_mask(uint32_t lw) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const uint32_t t = nib(lw, opp(i));
    m |= (t != kFluid && t != kPeriodic ? 1u : 0u) << i;
  }
  return m;
}
__device__ __forceinline__ uint32_t type_mask(uint32_t lw, uint32_t type) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 1; i < 9; ++i) m |= (nib(lw, opp(i)) == type ? 1u : 0u) << i;
  return m;
}
// edge_rules for the links of `mask`, wall value v (c_in or the node's own
// concentration)
__device__ __forceinline__ void edge_mask_rules(uint32_t mask, float v, float (&g)[9]) {
#pragma unroll
  for (int i = 1; i < 9; ++i)
    if (mask >> i & 1u) g[i] = fma_rn(2.0f * Lattice<float>::w(i), v, -g[i]);
}

template <int NS>
__global__ void __launch_bounds__(TwoStep<NS>::kBX, TwoStep<NS>::kBlocks)
    adr_two_step_kernel(const AdrArgs a, int rows) {
  using K = TwoStep<NS>;
  constexpr int BX = K::kBX;
  extern __shared__ float ring[];   // [4][NS * 9][BX]
  const int tid = threadIdx.x;
  const int x = blockIdx.x * K::kOwned - 1 + tid;
  // Columns and rows beyond an edge are the other side's, whether the edge is
  // periodic or not: only the link words say so, and they may be uploaded anew
  // between launches.  Without periodic links no node reads them.
  const int xw = x < 0 ? a.nx - 1 : x < a.nx ? x : x == a.nx ? 0 : -1;
  const bool owned = tid >= 1 && tid <= K::kOwned && x < a.nx;
  const bool edge = xw == 0 || xw == a.nx - 1;
  const int y0 = blockIdx.y * rows, y1 = min(y0 + rows, a.ny);
  const unsigned plane = static_cast<unsigned>(a.plane), np = a.nx_pad;
  const float *__restrict__ src = static_cast<const float *>(a.src);
  float *__restrict__ dst = static_cast<float *>(a.dst);
  const float *__restrict__ U = static_cast<const float *>(a.u);

  auto wrap_y = [&](int r) { return r < 0 ? r + a.ny : r >= a.ny ? r - a.ny : r; };
  struct Row {
    uint32_t lw;
    float ux, uy;
  };
  auto row = [&](int r) -> Row {
    const int y = wrap_y(r);
    Row k{kSolidNode, 0.0f, 0.0f};
    if (xw >= 0 && r <= y1) {
      const unsigned n = y * np + xw;
      k.lw = a.links[n];
      k.ux = U[n];
      k.uy = U[plane + n];
    }
    return k;
  };
  float g[NS][9];   // the loaded populations of row r, then of row r + 1
  auto load = [&](int r, uint32_t lw) {
    const int y = wrap_y(r);
    const unsigned n = y * np + xw;
    unsigned off[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) off[i] = i * plane + n - cy(i) * np - cx(i);
    if (lw != 0u) {
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const uint32_t t = nib(lw, opp(i));
        if (t == kPeriodic)
          off[i] = i * plane + static_cast<unsigned>(neighbour(xw, y, opp(i), a.nx, a.ny, np));
        else if (t != kFluid)
          off[i] = opp(i) * plane + n;
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
#pragma unroll
      for (int i = 0; i < 9; ++i) g[s][i] = src[s * 9 * plane + off[i]];
    }
  };

  Row prev{kSolidNode, 0.0f, 0.0f}, cur = row(y0 - 1), next = row(y0);
  if (cur.lw != kSolidNode) load(y0 - 1, cur.lw);
  int slot = 0;
  for (int r = y0 - 1; r <= y1; ++r, slot = (slot + 1) & 3) {
    // first step of row r
    if (cur.lw != kSolidNode) {
      float E[9], C[NS], ka[9], kb[9];
      bool cat = false;
      if (cur.lw != 0u) cat = link_rates(a, cur.lw, xw, wrap_y(r), ka, kb);
      eq_factors(cur.ux, cur.uy, E);
      const bool inlet = edge && xw == 0;
      const uint32_t emask = edge ? type_mask(cur.lw, inlet ? kInlet : kOutlet) : 0u;
      float *const o = ring + slot * K::kRow + tid;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        if (emask) {
          float v = a.fcin[s];
          if (!inlet) {
            float own[9];
            const unsigned n = wrap_y(r) * np + xw;
#pragma unroll
            for (int j = 0; j < 9; ++j) own[j] = src[(s * 9 + j) * plane + n];
            v = sum_rn(own);
          }
          if (!inlet || s == 0 || a.abb_all) edge_mask_rules(emask, v, g[s]);
        }
        C[s] = collide(a, s, E, g[s]);
        if (cat) add_source<NS>(a, s, cur.lw, ka, kb, C, g[s]);
#pragma unroll
        for (int i = 0; i < 9; ++i) o[(s * 9 + i) * BX] = g[s][i];
      }
    }
    {   // L2 prefetch, one segment per plane: whole 16-byte groups (nx_pad is
        // a multiple of 32, xs and xe of 4)
      const int yp = r + 1 + K::kPrefetch;
      if (tid < 9 * NS + 3 && yp < min(y1 + 1, a.ny)) {
        const int xl = blockIdx.x * K::kOwned - 1;
        const int xs = max(xl, 0) & ~3, xe = min((xl + BX + 3) & ~3, a.nx_pad);
        const unsigned bytes = 4u * static_cast<unsigned>(xe - xs);
        if (tid < 9 * NS) {
          const int yy = yp - cy(tid % 9);
          if (yy >= 0 && yy < a.ny)
            prefetch_l2(src + (static_cast<unsigned>(tid) * plane + yy * np + xs), bytes);
        } else if (tid < 9 * NS + 2) {
          prefetch_l2(U + ((tid - 9 * NS) * plane + yp * np + xs), bytes);
        } else {
          prefetch_l2(a.links + (yp * np + xs), bytes);
        }
      }
    }
    const Row after = row(r + 2);
    if (next.lw != kSolidNode) load(r + 1, next.lw);
    __syncthreads();
    // second step of row r - 1
    if (r > y0 && owned && prev.lw != kSolidNode) {
      const int y = wrap_y(r - 1);
      const unsigned n = y * np + xw;
      float E[9], C[NS], ka[9], kb[9];
      bool cat = false;
      if (prev.lw != 0u) cat = link_rates(a, prev.lw, xw, y, ka, kb);
      eq_factors(prev.ux, prev.uy, E);
      // ring rows of y - 1, y and y + 1
      const int row0[3] = {((slot + 2) & 3) * K::kRow + tid, ((slot + 3) & 3) * K::kRow + tid,
                           slot * K::kRow + tid};
      int at[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) at[i] = row0[1 - cy(i)] + i * BX - cx(i);
      uint32_t emask = 0u;
      const bool inlet = edge && xw == 0;
      if (prev.lw != 0u) {
        const uint32_t b = bounce_mask(prev.lw);
#pragma unroll
        for (int i = 1; i < 9; ++i)
          if (b >> i & 1u) at[i] = row0[1] + opp(i) * BX;
        if (edge) emask = type_mask(prev.lw, inlet ? kInlet : kOutlet);
      }
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        float h[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = ring[at[i] + s * 9 * BX];
        if (emask) {
          float v = a.fcin[s];
          if (!inlet) {
            float own[9];
#pragma unroll
            for (int j = 0; j < 9; ++j) own[j] = ring[row0[1] + (s * 9 + j) * BX];
            v = sum_rn(own);
          }
          if (!inlet || s == 0 || a.abb_all) edge_mask_rules(emask, v, h);
        }
        C[s] = collide(a, s, E, h);
        if (cat) add_source<NS>(a, s, prev.lw, ka, kb, C, h);
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(s * 9 + i) * plane + n] = h[i];
      }
    }
    prev = cur;
    cur = next;
    next = after;
  }
}

// Rows per run, and what a launch then costs (in iterations of all the chip's
// blocks).  A run of `rows` rows takes rows + 2 iterations and about 1.5 more
// to start (on a lattice of one run or two rows + 1.5: its edges are in L2); the
// blocks of all runs share the SMs, with 0.7 of a wave lost to the uneven end.
struct TwoStepPlan {
  int rows;
  double cost;
};
inline TwoStepPlan two_step_plan(int nx, int ny, int owned, int blocks) {
  const long long strips = (nx + owned - 1) / owned;
  TwoStepPlan best{4, -1.0};
  for (int rows = 4; rows <= 32; ++rows) {
    const long long n = strips * ((ny + rows - 1) / rows);
    const double c = (n / (double(kSMs) * blocks) + 0.7) * (rows + 3.5);
    if (best.cost < 0.0 || c <= best.cost) best = {rows, c};
  }
  if (ny <= 2 * best.rows) best.cost *= (best.rows + 1.5) / (best.rows + 3.5);
  return best;
}

}  // namespace lbm
