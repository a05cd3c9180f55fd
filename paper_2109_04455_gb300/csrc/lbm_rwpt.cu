// Random walk particle tracking (RWPT) of the paper's Sec. III.B: the second,
// independent method for the reaction efficiency of a 2D cross-section.
//
// Each particle (species A, B or C) moves per time step dt by
//   advection  x += dt u(x), u bilinear in the LBM velocity field,
//   diffusion  x += sqrt(4 D dt) (cos t, sin t), t uniform,
// reflects elastically off the channel walls and the fibers, reacts with
// probability k dt per step while within a reactive shell of width delta
// around a catalytic fiber (A -> B at rate k_AB, B -> C at rate k_BC), and
// is counted per species when it leaves through the outlet.  The entrance
// strip x in [-1/2, 1/2) is held at a fixed density of A: every step the A
// particles that ended there are removed and the strip is seeded anew.
//
// Random numbers: draw k of particle `id` at step t is the (64 t + k + 1)-th
// output of the particle's SplitMix64 stream (Steele, Lea and Flood, OOPSLA
// 2014), whose seed is output id + 1 of the stream of the run's seed.  A
// particle's path thus depends only on (seed, id), not on where it is
// stored.  The direction is drawn by rejection from the unit disc, and every
// floating-point step is an IEEE operation with one rounding (explicit
// round-to-nearest intrinsics, no contraction), so a plain CPU restatement
// of the same steps reproduces every position bit for bit.
//
// Storage: structure of arrays in two buffers (ping-pong); a step compacts
// the survivors of one buffer into the other (warp ballots, one atomic per
// warp) and appends the new entrance particles.  Counts live on the device,
// so steps need no host synchronisation.
//
// What bounds a step is the FP64 pipe (two lanes per clock and SM here, a
// 64th of the float rate), not memory (0.5% of HBM).  So decisions are taken
// in float or integers wherever those can be certain of the double's answer
// (which fibers are near, which direction candidates lie in the disc, the
// wall and edge tests), the double test runs only in between, and the
// direction's square root and divisions share their Newton steps.  The
// results are the same bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "lbm_internal.h"
#include "lbm_nvtx.h"

namespace lbm {
namespace rwpt {

constexpr unsigned long long kGamma = 0x9E3779B97F4A7C15ull;
constexpr int kDraws = 64;       // draws reserved per particle and step
constexpr int kTries = 16;       // direction candidates (2 draws each)
constexpr int kReactDraw = 40;   // draw index of the reaction test
constexpr int kSpawnDraw = 48;   // draws of a new particle's position
constexpr int kReflections = 4;  // reflection passes per step
constexpr int kThreads = 256;

__host__ __device__ inline unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ inline unsigned long long particle_seed(unsigned long long seed,
                                                   unsigned long long id) {
  return mix64(seed + (id + 1ull) * kGamma);
}
// uniform double in [0, 1): the top 53 bits of the draw
__device__ inline double draw(unsigned long long ps, long long t, int k) {
  const unsigned long long c =
      static_cast<unsigned long long>(t) * kDraws + static_cast<unsigned>(k) + 1ull;
  return static_cast<double>(mix64(ps + c * kGamma) >> 11) * 0x1.0p-53;
}

// a fiber as the particles see it
struct Fiber {
  double cx, cy;
  double rp;      // reflecting radius
  double kab, kbc;
  double nx, ny;  // side-by-side fiber: A -> B where (p - c).n >= 0
  int split;      // 1: side-by-side (rates by side), 0: rates everywhere
  int pad;
};

// the same for the float test of which fibers are near: centre, and a bound
// that the float distance squared exceeds only where the double distance is
// beyond both the reflecting radius and the shell
struct Near {
  float cx, cy, d2, pad;
};

struct Args {
  int nx, ny, nx_pad, nfib;
  int nspecies;
  int periodic;      // box periodic in x and y: no inlet, outlet or walls
  int homogeneous;   // every particle reacts, wherever it is
  int plain;         // step length outside unit_step's range
  int moves;         // step length above zero
  double dnx, dny;   // nx, ny
  double xout, ytop; // nx - 1/2, ny - 1/2
  double dt, len, delta;   // time step, diffusion step length, shell width
  double hk1, hk2;         // homogeneous rates (A -> B, B -> C)
  unsigned long long seed;
  const double *u;         // [2][ny][nx_pad]
  const Fiber *fib;
  const Near *near;
};

struct Buf {
  double *x, *y;
  unsigned long long *id;
  int *s;
};

// Counters (device, unsigned long long): three particle counts in turn (of
// the buffer read, of the buffer written, and one that the step clears for
// the next), the outflow of each species since the last reset, the overflow
// flag, and the blocks that have finished a step that may run out of room (zero
// between steps).  A count can pass the capacity when particles are dropped for
// lack of room (the appends count them, the slots refuse them), so every reader
// takes min(count, capacity).
enum { kCount = 0, kOut = 3, kOverflow = 6, kDone = 7, kCounters = 8 };

__device__ inline double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ inline double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ inline double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ inline double ddiv(double a, double b) { return __ddiv_rn(a, b); }

__device__ inline long long bits(double v) { return __double_as_longlong(v); }
// v < t, for a threshold t that is not zero, by integer comparison of the bit
// patterns (a comparison in double is an FP64 operation); a NaN counts as
// beyond the infinity of its sign
__device__ inline long long key(double v) {
  return bits(v) ^ ((bits(v) >> 63) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ inline bool below(double v, double t) { return key(v) < key(t); }
// the same where a NaN matters, which a velocity field may hold, of either
// sign: false for it (from -infinity up, by distance in one unsigned test)
__device__ inline bool number_below(double v, double t) {
  constexpr unsigned long long kLow = 0x800FFFFFFFFFFFFFull;   // key of -infinity
  return key(v) - kLow < key(t) - kLow;
}

// floor(v) as a double and as an integer.  Adding 1.5 * 2^52 rounded down
// leaves floor(v) in the low bits of the sum, for |v| < 2^30.
__device__ inline double floor_int(double v, int &i) {
  constexpr double kMagic = 6755399441055744.0;
  if ((__double2hiint(v) & 0x7FFFFFFF) < 0x41D00000) {
    const double m = __dadd_rd(v, kMagic);
    i = __double2loint(m);
    return dsub(m, kMagic);
  }
  const double f = floor(v);
  i = static_cast<int>(f);
  return f;
}

// u at (px, py): bilinear in the four nodes around the point (node indices
// clamped to the lattice)
__device__ inline void velocity(const Args &a, double px, double py,
                                double &ux, double &uy) {
  int i0, j0;
  const double fx0 = floor_int(px, i0), fy0 = floor_int(py, j0);
  const double fx = dsub(px, fx0), fy = dsub(py, fy0);
  int i1 = i0 + 1, j1 = j0 + 1;
  i0 = min(max(i0, 0), a.nx - 1);
  i1 = min(max(i1, 0), a.nx - 1);
  j0 = min(max(j0, 0), a.ny - 1);
  j1 = min(max(j1, 0), a.ny - 1);
  const double gx = dsub(1.0, fx), gy = dsub(1.0, fy);
  const double w00 = dmul(gx, gy), w10 = dmul(fx, gy);
  const double w01 = dmul(gx, fy), w11 = dmul(fx, fy);
  const long long plane = static_cast<long long>(a.nx_pad) * a.ny;
  const long long n00 = static_cast<long long>(j0) * a.nx_pad + i0;
  const long long n10 = static_cast<long long>(j0) * a.nx_pad + i1;
  const long long n01 = static_cast<long long>(j1) * a.nx_pad + i0;
  const long long n11 = static_cast<long long>(j1) * a.nx_pad + i1;
  ux = dadd(dadd(dadd(dmul(w00, a.u[n00]), dmul(w10, a.u[n10])),
                 dmul(w01, a.u[n01])), dmul(w11, a.u[n11]));
  uy = dadd(dadd(dadd(dmul(w00, a.u[plane + n00]), dmul(w10, a.u[plane + n10])),
                 dmul(w01, a.u[plane + n01])), dmul(w11, a.u[plane + n11]));
}

// 2 d - 1 of the draw d = k 2^-53 in [0, 1) whose generator output is z
// (k its top 53 bits): the low 52 bits of k are the mantissa of a number in
// [1, 2), which is exactly 1 or 2 above the result.
__device__ inline double centred(unsigned long long z) {
  const double m = __longlong_as_double(static_cast<long long>(
      ((z >> 11) & 0xFFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
  return dsub(m, (z >> 63) ? 1.0 : 2.0);
}
// the same to within 2^-23, in float
__device__ inline float centred_float(unsigned long long z) {
  return static_cast<float>(static_cast<int>(
             static_cast<unsigned>(z >> 32) ^ 0x80000000u)) * 0x1.0p-31f;
}

// v to float by shifting its bits, rounded towards zero (a conversion is an
// FP64 operation): within 2^-23 of v for 2^-126 <= |v| < 2^127, 0 for smaller
// values, NaN for larger ones.
__device__ inline float shift_to_float(double v) {
  constexpr unsigned kBias = (1023u - 127u) << 20;
  const unsigned hi = __double2hiint(v), lo = __double2loint(v);
  const unsigned mag = hi & 0x7FFFFFFFu;
  if (mag < kBias + (1u << 20)) return 0.0f;
  if (mag >= kBias + (254u << 20)) return __uint_as_float(0x7FC00000u);
  return __uint_as_float((hi & 0x80000000u) | ((mag - kBias) << 3) | (lo >> 29));
}
// a positive normal float to double
__device__ inline double shift_to_double(float f) {
  const unsigned e = __float_as_uint(f);
  return __hiloint2double(static_cast<int>((e >> 3) + ((1023u - 127u) << 20)),
                          static_cast<int>(e << 29));
}

// (len v1 / r, len v2 / r), r = sqrt(q), each operation correctly rounded.
// The square root is Goldschmidt's iteration from a float estimate with
// Markstein's final correction, the quotients Markstein's division by a
// shared reciprocal (P. Markstein, "Computation of elementary functions on
// the IBM RISC System/6000 processor", 1990): the reciprocal is correctly
// rounded except for an all-ones mantissa, which is divided plainly, and
// each quotient is corrected twice, the second time from an estimate within
// an ulp, whose remainder is exact.  24 double operations in place of the
// roughly 60 of one square root and two divisions.
__device__ inline void unit_step(const Args &a, double v1, double v2, double q,
                                 double &sx, double &sy) {
  const double n1 = dmul(a.len, v1), n2 = dmul(a.len, v2);
  if (a.plain) {   // a step length whose remainders could leave the range
    const double r = __dsqrt_rn(q);
    sx = ddiv(n1, r);
    sy = ddiv(n2, r);
    return;
  }
  const double y0 = shift_to_double(rsqrtf(shift_to_float(q)));
  double g = q * y0, h = 0.5 * y0;
  double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  const double r = fma(fma(-g, g, q), h, g);
  if ((bits(r) & 0xFFFFFFFFFFFFFll) == 0xFFFFFFFFFFFFFll) {
    sx = ddiv(n1, r);
    sy = ddiv(n2, r);
    return;
  }
  double y = h + h;
  y = fma(y, fma(-r, y, 1.0), y);
  y = fma(y, fma(-r, y, 1.0), y);
  double s1 = n1 * y, s2 = n2 * y;
  s1 = fma(fma(-s1, r, n1), y, s1);
  s2 = fma(fma(-s2, r, n2), y, s2);
  sx = fma(fma(-s1, r, n1), y, s1);
  sy = fma(fma(-s2, r, n2), y, s2);
}

// Whether fiber k may hold (fx, fy) within its reflecting radius or shell.
__device__ inline bool may_hold(const Near &f, float fx, float fy) {
  const float dx = fx - f.cx, dy = fy - f.cy;
  return !(dx * dx + dy * dy > f.d2);
}

// Mirror p at the circle of radius rp about c if p is inside it:
// the distance to the centre d becomes 2 rp - d along the same ray.
__device__ inline bool reflect_fiber(const Fiber &f, double &px, double &py) {
  const double dx = dsub(px, f.cx), dy = dsub(py, f.cy);
  const double d2 = dadd(dmul(dx, dx), dmul(dy, dy));
  const double r2 = dmul(f.rp, f.rp);
  if (!(d2 < r2)) return false;
  if (d2 == 0.0) {   // at the centre: out along +x
    px = dadd(f.cx, f.rp);
    return true;
  }
  const double d = __dsqrt_rn(d2);
  const double q = ddiv(dsub(dmul(2.0, f.rp), d), d);
  px = dadd(f.cx, dmul(q, dx));
  py = dadd(f.cy, dmul(q, dy));
  return true;
}

__device__ inline double wrap(double v, double lo, double span) {
  // v in [lo - span, lo + 2 span): back into [lo, lo + span)
  if (v < lo) return dadd(v, span);
  if (!(v < dadd(lo, span))) return dsub(v, span);
  return v;
}

// The rate that applies to a particle of species s at (px, py), or 0: the
// first fiber (list order) whose shell rp <= d < rp + delta holds the point
// and whose catalyst acts on s.  first: the first fiber that may hold it.
__device__ inline double shell_rate(const Args &a, int s, double px,
                                    double py, int first) {
  if (a.homogeneous) return s == 0 ? a.hk1 : (s == 1 ? a.hk2 : 0.0);
  if (first >= a.nfib) return 0.0;
  const float fx = shift_to_float(px), fy = shift_to_float(py);
  for (int j = first; j < a.nfib; ++j) {
    if (!may_hold(a.near[j], fx, fy)) continue;
    const Fiber &f = a.fib[j];
    const double dx = dsub(px, f.cx), dy = dsub(py, f.cy);
    const double d2 = dadd(dmul(dx, dx), dmul(dy, dy));
    const double ro = dadd(f.rp, a.delta);
    if (!(d2 >= dmul(f.rp, f.rp)) || !(d2 < dmul(ro, ro))) continue;
    double kab = f.kab, kbc = f.kbc;
    if (f.split) {
      const bool first = dadd(dmul(dx, f.nx), dmul(dy, f.ny)) >= 0.0;
      kab = first ? f.kab : 0.0;
      kbc = first ? 0.0 : f.kbc;
    }
    const double k = s == 0 ? kab : (s == 1 ? kbc : 0.0);
    if (k > 0.0) return k;
  }
  return 0.0;
}

// Append the kept lanes of a warp to `out` (count in *cnt): one atomic per
// warp.  Returns this lane's slot (or -1), -2 if the buffer is full.
__device__ inline long long warp_slot(bool keep, unsigned long long *cnt,
                                      long long cap, unsigned long long *overflow) {
  const unsigned mask = __ballot_sync(0xffffffffu, keep);
  const int lane = threadIdx.x & 31;
  const int leader = mask ? __ffs(mask) - 1 : 0;
  unsigned long long base = 0;
  if (mask && lane == leader) base = atomicAdd(cnt, static_cast<unsigned long long>(__popc(mask)));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (!keep) return -1;
  const long long slot =
      static_cast<long long>(base) + __popc(mask & ((1u << lane) - 1u));
  if (slot >= cap) {
    atomicExch(overflow, 1ull);
    return -2;
  }
  return slot;
}

// New particles of species A with ids id0 .. id0 + m - 1, uniform in the
// rectangle [x0, x0 + wx) x [-1/2, ny - 1/2), those inside a fiber dropped,
// appended to `out` by blocks block, block + blocks, ...
__device__ inline void spawn(const Args &a, const Buf &out,
                             unsigned long long *cnt, int kout, long long cap,
                             long long t, unsigned long long id0, long long m,
                             double x0, double wx, int block, int blocks) {
  const long long stride = static_cast<long long>(blocks) * kThreads;
  for (long long base = static_cast<long long>(block) * kThreads; base < m;
       base += stride) {
    const long long j = base + threadIdx.x;
    bool keep = j < m;
    double px = 0.0, py = 0.0;
    const unsigned long long id = id0 + static_cast<unsigned long long>(j);
    if (keep) {
      const unsigned long long ps = particle_seed(a.seed, id);
      px = dadd(x0, dmul(wx, draw(ps, t, kSpawnDraw)));
      py = dadd(-0.5, dmul(a.dny, draw(ps, t, kSpawnDraw + 1)));
      const float fx = shift_to_float(px), fy = shift_to_float(py);
      for (int k = 0; k < a.nfib && keep; ++k) {
        if (!may_hold(a.near[k], fx, fy)) continue;
        const Fiber &f = a.fib[k];
        const double dx = dsub(px, f.cx), dy = dsub(py, f.cy);
        if (dadd(dmul(dx, dx), dmul(dy, dy)) < dmul(f.rp, f.rp)) keep = false;
      }
    }
    const long long slot = warp_slot(keep, cnt + kout, cap, cnt + kOverflow);
    if (slot >= 0) {
      out.x[slot] = px;
      out.y[slot] = py;
      out.s[slot] = 0;
      out.id[slot] = id;
    }
  }
}

// The initial fill.
__global__ void __launch_bounds__(kThreads)
    rwpt_spawn_kernel(const Args a, Buf out, unsigned long long *cnt, int kout,
                      long long cap, long long t, unsigned long long id0,
                      long long m, double x0, double wx) {
  spawn(a, out, cnt, kout, cap, t, id0, m, x0, wx, blockIdx.x, gridDim.x);
}

// One time step: the blocks below `movers` move every particle of `in`
// (count in cnt[kin]) and append the survivors to `out` (count in cnt[kout],
// zero on entry), the others append the m new entrance particles; the third
// count, cnt[kclr], is cleared for the next step.  Particles in the box come
// before new ones: where there might not be room for all, the entrance
// particles wait until every survivor has its slot, and the last block to
// finish appends them.
__global__ void __launch_bounds__(kThreads)
    rwpt_step_kernel(const Args a, Buf in, Buf out, unsigned long long *cnt,
                     int kin, int kout, int kclr, long long cap, long long t,
                     unsigned long long id0, long long m, int movers) {
  if (blockIdx.x == 0 && threadIdx.x == 0) cnt[kclr] = 0ull;
  const long long n = min(static_cast<long long>(cnt[kin]), cap);
  const bool tight = n + m > cap;
  if (static_cast<int>(blockIdx.x) >= movers) {
    if (!tight)
      spawn(a, out, cnt, kout, cap, t, id0, m, -0.5, 1.0, blockIdx.x - movers,
            gridDim.x - movers);
    return;
  }
  const long long stride = static_cast<long long>(movers) * kThreads;
  for (long long base = static_cast<long long>(blockIdx.x) * kThreads; base < n;
       base += stride) {
    const long long i = base + threadIdx.x;
    bool keep = i < n;
    int outflow = -1;
    double px = 0.0, py = 0.0;
    int s = 0;
    unsigned long long id = 0;
    if (keep) {
      px = in.x[i];
      py = in.y[i];
      s = in.s[i];
      id = in.id[i];
      const unsigned long long ps = particle_seed(a.seed, id);
      // advection (Euler)
      if (a.u != nullptr) {
        double ux, uy;
        velocity(a, px, py, ux, uy);
        px = dadd(px, dmul(a.dt, ux));
        py = dadd(py, dmul(a.dt, uy));
      }
      // diffusion: a step of length sqrt(4 D dt) in a uniform direction, the
      // first candidate of the square inside the unit disc.  The float
      // squared radius is within 1e-6 of the double's, so only a candidate
      // near the rim or the centre needs the double.
      if (a.moves) {
        const unsigned long long c0 =
            ps + (static_cast<unsigned long long>(t) * kDraws + 1ull) * kGamma;
        unsigned long long z1 = 0, z2 = 0;
        bool found = false;
        for (int k = 0; k < kTries && !found; ++k) {
          z1 = mix64(c0 + static_cast<unsigned long long>(2 * k) * kGamma);
          z2 = mix64(c0 + static_cast<unsigned long long>(2 * k + 1) * kGamma);
          const float f1 = centred_float(z1), f2 = centred_float(z2);
          const float q = f1 * f1 + f2 * f2;
          if (q > 1.00001f) continue;
          found = true;
          if (!(q < 0.99999f && q > 1e-5f)) {
            const double c1 = centred(z1), c2 = centred(z2);
            const double q2 = dadd(dmul(c1, c1), dmul(c2, c2));
            found = q2 > 0.0 && q2 <= 1.0;
          }
        }
        const double v1 = found ? centred(z1) : 1.0, v2 = found ? centred(z2) : 0.0;
        const double q = dadd(dmul(v1, v1), dmul(v2, v2));
        double sx, sy;
        unit_step(a, v1, v2, q, sx, sy);
        px = dadd(px, sx);
        py = dadd(py, sy);
      }
      // elastic reflections: walls y = -1/2, ny - 1/2 and the fibers
      int first = a.nfib;   // the first fiber that may hold the particle
      for (int pass = 0; pass < kReflections; ++pass) {
        bool hit = false;
        if (a.periodic) {
          px = wrap(px, -0.5, a.dnx);
          py = wrap(py, -0.5, a.dny);
        } else {
          if (below(py, -0.5)) {
            py = dsub(-1.0, py);
            hit = true;
          } else if (below(a.ytop, py)) {
            py = dsub(dmul(2.0, a.ytop), py);
            hit = true;
          }
        }
        float fx = shift_to_float(px), fy = shift_to_float(py);
        first = a.nfib;
        for (int k = 0; k < a.nfib; ++k) {
          if (!may_hold(a.near[k], fx, fy)) continue;
          first = min(first, k);
          if (reflect_fiber(a.fib[k], px, py)) {
            hit = true;
            fx = shift_to_float(px);
            fy = shift_to_float(py);
          }
        }
        if (!hit) break;
        first = 0;   // moved: any fiber may hold it now
      }
      // reaction with probability k dt
      if (s < a.nspecies - 1) {
        const double k = shell_rate(a, s, px, py, first);
        if (k > 0.0 && draw(ps, t, kReactDraw) < dmul(k, a.dt)) s += 1;
      }
      // inlet and outlet (a particle whose x is NaN leaves; a NaN of y costs
      // further reflection passes above that move nothing, and turns x into
      // NaN with the next step's advection)
      if (!a.periodic) {
        if (!number_below(px, a.xout)) {
          outflow = s;
          keep = false;
        } else if (below(px, -0.5)) {
          if (s == 0)
            keep = false;          // back into the reservoir of A
          else
            px = dsub(-1.0, px);   // B and C: the entrance reflects
        }
        if (keep && s == 0 && below(px, 0.5)) keep = false;  // strip: re-seeded
      }
    }
    // outflow counts (one atomic per warp and species)
#pragma unroll
    for (int sp = 0; sp < 3; ++sp) {
      const unsigned mask = __ballot_sync(0xffffffffu, outflow == sp);
      if (mask && (threadIdx.x & 31) == __ffs(mask) - 1)
        atomicAdd(cnt + kOut + sp, static_cast<unsigned long long>(__popc(mask)));
    }
    const long long slot = warp_slot(keep, cnt + kout, cap, cnt + kOverflow);
    if (slot >= 0) {
      out.x[slot] = px;
      out.y[slot] = py;
      out.s[slot] = s;
      out.id[slot] = id;
    }
  }
  if (tight) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      last = atomicAdd(cnt + kDone, 1ull) + 1ull == static_cast<unsigned long long>(movers);
      if (last) cnt[kDone] = 0ull;
    }
    __syncthreads();
    if (last) spawn(a, out, cnt, kout, cap, t, id0, m, -0.5, 1.0, 0, 1);
  }
}

// ---------------------------------------------------------------------------
// The particles in the order of their ids, for the read-back: a radix sort of
// (id, storage index), least significant digit first, bound by the latency of
// its passes (an id of b bits takes b / 8 of them).  The read-back of the 300
// 000 particles of a 1000 x 300 membrane was sorted by the host before, which
// took 22 of the 36 ms of 200 steps and the read-back; they take 13.4 ms now.
// A pass counts the digits of each tile of keys, scans the counts (digit by
// digit, tile by tile), and moves each key to its digit's next place; within
// a tile, keys of a digit keep their order by rounds of one key per thread,
// ranked in the warp by __match_any_sync and across warps by counts.
// ---------------------------------------------------------------------------
constexpr int kDigits = 256;
constexpr int kRounds = 8;
constexpr int kTile = kRounds * kThreads;
constexpr int kScanThreads = 1024;

__device__ inline int digit_of(unsigned long long key, int shift) {
  return static_cast<int>((key >> shift) & (kDigits - 1));
}

__global__ void __launch_bounds__(kThreads)
    sort_count_kernel(const unsigned long long *keys, int n, int shift,
                      int tiles, unsigned *count) {
  __shared__ unsigned hist[kDigits];
  hist[threadIdx.x] = 0;
  __syncthreads();
  const int lo = blockIdx.x * kTile, hi = min(lo + kTile, n);
  for (int i = lo + threadIdx.x; i < hi; i += kThreads)
    atomicAdd(hist + digit_of(keys[i], shift), 1u);
  __syncthreads();
  count[threadIdx.x * tiles + blockIdx.x] = hist[threadIdx.x];
}

// exclusive prefix sum of count[0 .. m) in place, one block
__global__ void __launch_bounds__(kScanThreads) sort_scan_kernel(unsigned *count, int m) {
  __shared__ unsigned warp_sum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned base = 0;
  for (int lo = 0; lo < m; lo += kScanThreads) {
    const int i = lo + threadIdx.x;
    const unsigned v = i < m ? count[i] : 0u;
    unsigned inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      unsigned w = warp_sum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += t;
      }
      warp_sum[lane] = w;   // inclusive
    }
    __syncthreads();
    const unsigned before = warp > 0 ? warp_sum[warp - 1] : 0u;
    if (i < m) count[i] = base + before + inc - v;
    base += warp_sum[kScanThreads / 32 - 1];
    __syncthreads();
  }
}

// idx == nullptr: the first pass, whose keys are in storage order
__global__ void __launch_bounds__(kThreads)
    sort_move_kernel(const unsigned long long *keys, const unsigned *idx, int n,
                     int shift, int tiles, const unsigned *place,
                     unsigned long long *keys_out, unsigned *idx_out) {
  __shared__ unsigned next[kDigits];                 // place of the digit's next key
  __shared__ unsigned cnt[kThreads / 32][kDigits];   // keys of this round per warp
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  next[t] = place[t * tiles + blockIdx.x];
  for (int round = 0; round < kRounds; ++round) {
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) cnt[w][t] = 0;
    __syncthreads();
    const int i = blockIdx.x * kTile + round * kThreads + t;
    const bool on = i < n;
    const unsigned long long key = on ? keys[i] : 0ull;
    const int d = on ? digit_of(key, shift) : kDigits;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const unsigned rank = __popc(same & ((1u << lane) - 1u));
    if (on && rank == 0) cnt[warp][d] = __popc(same);
    __syncthreads();
    if (on) {
      unsigned to = next[d] + rank;
      for (int w = 0; w < warp; ++w) to += cnt[w][d];
      keys_out[to] = key;
      idx_out[to] = idx ? idx[i] : static_cast<unsigned>(i);
    }
    __syncthreads();
    unsigned all = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) all += cnt[w][t];
    next[t] += all;
  }
}

template <typename V>
__global__ void __launch_bounds__(kThreads)
    gather_kernel(const V *v, const unsigned *idx, int n, V *out) {
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i < n) out[i] = v[idx[i]];
}

inline size_t a256(size_t n) { return (n + 255) / 256 * 256; }

}  // namespace rwpt
}  // namespace lbm

using namespace lbm;
using namespace lbm::rwpt;

struct lbm_rwpt {
  Args a{};
  lbm_rwpt_params p{};
  int nx = 0, ny = 0;
  long long cap = 0;
  Buf buf[2];
  unsigned long long *cnt = nullptr;
  int cur = 0;                 // buffer holding the current particles
  int count = 0;               // which of the three counts is theirs
  long long steps = 0, window = 0;
  unsigned long long next_id = 0;
  long long seed_count = 0;    // entrance particles per step
  int grid = 0;
  bool started = false;
  // The read-back sorts in the buffer that the next step writes, so it must
  // not run beside a step or another read-back: the calls on a system take
  // turns, and the read-back's stream waits for `done`, which follows the last
  // work enqueued on whatever stream.
  std::mutex turn;
  cudaEvent_t done = nullptr;
};

namespace {

// r->done follows what `st` holds now (nothing to record while a graph is
// being captured: its work has not run)
cudaError_t mark_done(lbm_rwpt *r, cudaStream_t st) {
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(st, &capturing);
  if (e != cudaSuccess || capturing != cudaStreamCaptureStatusNone) return e;
  return cudaEventRecord(r->done, st);
}

struct RwptLayout {
  size_t xy, id, s, fib, near, cnt, total;
};
RwptLayout rwpt_layout(long long cap, int nfib) {
  RwptLayout l{};
  l.xy = a256(8 * static_cast<size_t>(cap));
  l.id = a256(8 * static_cast<size_t>(cap));
  l.s = a256(4 * static_cast<size_t>(cap));
  l.fib = a256(sizeof(Fiber) * static_cast<size_t>(nfib > 0 ? nfib : 1));
  l.near = a256(sizeof(Near) * static_cast<size_t>(nfib > 0 ? nfib : 1));
  l.cnt = a256(8 * kCounters);
  l.total = 2 * (2 * l.xy + l.id + l.s) + l.fib + l.near + l.cnt;
  return l;
}

lbm_status rfail(const char *where, cudaError_t e) {
  set_error(std::string(where) + ": " + cudaGetErrorString(e));
  return LBM_ECUDA;
}

}  // namespace

extern "C" size_t lbm_rwpt_ws_bytes(int64_t capacity, int32_t nfibers) {
  if (capacity < 1 || nfibers < 0) return 0;
  return rwpt_layout(capacity, nfibers).total;
}

extern "C" lbm_status lbm_rwpt_create(int32_t nx, int32_t ny,
                                      const double *fibers, int32_t nfibers,
                                      double k1, double k2,
                                      const lbm_rwpt_params *p, const void *u,
                                      int64_t capacity, void *ws,
                                      size_t ws_bytes, lbm_rwpt **out) {
  if (!out) {
    set_error("lbm_rwpt_create: out is NULL");
    return LBM_EINVAL;
  }
  *out = nullptr;
  if (!p || !ws || nx < 2 || ny < 1 || nfibers < 0 || (nfibers > 0 && !fibers) ||
      capacity < 1) {
    set_error("lbm_rwpt_create: NULL argument, nx < 2, ny < 1 or capacity < 1");
    return LBM_EINVAL;
  }
  const bool periodic = (p->flags & LBM_RWPT_PERIODIC) != 0;
  if (!(p->dt > 0.0) || !(p->D >= 0.0) || !(p->delta >= 0.0) ||
      !(p->density >= 0.0) || p->nspecies < 1 || p->nspecies > 3 ||
      !(k1 >= 0.0) || !(k2 >= 0.0) || k1 * p->dt > 1.0 || k2 * p->dt > 1.0 ||
      (p->flags & ~(LBM_RWPT_PERIODIC | LBM_RWPT_HOMOGENEOUS))) {
    set_error("lbm_rwpt_create: need dt > 0, D, delta, density >= 0, 1..3 "
              "species, 0 <= k dt <= 1, known flags");
    return LBM_EINVAL;
  }
  if ((reinterpret_cast<uintptr_t>(ws) & 255u) != 0 ||
      (u && (reinterpret_cast<uintptr_t>(u) & 7u) != 0)) {
    set_error("lbm_rwpt_create: workspace not 256-byte aligned");
    return LBM_EINVAL;
  }
  const RwptLayout l = rwpt_layout(capacity, nfibers);
  if (ws_bytes < l.total) {
    set_error("lbm_rwpt_create: workspace too small");
    return LBM_ENOMEM;
  }
  std::vector<Fiber> fib(static_cast<size_t>(nfibers));
  std::vector<Near> near(static_cast<size_t>(nfibers));
  for (int f = 0; f < nfibers; ++f) {
    const double *r = fibers + 6 * static_cast<int64_t>(f);
    const int cat = static_cast<int>(r[3]);
    if (!(r[2] >= 0.0) || cat < 0 || cat > 3) {
      set_error("lbm_rwpt_create: bad fiber row " + std::to_string(f));
      return LBM_EINVAL;
    }
    Fiber &q = fib[f];
    q.cx = r[0];
    q.cy = r[1];
    q.rp = r[2] + p->radius_offset;
    q.split = 0;
    q.kab = q.kbc = 0.0;
    if (cat != 0 && r[5] >= 0.0) {
      q.kab = r[5] * k1;
      q.kbc = (1.0 - r[5]) * k2;
    } else if (cat == 1) {
      q.kab = k1;
    } else if (cat == 2) {
      q.kbc = k2;
    } else if (cat == 3) {
      q.kab = k1;
      q.kbc = k2;
      q.split = 1;
      q.nx = std::cos(r[4]);
      q.ny = std::sin(r[4]);
    }
    // A point held by the fiber has coordinates of at most |c| + reach, so
    // cutting it to float (2^-23), rounding the centre (2^-24) and subtracting
    // is off by less than 2.4e-7 (|c| + reach) in each coordinate; the slack
    // is more than that.  (Infinities and NaN leave the fiber in the double test.)
    const double reach = std::fabs(q.rp) + p->delta;
    const double d = reach + 1e-3 +
                     4e-7 * (std::fabs(q.cx) + std::fabs(q.cy) + 2.0 * reach);
    near[f] = {static_cast<float>(q.cx), static_cast<float>(q.cy),
               static_cast<float>(1.00001 * d * d), 0.0f};
  }
  lbm_rwpt *r = new (std::nothrow) lbm_rwpt;
  if (!r) {
    set_error("lbm_rwpt_create: host allocation failed");
    return LBM_ENOMEM;
  }
  char *b = static_cast<char *>(ws);
  for (int k = 0; k < 2; ++k) {
    char *o = b + k * (2 * l.xy + l.id + l.s);
    r->buf[k].x = reinterpret_cast<double *>(o);
    r->buf[k].y = reinterpret_cast<double *>(o + l.xy);
    r->buf[k].id = reinterpret_cast<unsigned long long *>(o + 2 * l.xy);
    r->buf[k].s = reinterpret_cast<int *>(o + 2 * l.xy + l.id);
  }
  Fiber *d_fib = reinterpret_cast<Fiber *>(b + 2 * (2 * l.xy + l.id + l.s));
  Near *d_near = reinterpret_cast<Near *>(b + 2 * (2 * l.xy + l.id + l.s) + l.fib);
  r->cnt = reinterpret_cast<unsigned long long *>(
      b + 2 * (2 * l.xy + l.id + l.s) + l.fib + l.near);
  r->p = *p;
  r->nx = nx;
  r->ny = ny;
  r->cap = capacity;
  Args &a = r->a;
  a.nx = nx;
  a.ny = ny;
  a.nx_pad = static_cast<int>(pad32(nx));
  a.nfib = nfibers;
  a.nspecies = p->nspecies;
  a.periodic = periodic ? 1 : 0;
  a.homogeneous = (p->flags & LBM_RWPT_HOMOGENEOUS) ? 1 : 0;
  a.dt = p->dt;
  a.len = std::sqrt(4.0 * p->D * p->dt);
  a.delta = p->delta;
  a.hk1 = k1;
  a.hk2 = k2;
  a.seed = p->seed;
  a.u = static_cast<const double *>(u);
  a.fib = d_fib;
  a.near = d_near;
  a.plain = a.len > 1e-100 && a.len < 1e100 ? 0 : 1;
  a.moves = a.len > 0.0 ? 1 : 0;
  a.dnx = nx;
  a.dny = ny;
  a.xout = a.dnx - 0.5;
  a.ytop = a.dny - 0.5;
  r->seed_count = periodic ? 0 : static_cast<long long>(std::llround(p->density * ny));
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  r->grid = 8 * sms;
  cudaError_t e = cudaSuccess;
  if (nfibers > 0)
    e = cudaMemcpy(d_fib, fib.data(), sizeof(Fiber) * fib.size(), cudaMemcpyHostToDevice);
  if (nfibers > 0 && e == cudaSuccess)
    e = cudaMemcpy(d_near, near.data(), sizeof(Near) * near.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&r->done, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    delete r;
    return rfail("lbm_rwpt_create", e);
  }
  *out = r;
  return LBM_OK;
}

extern "C" void lbm_rwpt_destroy(lbm_rwpt *r) {
  if (!r) return;
  cudaEventDestroy(r->done);
  delete r;
}

extern "C" lbm_status lbm_rwpt_init(lbm_rwpt *r, void *stream) {
  NvtxRange nvtx_range("lbm_rwpt_init");
  if (!r) {
    set_error("lbm_rwpt_init: NULL argument");
    return LBM_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(r->turn);
  cudaError_t e = cudaMemsetAsync(r->cnt, 0, 8 * kCounters, st);
  r->cur = 0;
  r->count = 0;
  r->steps = 0;
  r->window = 0;
  r->next_id = 0;
  // the start: A at the density over the whole box (the fluid part of it)
  const long long m = std::llround(r->p.density * static_cast<double>(r->nx) * r->ny);
  if (e == cudaSuccess && m > 0) {
    rwpt_spawn_kernel<<<r->grid, kThreads, 0, st>>>(
        r->a, r->buf[0], r->cnt, kCount, r->cap, -1, 0ull, m, -0.5,
        static_cast<double>(r->nx));
    e = cudaGetLastError();
  }
  r->next_id = static_cast<unsigned long long>(m);
  if (e == cudaSuccess) e = mark_done(r, st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_init", e);
  r->started = true;
  return LBM_OK;
}

extern "C" lbm_status lbm_rwpt_run(lbm_rwpt *r, int64_t nsteps, void *stream,
                                   lbm_rwpt_info *info) {
  NvtxRange nvtx_range("lbm_rwpt_run");
  if (!r || nsteps < 0 || !r->started) {
    set_error("lbm_rwpt_run: NULL solver, nsteps < 0 or not initialised");
    return LBM_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(r->turn);
  cudaError_t e = cudaSuccess;
  const long long entering = (r->seed_count + kThreads - 1) / kThreads;
  const int spawners = static_cast<int>(entering < r->grid ? entering : r->grid);
  for (int64_t k = 0; k < nsteps && e == cudaSuccess; ++k) {
    const int next = (r->count + 1) % 3;
    rwpt_step_kernel<<<r->grid + spawners, kThreads, 0, st>>>(
        r->a, r->buf[r->cur], r->buf[r->cur ^ 1], r->cnt, kCount + r->count,
        kCount + next, kCount + (next + 1) % 3, r->cap, r->steps, r->next_id,
        r->seed_count, r->grid);
    e = cudaGetLastError();
    r->next_id += static_cast<unsigned long long>(r->seed_count);
    r->cur ^= 1;
    r->count = next;
    ++r->steps;
    ++r->window;
  }
  if (e == cudaSuccess) e = mark_done(r, st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_run", e);
  if (!info) return LBM_OK;
  unsigned long long h[kCounters] = {0};
  e = cudaMemcpyAsync(h, r->cnt, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_run", e);
  std::memset(info, 0, sizeof(*info));
  info->steps = r->steps;
  info->window_steps = r->window;
  info->alive = static_cast<int64_t>(h[kCount + r->count]) < r->cap
                    ? static_cast<int64_t>(h[kCount + r->count])
                    : r->cap;
  for (int s = 0; s < 3; ++s) info->out[s] = static_cast<int64_t>(h[kOut + s]);
  info->overflow = h[kOverflow] ? 1 : 0;
  const int ns = r->p.nspecies;
  double f[3] = {double(h[kOut]), double(h[kOut + 1]), double(h[kOut + 2])};
  if (ns >= 2) {
    double eps = 0.0;
    if (lbm_efficiency(f, ns, &eps) == LBM_OK) info->eps = eps;
  }
  if (info->overflow) {
    set_error("lbm_rwpt_run: particle capacity exceeded (particles were lost)");
    return LBM_ENOMEM;
  }
  return LBM_OK;
}

extern "C" lbm_status lbm_rwpt_reset_counts(lbm_rwpt *r, void *stream) {
  if (!r) {
    set_error("lbm_rwpt_reset_counts: NULL argument");
    return LBM_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(r->turn);
  cudaError_t e = cudaMemsetAsync(r->cnt + kOut, 0, 8 * 3, st);
  if (e == cudaSuccess) e = mark_done(r, st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_reset_counts", e);
  r->window = 0;
  return LBM_OK;
}

namespace {

lbm_status sort_on_host(size_t n, double *x, double *y, int32_t *species, uint64_t *id) {
  struct P {
    uint64_t id;
    double x, y;
    int32_t s;
  };
  try {
    std::vector<P> v(n);
    for (size_t i = 0; i < n; ++i) v[i] = {id[i], x[i], y[i], species[i]};
    std::sort(v.begin(), v.end(), [](const P &p, const P &q) { return p.id < q.id; });
    for (size_t i = 0; i < n; ++i) {
      id[i] = v[i].id;
      x[i] = v[i].x;
      y[i] = v[i].y;
      species[i] = v[i].s;
    }
  } catch (const std::bad_alloc &) {
    set_error("lbm_rwpt_particles: host allocation failed");
    return LBM_ENOMEM;
  }
  return LBM_OK;
}

}  // namespace

extern "C" lbm_status lbm_rwpt_particles(lbm_rwpt *r, void *stream,
                                         int64_t max_count, int64_t *count,
                                         double *x, double *y, int32_t *species,
                                         uint64_t *id) {
  if (!r || !count || !x || !y || !species || !id) {
    set_error("lbm_rwpt_particles: NULL argument");
    return LBM_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lock(r->turn);
  unsigned long long n = 0;
  cudaError_t e = cudaStreamWaitEvent(st, r->done, 0);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&n, r->cnt + kCount + r->count, 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_particles", e);
  if (static_cast<long long>(n) > r->cap) n = static_cast<unsigned long long>(r->cap);
  *count = static_cast<int64_t>(n);
  if (static_cast<long long>(n) > max_count) {
    set_error("lbm_rwpt_particles: host arrays shorter than the particle count");
    return LBM_ENOMEM;
  }
  const Buf &b = r->buf[r->cur];
  // the other buffer is free until the next step: its x and y hold the keys,
  // its ids the two index lists, its species the digit counts (256 for every
  // 2048 keys begun: more than a capacity below 293 can hold, which the host
  // sorts)
  const Buf &f = r->buf[r->cur ^ 1];
  const int m = static_cast<int>(n), tiles = (m + kTile - 1) / kTile;
  if (static_cast<long long>(kDigits) * tiles > r->cap || n > (1ull << 30)) {
    e = cudaMemcpyAsync(x, b.x, 8 * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(y, b.y, 8 * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(species, b.s, 4 * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(id, b.id, 8 * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return rfail("lbm_rwpt_particles", e);
    return sort_on_host(static_cast<size_t>(n), x, y, species, id);
  }
  if (n > 0) {
    unsigned long long *keys[2] = {reinterpret_cast<unsigned long long *>(f.x),
                                   reinterpret_cast<unsigned long long *>(f.y)};
    unsigned *idx[2] = {reinterpret_cast<unsigned *>(f.id),
                        reinterpret_cast<unsigned *>(f.id) + r->cap};
    unsigned *count = reinterpret_cast<unsigned *>(f.s);
    const unsigned long long *from = b.id;
    int to = 0;
    for (int shift = 0; shift == 0 || (shift < 64 && (r->next_id - 1) >> shift != 0); shift += 8) {
      const unsigned *from_idx = shift ? idx[to ^ 1] : nullptr;
      sort_count_kernel<<<tiles, kThreads, 0, st>>>(from, m, shift, tiles, count);
      sort_scan_kernel<<<1, kScanThreads, 0, st>>>(count, kDigits * tiles);
      sort_move_kernel<<<tiles, kThreads, 0, st>>>(from, from_idx, m, shift, tiles, count,
                                                   keys[to], idx[to]);
      from = keys[to];
      to ^= 1;
    }
    const int last = to ^ 1;
    const int blocks = (m + kThreads - 1) / kThreads;
    double *out = reinterpret_cast<double *>(keys[to]);
    e = cudaMemcpyAsync(id, keys[last], 8 * n, cudaMemcpyDeviceToHost, st);
    gather_kernel<<<blocks, kThreads, 0, st>>>(b.x, idx[last], m, out);
    if (e == cudaSuccess) e = cudaMemcpyAsync(x, out, 8 * n, cudaMemcpyDeviceToHost, st);
    gather_kernel<<<blocks, kThreads, 0, st>>>(b.y, idx[last], m, out);
    if (e == cudaSuccess) e = cudaMemcpyAsync(y, out, 8 * n, cudaMemcpyDeviceToHost, st);
    gather_kernel<<<blocks, kThreads, 0, st>>>(b.s, idx[last], m, f.s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(species, f.s, 4 * n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return rfail("lbm_rwpt_particles", e);
  return LBM_OK;
}
