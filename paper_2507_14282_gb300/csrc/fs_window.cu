// fs_window.cu -- the differentiable window of the 1D faux-shock box: a
// forward pass of `steps` hybrid steps that keeps checkpoints, and the
// reverse (adjoint) sweep that gives the gradient of a loss at the window's
// end with respect to theta = (a_1..a_M, u_cr, u2): the amplitudes of seeded
// transverse-B modes, the cosmic-ray drift speed and the faux-shock kick.
//
// The step is the engine's (Sec. 2): CIC gather, Boris push, move, open far
// wall, faux-shock return (Eq. 1) at x = 0, thermal inflow at x = L and the
// cosmic-ray source at x = 0, CIC deposit, RK4 Ohm's law + Faraday with the
// moments frozen. The window keeps its particles in fixed slots (birth
// order; removed particles keep a dead slot), so that each particle's tape
// and adjoint stay in place across steps. Branches (crossings, returns,
// escapes, the density floor) and random draws are frozen: the backward
// differentiates the discrete map along the forward's branches. Every
// segment of `ckpt` steps is recomputed from its checkpoint during the
// backward; the deposit sums are int64 fixed point, so a recomputed segment
// reproduces the forward exactly in either precision.
#include <algorithm>
#include <vector>

#include "fs_engine.cuh"

namespace fsx {
namespace win {

constexpr double kUnfix = 1.0 / 1099511627776.0;
enum : uint8_t { kEvNone = 0, kEvReturned = 1, kEvRemoved = 2 };

template <typename T>
struct Slots {  // particle slots: cell (-1: removed), offset, velocity, id
  int* ci;
  T* f;
  T* v;  // [3][cap]
  uint32_t* id;
};

// The state at the start of a step: slots (no ids), B [3][nx], the moments
// [nxn], [3][nxn], [nxn] and E, Bbar [3][nxn]. A plain forward has one (its B
// in two buffers); a recomputed segment has one per step (the tape).
template <typename T>
struct State {
  Slots<T> s;
  T *B, *n, *u, *nraw, *E, *Bb;
};

template <typename T>
struct Win {
  int cap;  // particle slots
  Slots<T> s;
  T *B[2], *E, *Bb, *n, *u, *nraw;
  unsigned long long* q[2];    // fixed-point deposit sums [4][nxn] (one in use, one cleared)
  unsigned long long* ctr;     // incident, returned, transmitted, escaped
  // adjoint
  T *lf, *lv;                  // particle adjoints: offset, velocity [3][cap]
  double *lB, *lBx;            // of B [3][nx] (and the buffer the next one goes to)
  double *lE[2], *lBb[2];      // of E, Bbar [3][nxn] (one in use, one cleared)
  T *lNr, *lJ;                 // of the deposit sums (raw density, current), run precision
  double* grad;                // d loss / d theta [M + 2]
};

// ------------------------------------------------ sums over a block's cells
// A block's items (a particle per thread, key = its cell, -1: none) in key
// order, for sums per cell: the slots of a block sit in a few neighbouring
// cells (birth order), so each cell's items are then a run that one warp adds
// up in registers and hands to memory once per cell and quantity, instead of
// per particle, per lane group or by long shuffle reductions.
constexpr int kSortKeys = 64;
constexpr int kSortPiece = 32;  // items of a cell one warp takes at a time
struct CellSort {
  int lo[kBlock / 32], hi[kBlock / 32];
  int cnt[kSortKeys];
  int first[kSortKeys];
  // the pieces: cell, first and end item; their number
  short cell[kSortKeys + kBlock / kSortPiece], from[kSortKeys + kBlock / kSortPiece],
      to[kSortKeys + kBlock / kSortPiece];
  int pieces;
};
// Returns the thread's position; base: the lowest cell; range: the number of
// cells spanned (0: no item; above kSortKeys: not sorted, take each item on
// its own). Block barriers inside: every thread calls it.
__device__ __forceinline__ int cell_sort(CellSort& cs, int key, int& base, int& range) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mn = __reduce_min_sync(0xffffffffu, key < 0 ? 0x7fffffff : key);
  const int mx = __reduce_max_sync(0xffffffffu, key);
  if (lane == 0) {
    cs.lo[warp] = mn;
    cs.hi[warp] = mx;
  }
  if (threadIdx.x < kSortKeys) cs.cnt[threadIdx.x] = 0;
  __syncthreads();
  int a = cs.lo[0], b = cs.hi[0];
#pragma unroll
  for (int w = 1; w < kBlock / 32; ++w) {
    a = min(a, cs.lo[w]);
    b = max(b, cs.hi[w]);
  }
  base = a;
  range = b < 0 ? 0 : b - a + 1;
  if (range == 0 || range > kSortKeys) return 0;  // (uniform over the block)
  const int k = key - a;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int leader = __ffs(peers) - 1;
  int at = 0;
  if (lane == leader && key >= 0) at = atomicAdd(&cs.cnt[k], __popc(peers));
  at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
  __syncthreads();
  if (warp == 0) {
    constexpr int PS = kSortPiece;
    const int c[2] = {cs.cnt[2 * lane], cs.cnt[2 * lane + 1]};
    const int n[2] = {(c[0] + PS - 1) / PS, (c[1] + PS - 1) / PS};
    // one scan for both: items in the low half, pieces in the high half
    int inc = (c[0] + c[1]) | ((n[0] + n[1]) << 16);
    const int own = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) cs.pieces = inc >> 16;
    int at0 = (inc - own) & 0xFFFF, p = (inc - own) >> 16;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      cs.first[2 * lane + r] = at0;
      for (int b0 = 0; b0 < c[r]; b0 += PS, ++p) {
        cs.cell[p] = (short)(2 * lane + r);
        cs.from[p] = (short)(at0 + b0);
        cs.to[p] = (short)(at0 + min(b0 + PS, c[r]));
      }
      at0 += c[r];
    }
  }
  __syncthreads();
  return key >= 0 ? cs.first[k] + at : 0;
}

// ---------------------------------------------------------------- forward
// Gather, Boris push, move, far wall and faux-shock crossing of slot p of
// state a into the slots out; ci, f, v: the result (ci < 0: no particle).
template <typename T>
__device__ __forceinline__ void push_slot(int p, const Win<T>& w, const State<T>& a,
                                          const Slots<T>& out, uint8_t* ev, uint32_t id,
                                          const Geo& g, const Phys& ph, const PushConst<T>& pc,
                                          long long step, int& ci, T& f, T (&v)[3]) {
  const int nxn = g.nxn;
  ci = a.s.ci[p];
  if (ci < 0) {
    if (ev) ev[p] = kEvRemoved;
    if (out.ci != a.s.ci) out.ci[p] = -1;
    return;
  }
  f = a.s.f[p];
  T vx = a.s.v[p], vy = a.s.v[w.cap + p], vz = a.s.v[2 * w.cap + p];
  uint8_t e = kEvNone;
  const T g0 = (T)1 - f;
  T Ep[3], Bp[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Ep[c] = fmaT(f, a.E[c * nxn + ci + 1], g0 * a.E[c * nxn + ci]);
    Bp[c] = fmaT(f, a.Bb[c * nxn + ci + 1], g0 * a.Bb[c * nxn + ci]);
  }
  boris<T>(vx, vy, vz, Ep, Bp, pc.hdt);
  const T fr = fmaT(vx, pc.dtdx, f);
  const T k = Num<T>::fl(fr);
  int inew = ci + (int)k;
  T fn = fr - k;
  if (fn >= (T)1) fn = Num<T>::offmax;
  if (inew >= g.nx) {
    atomicAdd(&w.ctr[3], 1ull);
    e = kEvRemoved;
  } else if (inew < 0) {
    atomicAdd(&w.ctr[0], 1ull);
    const int mode = (id & kIdCR) ? FS_SHOCK : ph.fs_mode_thermal;
    double dvx = vx, dvy = vy, dvz = vz;
    if (mode == FS_SHOCK &&
        fs_return(dvx, dvy, dvz, ph.u2, ph.fs_frame, ph.seed, id & kIdMask, step)) {
      atomicAdd(&w.ctr[1], 1ull);
      const double Xo = __dadd_rn((double)ci, (double)f);
      const double Xn = __dadd_rn((double)ci, (double)fr);
      const double gfr = __ddiv_rn(Xn, __dsub_rn(Xn, Xo));
      double ff = __dmul_rn(gfr, __dmul_rn(dvx, ph.dtdx));
      if (ff < 0.0) ff = 0.0;
      if (ff >= 1.0) ff = (double)Num<double>::offmax;
      T ft = (T)ff;
      if (ft >= (T)1) ft = Num<T>::offmax;
      fn = ft;
      inew = 0;
      vx = (T)dvx;
      vy = (T)dvy;
      vz = (T)dvz;
      e = kEvReturned;
    } else {
      atomicAdd(&w.ctr[2], 1ull);
      e = kEvRemoved;
    }
  }
  if (ev) ev[p] = e;
  ci = e == kEvRemoved ? -1 : inew;
  out.ci[p] = ci;
  if (ci < 0) return;
  f = fn;
  v[0] = vx;
  v[1] = vy;
  v[2] = vz;
  out.f[p] = fn;
  out.v[p] = vx;
  out.v[w.cap + p] = vy;
  out.v[2 * w.cap + p] = vz;
}

// The velocity and placement of a new cosmic ray (speed p_iso, direction
// flux-weighted in the frame drifting at u_cr), drawn as the engine draws
// it. Returns X in cells; U (optional) = {sqrt(U1), cos, sin, U_place}.
__device__ __forceinline__ double cr_draw(const Phys& ph, uint32_t pid, long long step,
                                          double* v, double* U) {
  const Philox4 rc = draw4(ph.seed, pid, step, kPurposeInjCR);
  const double s1 = __dsqrt_rn(u01(rc.x[0]));
  const double a = __ddiv_rn(ph.u_cr, ph.p_iso_v);
  const double mu = __dadd_rn(a, __dmul_rn(__dsub_rn(1.0, a), s1));
  const double sn = __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(mu, mu)));
  double c, s;
  fs_sincos2pi(u01(rc.x[1]), &c, &s);
  const double ws = __dmul_rn(ph.p_iso_v, sn);
  v[0] = __dsub_rn(__dmul_rn(ph.p_iso_v, mu), ph.u_cr);
  v[1] = __dmul_rn(ws, c);
  v[2] = __dmul_rn(ws, s);
  if (U) {
    U[0] = s1;
    U[1] = c;
    U[2] = s;
    U[3] = u01(rc.x[2]);
  }
  return __dmul_rn(__dmul_rn(u01(rc.x[2]), v[0]), ph.dtdx);
}

// Every ion the window injects, drawn once at its start into its slot (slots
// n_init .. np_at[steps], birth order: per step its thermal ions at x = L,
// then its cosmic rays at x = 0; ids are slot numbers): one thread per slot,
// np_at[n] = slots at the start of step n. A draw depends on the slot, the step
// and theta alone, and a step takes part only in slots below its np_at, so
// the long FP64 draw chain is off the steps (14 us of push and injection per
// step of a 262 K-ion window before, the chain most of it).
template <typename T>
__global__ void k_win_draw(Win<T> w, Geo g, Phys ph, const int* __restrict__ np_at, int steps) {
  const int p = np_at[0] + blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np_at[steps]) return;
  int lo = 0, hi = steps;  // np_at[lo] <= p < np_at[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (np_at[mid] <= p) lo = mid;
    else hi = mid;
  }
  const long long step = lo;
  const int kinds = (ph.inject_thermal ? 1 : 0) + (ph.cr_enable ? 1 : 0);
  const int k = p - np_at[lo], n_new = (np_at[lo + 1] - np_at[lo]) / kinds;
  const int nth = ph.inject_thermal ? n_new : 0;
  const uint32_t pid = (uint32_t)p;
  const int nx = g.nx;
  double vx, vy, vz, X;
  uint32_t id = pid;
  if (k < nth) {
    const Philox4 ra = draw4(ph.seed, pid, step, kPurposeInjA);
    const Philox4 rb = draw4(ph.seed, pid, step, kPurposeInjB);
    double g0, g1, g2, g3;
    gauss2(u01(ra.x[0]), u01(ra.x[1]), &g0, &g1);
    gauss2(u01(ra.x[2]), u01(ra.x[3]), &g2, &g3);
    vx = __dsub_rn(__dmul_rn(ph.vth, g0), ph.mach_a);
    vy = __dmul_rn(ph.vth, g1);
    vz = __dmul_rn(ph.vth, g2);
    X = __dsub_rn((double)nx, __dmul_rn(__dmul_rn(u01(rb.x[0]), fabs(vx)), ph.dtdx));
  } else {
    double v[3];
    X = cr_draw(ph, pid, step, v, nullptr);
    vx = v[0];
    vy = v[1];
    vz = v[2];
    id |= kIdCR;
  }
  const double ix = floor(X);
  int i = (int)ix;
  double fx = __dsub_rn(X, ix);
  if (i >= nx) { i = nx - 1; fx = Num<double>::offmax; }
  if (i < 0) { i = 0; fx = 0.0; }
  if (fx >= 1.0) fx = Num<double>::offmax;
  T ft = (T)fx;
  if (ft >= (T)1) ft = Num<T>::offmax;
  w.s.ci[p] = i;
  w.s.f[p] = ft;
  w.s.v[p] = (T)vx;
  w.s.v[w.cap + p] = (T)vy;
  w.s.v[2 * w.cap + p] = (T)vz;
  w.s.id[p] = id;
}

// c * 2^40 rounded to the nearest integer, ties to even (the value of
// __double2ll_rn(c * 2^40) for |c| < 2^23), on the bit pattern with integer
// operations: the significand shifted right by 1035 - e with the rounding
// of the bits shifted out, kept off the FP64 pipe.
__device__ __forceinline__ unsigned long long fix(double c) {
  const long long b = __double_as_longlong(c);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long mant = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
  const int sh = 1035 - e;
  long long r;
  if (e == 0 || sh > 53) {
    r = 0;  // zero, subnormal, or |c| 2^40 < 1/2
  } else if (sh <= 0) {
    r = mant << (-sh);
  } else {
    const long long q = mant >> sh;
    const long long rem = mant - (q << sh);
    const long long half = 1LL << (sh - 1);
    r = q + ((rem > half || (rem == half && (q & 1))) ? 1 : 0);
  }
  return (unsigned long long)(b < 0 ? -r : r);
}

// c * 2^40 rounded to the nearest integer for an FP32 value c (|c| < 2^23):
// the scaling is exact; below 2^30 the int32 conversion rounds to nearest
// (ties to even), at or above it the value is an integer already (its ulp is
// at least 2^7) and its significand is shifted into place. (The conversion
// instruction to 64 bits measured slower: 15.9 against 14.8 us per launch.)
__device__ __forceinline__ long long fix32(float c) {
  const float y = c * 0x1p40f;
  if (fabsf(y) < 0x1p30f) return (long long)__float2int_rn(y);
  const int b = __float_as_int(y);
  const int e = (b >> 23) & 0xFF;
  const long long r = (long long)((b & 0x7FFFFF) | 0x800000) << (e - 150);
  return b < 0 ? -r : r;
}

__device__ __forceinline__ long long fixT(float c) { return fix32(c); }
__device__ __forceinline__ long long fixT(double c) { return (long long)fix(c); }

// One step's particles: push slots 0 .. np - 1 of state a into the slots out,
// take over the slots np .. np1 - 1 born in the step from `drawn`, and deposit
// all of them into the fixed-point sums q (CIC; integer sums, so the result
// does not depend on the grouping; contributions in the run's precision, FP32
// runs with no FP64 instruction). The block's particles are sorted by cell
// (cell_sort); a warp adds a cell's eight quantities (n, J at its two nodes)
// with four lanes each, 32 particles at a time. Push and deposit in one launch: the deposit
// needs no second read of the slots, and the sums it replaces (lane groups
// by match and 24 reductions, then atomics per warp and cell) were half of
// the window. 262 K ions: FP32 14 + 30 -> 13.2 us, FP64 (39 K) 16 + 17 -> 17.0 us.
template <typename T>
__global__ void __launch_bounds__(kBlock)
    k_win_push_deposit(Win<T> w, State<T> a, Slots<T> out, Slots<T> drawn, uint8_t* ev,
                       unsigned long long* __restrict__ q, Geo g, Phys ph, PushConst<T> pc,
                       long long step, int np, int np1) {
  __shared__ CellSort cs;
  __shared__ T rec[5][kBlock];  // corner weights (left, right), velocity
  const int nxn = g.nxn;
  const int p = blockIdx.x * kBlock + threadIdx.x;
  int ci = -1;
  T f = (T)0, v[3] = {(T)0, (T)0, (T)0}, wp = (T)0;
  if (p < np1) {
    const uint32_t id = w.s.id[p];
    if constexpr (sizeof(T) == 4) wp = (id & kIdCR) ? pc.wcr : pc.wth;
    else wp = (id & kIdCR) ? ph.w_cr : ph.w_th;
    if (p < np) {
      push_slot<T>(p, w, a, out, ev, id, g, ph, pc, step, ci, f, v);
    } else {
      ci = drawn.ci[p];
      f = drawn.f[p];
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = drawn.v[c * w.cap + p];
      if (out.ci != drawn.ci) {
        out.ci[p] = ci;
        out.f[p] = f;
#pragma unroll
        for (int c = 0; c < 3; ++c) out.v[c * w.cap + p] = v[c];
      }
    }
  }
  const T c0 = wp * ((T)1 - f), c1 = wp * f;
  int base, range;
  const int pos = cell_sort(cs, ci, base, range);
  if (range > kSortKeys) {  // cells far apart
    if (ci < 0) return;
    atomicAdd(&q[ci], (unsigned long long)fixT(c0));
    atomicAdd(&q[ci + 1], (unsigned long long)fixT(c1));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      atomicAdd(&q[(c + 1) * nxn + ci], (unsigned long long)fixT(c0 * v[c]));
      atomicAdd(&q[(c + 1) * nxn + ci + 1], (unsigned long long)fixT(c1 * v[c]));
    }
    return;
  }
  if (ci >= 0) {
    rec[0][pos] = c0;
    rec[1][pos] = c1;
#pragma unroll
    for (int c = 0; c < 3; ++c) rec[2 + c][pos] = v[c];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, side = lane & 1, comp = (lane >> 1) & 3;
  const int pieces = range ? cs.pieces : 0;
  for (int k = threadIdx.x >> 5; k < pieces; k += kBlock / 32) {
    const int b1 = cs.to[k];
    long long s = 0;
#pragma unroll 4
    for (int i = cs.from[k] + (lane >> 3); i < b1; i += 4) {
      const T c = rec[side][i];
      s += fixT(comp ? c * rec[1 + comp][i] : c);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    if (lane < 8) atomicAdd(&q[comp * nxn + base + cs.cell[k] + side], (unsigned long long)s);
  }
}

// Quantity c (0: density, 1 .. 3: current) at node i from the fixed-point sums:
// wall nodes x2.
template <typename T>
__device__ __forceinline__ T moment_sum(int i, int c, const unsigned long long* q, const Geo& g) {
  const double sc = (i == 0 || i == g.nx) ? 2.0 * kUnfix : kUnfix;
  return (T)((double)(long long)q[c * g.nxn + i] * sc);
}

// The moments at the start of the window.
template <typename T>
__global__ void k_win_moments(Win<T> w, const unsigned long long* q, Geo g, Phys ph) {
  const int nxn = g.nxn;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nxn) return;
  const T nr = moment_sum<T>(i, 0, q, g);
  const T nf = (T)ph.n_floor, n = nr < nf ? nf : nr;
  w.nraw[i] = nr;
  w.n[i] = n;
#pragma unroll
  for (int c = 0; c < 3; ++c) w.u[c * nxn + i] = moment_sum<T>(i, c + 1, q, g) / n;
}

// B = B0 + sum_m a_m (cos, sin)(2 pi m x / L + phi_m) at the centres. A block
// takes 16 cells: 16 threads a cell form the terms, one adds them in order (a
// thread per cell: 46 us for 16 modes, the FP64 chain of its 16 sincos).
constexpr int kSeedCells = 16;
template <typename T>
__global__ void __launch_bounds__(kBlock)
    k_win_seed_B(T* B, Geo g, Phys ph, double dx, const double* amps, const double* phases, int M) {
  __shared__ double term[2][kSeedCells][17];
  const int cell = threadIdx.x / 16, m0 = threadIdx.x & 15;
  const int i = blockIdx.x * kSeedCells + cell;
  const double x = ((double)i + 0.5) * dx;
  const double L = (double)g.nx * dx;
  double by = ph.b0y, bz = ph.b0z;
  for (int mb = 0; mb < M; mb += 16) {
    const int m = mb + m0;
    if (m < M) {
      const double arg = 2.0 * 3.14159265358979323846 * (double)(m + 1) * x / L + phases[m];
      double s, c;
      sincos(arg, &s, &c);
      term[0][cell][m0] = c;
      term[1][cell][m0] = s;
    }
    __syncthreads();
    if (m0 == 0)
      for (int k = 0; k < min(16, M - mb); ++k) {
        by += amps[mb + k] * term[0][cell][k];
        bz += amps[mb + k] * term[1][cell][k];
      }
    __syncthreads();
  }
  if (m0 || i >= g.nx) return;
  B[i] = (T)ph.b0x;
  B[g.nx + i] = (T)by;
  B[2 * g.nx + i] = (T)bz;
}

// loss = sum_{i >= i0} |B_perp - B0_perp|^2 dx (into *out), and its
// gradient with respect to B times `scale` (into lB) when lB is given. One
// CTA: the sum is taken in a fixed order, so the loss is reproducible.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_win_loss(const T* B, Geo g, Phys ph, int i0, double dx,
                                                     double* out, double* lB, double scale) {
  __shared__ double red[kBlock / 32];
  double s = 0.0;
  for (int i = threadIdx.x; i < g.nx; i += blockDim.x) {
    double dy = 0.0, dz = 0.0;
    if (i >= i0) {
      dy = (double)B[g.nx + i] - ph.b0y;
      dz = (double)B[2 * g.nx + i] - ph.b0z;
      s += (dy * dy + dz * dz) * dx;
    }
    if (lB) {
      lB[i] = 0.0;
      lB[g.nx + i] = scale * (2.0 * dy * dx);
      lB[2 * g.nx + i] = scale * (2.0 * dz * dx);
    }
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0 && out) {
    double tot = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) tot += red[k];
    *out = tot;
  }
}

// ---------------------------------------------------------------- adjoint
// Adjoint of Ohm's law at one node of the 1D grid with n, u frozen. In: the
// centre fields Bm, Bp of the node's two cells (clamped at the walls), 1/n
// at the node (in) and the pressure term pgx = -T_e (n(i+1) - n(i-1))/(2 dx)
// (neighbours mirrored at the walls; both fixed while n is), u at the node
// and the adjoint (lex, ley, lez) of E there. Out: the
// adjoints of Bbar_y, Bbar_z, dB_y/dx, dB_z/dx at the node (P), that of n at
// the node (ln), the weight lp of n at the right neighbour (its negative at
// the left one: the pressure term's two-point difference) and the adjoint
// of u (lu).
//   E = ((curl B - jcr x) x Bbar - T_e grad n)/n - u x Bbar + eta curl B,
//   curl B = (0, -dB_z/dx, dB_y/dx)
struct OhmAdj {
  double P[4], ln, lp, lu[3];
};
__device__ __forceinline__ OhmAdj ohm_adj_point(const double Bm[3], const double Bp[3],
                                                double in, double pgx, const double u[3],
                                                double lex, double ley, double lez,
                                                const Phys& ph) {
  const double idx = ph.idx, te = ph.te, jcr = ph.jcr, eta = ph.eta;
  const double bbx = 0.5 * (Bm[0] + Bp[0]);
  const double bby = 0.5 * (Bm[1] + Bp[1]);
  const double bbz = 0.5 * (Bm[2] + Bp[2]);
  const double dby = (Bp[1] - Bm[1]) * idx;
  const double dbz = (Bp[2] - Bm[2]) * idx;
  const double ux = u[0], uy = u[1], uz = u[2];
  OhmAdj r;
  r.P[0] = lex * (-dby * in + uz) + lez * (-jcr * in - ux);
  r.P[1] = lex * (-dbz * in - uy) + ley * (jcr * in + ux);
  r.P[2] = lex * (-bby * in) + ley * (bbx * in) + lez * eta;
  r.P[3] = lex * (-bbz * in) + lez * (bbx * in) - ley * eta;
  const double cax = -dbz * bbz - dby * bby;
  const double cay = dby * bbx + jcr * bbz;
  const double caz = -jcr * bby + dbz * bbx;
  r.ln = -(lex * (pgx + cax) + ley * cay + lez * caz) * in * in;
  r.lp = -lex * in * te * ph.hdx;
  r.lu[0] = ley * bbz - lez * bby;
  r.lu[1] = -lex * bbz + lez * bbx;
  r.lu[2] = lex * bby - ley * bbx;
  return r;
}

// Centre part: the adjoint (ly, lz) of B_y, B_z at cell c from the node
// partials of its two nodes c (Pc) and c + 1 (Pc1) (Bbar = (Bm + Bp)/2,
// dB = (Bp - Bm)/dx); the wall nodes 0 and nx read cell 0 or nx - 1 twice.
__device__ __forceinline__ void curl_adj_point(const double Pc[4], const double Pc1[4],
                                               bool left_wall, bool right_wall, double idx,
                                               double& ly, double& lz) {
  ly = 0.0;
  lz = 0.0;
  ly += 0.5 * Pc[0] + Pc[2] * idx;  // node c sees cell c as its p side
  lz += 0.5 * Pc[1] + Pc[3] * idx;
  ly += 0.5 * Pc1[0] - Pc1[2] * idx;  // node c + 1 sees it as its m side
  lz += 0.5 * Pc1[1] - Pc1[3] * idx;
  if (left_wall) {  // node 0: m side clamped to cell 0
    ly += 0.5 * Pc[0] - Pc[2] * idx;
    lz += 0.5 * Pc[1] - Pc[3] * idx;
  }
  if (right_wall) {  // node nx: p side clamped to cell nx - 1
    ly += 0.5 * Pc1[0] + Pc1[2] * idx;
    lz += 0.5 * Pc1[1] + Pc1[3] * idx;
  }
}

// Adjoint of the moments at node i: from the adjoints ln, lu of n (floored)
// and u = J / n to those of the raw sums (wall nodes x2, no gradient through
// a floored density).
template <typename T>
__device__ __forceinline__ void moments_adj_node(int i, double inv_n, const T* uN,
                                                 const T* nraw, double ln, const double lu[3],
                                                 T* lNr, T* lJ, const Geo& g,
                                                 const Phys& ph) {
  const int nxn = g.nxn;
  const double sc = (i == 0 || i == g.nx) ? 2.0 : 1.0;
  for (int c = 0; c < 3; ++c) {
    const double l = lu[c] * inv_n;
    lJ[c * nxn + i] = (T)(l * sc);
    ln -= l * (double)uN[c * nxn + i];
  }
  lNr[i] = (T)(((double)nraw[i] < ph.n_floor) ? 0.0 : ln * sc);
}

// ------------------------------------------------ blocked field kernels
// A step's field work is tens of dependent phases over a small 1D grid. Each
// CTA owns kTbCells cells (and their left nodes; the last CTA also node nx)
// and runs all phases of the step in shared memory over its cells plus a
// halo, recomputing the halo: the stencils reach one cell per phase, so
// wrong values enter from a tile's inner edges (read there with clamped
// indices) at one cell per phase and never reach the owned cells while the
// halo is at least the number of phases. At the domain walls the tile edge is
// the wall and the clamped and mirrored indices are the walls' own. No
// synchronisation between CTAs, and the FP64 work spreads over the SMs.
constexpr int kTbCells = 16;
// halos: the forward's 4 n_sub stages and final Ohm; the adjoint's stage
// recompute, its 4 n_sub reverse stages and the moment adjoints
__host__ __device__ constexpr int halo_fields(int n_sub) { return 4 * n_sub + 2; }
__host__ __device__ constexpr int halo_rk4_adj(int n_sub) { return 8 * n_sub + 3; }

struct Tile {
  int c0, c1;  // owned cells [c0, c1)
  int lo, L;   // local cells lo .. lo + L - 1, local nodes lo .. lo + L
  int nx;
  __device__ __forceinline__ Tile(int b, int nx_, int halo) : nx(nx_) {
    c0 = b * kTbCells;
    c1 = min(nx, c0 + kTbCells);
    lo = max(0, c0 - halo);
    L = min(nx, c1 + halo) - lo;
  }
  // global node (mirrored at the walls) -> local node (clamped to the tile)
  __device__ __forceinline__ int node(int i) const {
    i = (i < 0) ? -i : ((i > nx) ? 2 * nx - i : i);
    return min(max(i - lo, 0), L);
  }
  __device__ __forceinline__ bool owns_cell(int c) const { return c >= c0 && c < c1; }
  __device__ __forceinline__ bool owns_node(int i) const {
    return (i >= c0 && i < c1) || (i == nx && c1 == nx);
  }
};

constexpr size_t kMaxSmem = 227 * 1024;  // shared memory a CTA may opt in to

constexpr int fields_threads(int n_sub) {
  return tile1_threads(kTbCells + 2 * halo_fields(n_sub));
}
constexpr int rk4_adj_threads(int n_sub) {
  return tile1_threads(kTbCells + 2 * halo_rk4_adj(n_sub));
}
constexpr int kTbMaxSub = 10;
constexpr size_t fields_smem(int n_sub, size_t tsz) {
  const size_t L = kTbCells + 2 * halo_fields(n_sub);
  return tsz * (tile1_words(L, tsz) + 6 * (L + 1));
}
constexpr size_t rk4_adj_smem(int n_sub, size_t tsz) {
  const size_t L = kTbCells + 2 * halo_rk4_adj(n_sub), Ln = L + 1;
  return 8 * (8 * L + 11 * Ln) + tsz * (tile1_words(L, tsz) + (8 * (size_t)n_sub) * L);
}

// this thread's part of a tile
template <typename T>
__device__ __forceinline__ Tile1<T> window_tile(const Tile& t, T* mem) {
  Tile1<T> r;
  r.L = t.L;
  r.half = blockDim.x / 2;
  r.comp = (int)threadIdx.x >= r.half;
  r.a = threadIdx.x - r.comp * r.half;
  r.S = mem;
  r.E = mem + 2 * t.L;
  return r;
}

// One step's moments from the deposit sums q, the n_sub RK4 substeps of Ohm +
// Faraday with n, u frozen, then E, Bbar for the next gather and the new B,
// all into state b (B is read by neighbouring tiles: its buffer is another).
// Clears qz, the sums of the step after this one. A chain of dependent passes
// with few operations each (tile1_substep; the moments one quantity per
// thread, the division once): 9.4 -> 6.5 us FP32,
// 22.6 -> 13.0 us FP64 per step.
template <typename T>
__global__ void __launch_bounds__(fields_threads(kTbMaxSub))
    k_win_fields(const T* __restrict__ Bin, State<T> b, const unsigned long long* __restrict__ q,
                 unsigned long long* __restrict__ qz, Geo g, Phys ph, FieldConst<T> fc,
                 int n_sub) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nx = g.nx, nxn = g.nxn, t0 = threadIdx.x, nt = blockDim.x;
  const Tile t(blockIdx.x, nx, halo_fields(n_sub));
  const int L = t.L, Ln = L + 1;
  Tile1<T> w = window_tile<T>(t, (T*)smem);
  T* sn = w.S + tile1_words(L, sizeof(T));  // [Ln] n
  T* sinv = sn + Ln;                        // [Ln] 1/n
  T* spg = sinv + Ln;                       // [Ln] pressure term
  T* su = spg + Ln;                         // [3][Ln] J, then u
  const int a = w.a, gc = t.lo + a;         // this thread's cell and node
  T bxm = (T)0, bxc = (T)0, bxp = (T)0;
  w.b = (T)0;
  if (a < L) {
    w.b = Bin[(w.comp + 1) * nx + gc];
    w.S[w.comp * L + a] = w.b;
    bxp = Bin[t.lo + min(a + 1, L - 1)];
  }
  if (a < Ln) {
    bxm = Bin[t.lo + max(a - 1, 0)];
    bxc = Bin[t.lo + min(a, L - 1)];
  }
  for (int k = t0; k < 4 * Ln; k += nt) {
    const int c = k / Ln, i = k - c * Ln, gi = t.lo + i;
    const T v = moment_sum<T>(gi, c, q, g);
    if (c == 0) {
      const T nf = (T)ph.n_floor, n = v < nf ? nf : v;
      sn[i] = n;
      if (t.owns_node(gi)) {
        b.n[gi] = n;
        b.nraw[gi] = v;
      }
    } else {
      su[(c - 1) * Ln + i] = v;
    }
    if (t.owns_node(gi)) qz[c * nxn + gi] = 0ull;
  }
  __syncthreads();
  for (int k = t0; k < 5 * Ln; k += nt) {
    const int c = k / Ln, i = k - c * Ln, gi = t.lo + i;
    if (c < 4) {  // u = J / n, then 1/n
      const T v = (c < 3 ? su[k] : (T)1) / sn[i];
      if (c == 3) {
        sinv[i] = v;
      } else {
        su[k] = v;
        if (t.owns_node(gi)) b.u[c * nxn + gi] = v;
      }
    } else {
      const T dnx = (sn[t.node(gi + 1)] - sn[t.node(gi - 1)]) * fc.hdx;
      spg[i] = -(fc.te * dnx);
    }
  }
  __syncthreads();
  auto node = [&](int i, T bm, T bp) {
    return Node1<T>{sinv[i], (T)0.5 * (bm + bp), su[i], su[Ln + i], su[2 * Ln + i]};
  };
  if (a < Ln) w.n0 = node(a, bxm, bxc);
  if (sizeof(T) == 4 && a < L) w.n1 = node(a + 1, bxc, bxp);
  for (int sub = 0; sub < n_sub; ++sub) tile1_substep<T>(w, fc, nullptr);
  if (w.comp == 0 && a < Ln && t.owns_node(gc)) {
    T E[3], Bb[3];
    tile1_ohm<T>(w.S, L, max(a - 1, 0), min(a, L - 1), w.n0, spg[a], fc, E, Bb);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      b.E[c * nxn + gc] = E[c];
      b.Bb[c * nxn + gc] = Bb[c];
    }
  }
  if (a < L && t.owns_cell(gc)) {
    b.B[(w.comp + 1) * nx + gc] = w.b;
    if (w.comp == 0) b.B[gc] = bxc;
  }
}

// Reverse of one step's field update and moments. In: B^n (Bn), B^{n+1},
// M^{n+1} (b), the adjoints lE, lBb of E^{n+1}, Bbar^{n+1} (the next step's
// particles), lBin of B^{n+1} from the later steps. Per tile:
//   1. the RK4 stage inputs from B^n with n, u frozen at M^{n+1}, recomputed
//      with the forward's arithmetic (Y);
//   2. the adjoint of E^{n+1}'s Ohm: its shares of the adjoints of B^{n+1} and
//      of M^{n+1} (every node of the tile, from global memory: no halo needed);
//   3. the stages in reverse, one transverse component per half of the block:
//      E's adjoint at the nodes from K's, its curl and Bbar parts to the two
//      cells of a node, the running sum and the next stage's adjoint; after
//      each substep the n and u adjoints of its four stages, two stages per
//      half (E_x's adjoint is zero in the stages: no pressure term, and B_x
//      is constant, so n's and u's adjoints are four running sums that take
//      their node factors once at the end);
//   4. the adjoints of the raw deposit sums (lNr, lJ) from those of M^{n+1}.
// lE, lBb of the step before are cleared (lEz, lBbz). A thread has one cell
// and one node; its factors and sums stay in registers. Bound by the FP64
// pipe: an FP64 instruction holds an SM quarter for 64 cycles, so the time is
// the FP64 instruction count per warp: 8 per reverse stage, four warps,
// against about 110, two warps and a launch of its own for 2. before: 43 + 8.6
// -> 17.2 us per step FP32, 54 + 8 -> 21.0 us FP64. FP32 values are widened by integer
// operations, off that pipe.
template <typename T>
__global__ void __launch_bounds__(rk4_adj_threads(kTbMaxSub))
    k_win_rk4_adj(Geo g, Phys ph, FieldConst<T> fc, int ns, const T* __restrict__ Bn, State<T> b,
                  const double* __restrict__ lE, const double* __restrict__ lBb,
                  double* __restrict__ lEz, double* __restrict__ lBbz,
                  const double* __restrict__ lBin, double* __restrict__ lBout,
                  T* __restrict__ lNr, T* __restrict__ lJ) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nx = g.nx, nxn = g.nxn;
  const Tile t(blockIdx.x, nx, halo_rk4_adj(ns));
  const int L = t.L, Ln = L + 1;
  double* gk = (double*)smem;    // [4][2][L] stage adjoints of one substep
  double* Pp = gk + 8 * L;       // [2][Ln] a node's part for its right cell
  double* Pm = Pp + 2 * Ln;      // [2][Ln] and for its left cell
  double* lp = Pm + 2 * Ln;      // [Ln] pressure weight of E^{n+1}'s Ohm
  double* lM = lp + Ln;          // [4][Ln] the moments' sums of half 1 for half 0
  double* lUx = lM + 4 * Ln;     // [Ln] u_x's part of E^{n+1}'s Ohm
  Tile1<T> w = window_tile<T>(t, (T*)(lUx + Ln));
  T* Y = w.S + tile1_words(L, sizeof(T));  // [4 ns][2][L] stage inputs
  const double h = ph.h, hh = ph.hh, h6 = ph.h6, idx = ph.idx;
  const int comp = w.comp, a = w.a, gi = t.lo + a;  // this thread's cell and node
  const bool node = a < Ln, cell = a < L;
  const int cm = max(a - 1, 0), cp = min(a, L - 1);
  T bxm = (T)0, bxc = (T)0, bxp = (T)0, n0 = (T)1, n1 = (T)1;
  w.b = (T)0;
  if (cell) {
    w.b = Bn[(comp + 1) * nx + gi];
    w.S[comp * L + a] = w.b;
  }
  if (node) {
    bxm = Bn[t.lo + cm];
    bxc = Bn[t.lo + cp];
    n0 = b.n[gi];
    w.n0.ux = b.u[gi];
    w.n0.uy = b.u[nxn + gi];
    w.n0.uz = b.u[2 * nxn + gi];
    if (sizeof(T) == 4 && cell) {
      bxp = Bn[t.lo + min(a + 1, L - 1)];
      n1 = b.n[gi + 1];
      w.n1.ux = b.u[gi + 1];
      w.n1.uy = b.u[nxn + gi + 1];
      w.n1.uz = b.u[2 * nxn + gi + 1];
    }
    if (comp == 0 && t.owns_node(gi)) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        lEz[c * nxn + gi] = 0.0;
        lBbz[c * nxn + gi] = 0.0;
      }
    }
  }
  w.n0.inv = (T)1 / n0;
  w.n0.bbx = (T)0.5 * (bxm + bxc);
  if (sizeof(T) == 4) {
    w.n1.inv = (T)1 / n1;
    w.n1.bbx = (T)0.5 * (bxc + bxp);
  }
  const double in = sizeof(T) == 8 ? (double)w.n0.inv : 1.0 / wide_double(n0);
  const double bbx = wide_double(w.n0.bbx);
  __syncthreads();
  // 1.
  for (int sub = 0; sub < ns; ++sub) tile1_substep<T>(w, fc, Y + (size_t)8 * sub * L);
  // 2. half 0: B's part, half 1: the moments' part
  double m0 = 0.0, m1 = 0.0, m2 = 0.0;  // half 1: n's and u_y's, u_z's parts
  if (node) {
    const int im = min(max(gi - 1, 0), nx - 1), ip = min(gi, nx - 1);
    const double Bm[3] = {wide_double(b.B[im]), wide_double(b.B[nx + im]),
                          wide_double(b.B[2 * nx + im])};
    const double Bp[3] = {wide_double(b.B[ip]), wide_double(b.B[nx + ip]),
                          wide_double(b.B[2 * nx + ip])};
    const double u[3] = {wide_double(w.n0.ux), wide_double(w.n0.uy), wide_double(w.n0.uz)};
    const double lex = lE[gi], ley = lE[nxn + gi], lez = lE[2 * nxn + gi];
    if (comp == 0) {
      const OhmAdj r = ohm_adj_point(Bm, Bp, in, 0.0, u, lex, ley, lez, ph);
      const double hy = 0.5 * (r.P[0] + lBb[nxn + gi]), hz = 0.5 * (r.P[1] + lBb[2 * nxn + gi]);
      const double dy = r.P[2] * idx, dz = r.P[3] * idx;
      Pp[a] = hy + dy;
      Pp[Ln + a] = hz + dz;
      Pm[a] = hy - dy;
      Pm[Ln + a] = hz - dz;
    } else {
      const int ipn = (gi + 1 > nx) ? 2 * nx - (gi + 1) : gi + 1;
      const int imn = (gi - 1 < 0) ? -(gi - 1) : gi - 1;
      const double pgn = -(ph.te * ((wide_double(b.n[ipn]) - wide_double(b.n[imn])) * ph.hdx));
      const OhmAdj r = ohm_adj_point(Bm, Bp, in, pgn, u, lex, ley, lez, ph);
      m0 = r.ln;
      // (a wall node's pressure difference is zero by the mirrored density)
      lp[a] = (gi == 0 || gi == nx) ? 0.0 : r.lp;
      lUx[a] = r.lu[0];
      m1 = r.lu[1];
      m2 = r.lu[2];
    }
  }
  // the stage adjoint's node factors (times 1/dx: E's adjoint from K's)
  const double a5 = 0.5 * (ph.jcr * in + wide_double(w.n0.ux)), ei = ph.eta * idx;
  const double e1 = (a5 - ei) * idx, e2 = (a5 + ei) * idx, bi = bbx * in * idx * idx;
  __syncthreads();
  // a cell's part from its two nodes (the wall nodes read cell 0 or nx - 1 twice)
  const double* pp = Pp + comp * Ln;
  const double* pm = Pm + comp * Ln;
  auto cell_part = [&]() {
    double l = pp[a] + pm[a + 1];
    if (gi == 0) l += pm[0];
    if (gi == nx - 1) l += pp[a + 1];
    return l;
  };
  double lsum = 0.0;  // the adjoint of B at the thread's cell
  if (cell) lsum = lBin[(comp + 1) * nx + gi] + cell_part();
  // 3. lambda_start = lambda_end + sum over the stages of lambda_Y; the stage
  //    adjoints g4 = h6 lend, g3 = 2 h6 lend + h lY4, g2 = 2 h6 lend + hh lY3,
  //    g1 = h6 lend + hh lY2
  double A[4] = {0.0, 0.0, 0.0, 0.0};  // the n and u adjoints' sums
  // (a K's adjoint is read at cells gi - 1 and gi; none beyond a wall)
  const bool left = gi >= 1, right = gi < nx;
  for (int sub = ns - 1; sub >= 0; --sub) {
    const double hl = h6 * lsum, hl2 = hl + hl;
    if (cell) gk[6 * L + comp * L + a] = hl;
    __syncthreads();
#pragma unroll
    for (int s = 3; s >= 0; --s) {
      const double* G = gk + 2 * s * L;
      if (node) {
        const double gym = left ? G[cm] : 0.0, gy = right ? G[cp] : 0.0;
        const double gzm = left ? G[L + cm] : 0.0, gz = right ? G[L + cp] : 0.0;
        const double ley = gz - gzm, lez = gym - gy;
        if (comp == 0) {
          const double x = ley * bi;
          Pp[a] = __fma_rn(-lez, e1, x);
          Pm[a] = __fma_rn(-lez, e2, -x);
        } else {
          const double x = lez * bi;
          Pp[Ln + a] = __fma_rn(ley, e1, x);
          Pm[Ln + a] = __fma_rn(ley, e2, -x);
        }
      }
      __syncthreads();
      if (cell) {
        const double l = cell_part();
        lsum += l;
        if (s > 0)
          gk[(2 * (s - 1) + comp) * L + a] = __fma_rn(s == 3 ? h : hh, l, s == 1 ? hl : hl2);
      }
      __syncthreads();
    }
    // the n and u adjoints of the substep's stages: stages comp and comp + 2
    if (node) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int s = comp + 2 * r;
        const double* G = gk + 2 * s * L;
        const T* y = Y + (size_t)(2 * (4 * sub + s)) * L;
        const double gym = left ? G[cm] : 0.0, gy = right ? G[cp] : 0.0;
        const double gzm = left ? G[L + cm] : 0.0, gz = right ? G[L + cp] : 0.0;
        const double ley = gz - gzm, lez = gym - gy;  // (x 1/dx at the end)
        const double ym = wide_double(y[cm]), yp = wide_double(y[cp]);
        const double zm = wide_double(y[L + cm]), zp = wide_double(y[L + cp]);
        A[0] = __fma_rn(lez, zp - zm, __fma_rn(ley, yp - ym, A[0]));    // curl part of n's
        A[1] = __fma_rn(-lez, yp + ym, __fma_rn(ley, zp + zm, A[1]));  // u_x's, j_ext's
        A[2] += lez;                                                    // u_y's
        A[3] += ley;                                                    // u_z's
      }
    }
    __syncthreads();
  }
  if (cell && t.owns_cell(gi)) lBout[(comp + 1) * nx + gi] = lsum;
  // 4. half 1's sums to half 0
  if (node && comp == 1) {
    const double i2 = in * in;
    lM[a] = m0 - i2 * (idx * idx * bbx * A[0] + ph.jcr * (0.5 * idx * A[1]));
    lM[Ln + a] = lUx[a] + 0.5 * idx * A[1];
    lM[2 * Ln + a] = m1 + bbx * (idx * A[2]);
    lM[3 * Ln + a] = m2 - bbx * (idx * A[3]);
  }
  __syncthreads();
  if (node && comp == 0 && t.owns_node(gi)) {
    const double ux = 0.5 * idx * A[1];
    double ln = lM[a] - in * in * (idx * idx * bbx * A[0] + ph.jcr * ux);
    if (gi >= 1) ln += lp[a - 1];  // (own nodes have both neighbours in the tile)
    if (gi + 1 <= nx) ln -= lp[a + 1];
    const double lu[3] = {lM[Ln + a] + ux, lM[2 * Ln + a] + bbx * (idx * A[2]),
                          lM[3 * Ln + a] - bbx * (idx * A[3])};
    moments_adj_node<T>(gi, in, b.u, b.nraw, ln, lu, lNr, lJ, g, ph);
  }
}

// The adjoint of Ohm's law at the start of the window (B^0 and M^0 in a), after
// the first step's particles (lE, lBb): lB += its share.
template <typename T>
__global__ void __launch_bounds__(32)
    k_win_ohm_adj_start(State<T> a, Geo g, Phys ph, const double* __restrict__ lE,
                        const double* __restrict__ lBb, double* __restrict__ lB) {
  __shared__ double P[4][kTbCells + 1];
  const int nx = g.nx, nxn = g.nxn, t0 = threadIdx.x, nt = blockDim.x;
  const int c0 = blockIdx.x * kTbCells, c1 = min(nx, c0 + kTbCells);
  for (int k = t0; k <= c1 - c0; k += nt) {  // nodes c0 .. c1
    const int gi = c0 + k;
    const int im = min(max(gi - 1, 0), nx - 1), ip = min(gi, nx - 1);
    const double Bm[3] = {(double)a.B[im], (double)a.B[nx + im], (double)a.B[2 * nx + im]};
    const double Bp[3] = {(double)a.B[ip], (double)a.B[nx + ip], (double)a.B[2 * nx + ip]};
    const double u[3] = {(double)a.u[gi], (double)a.u[nxn + gi], (double)a.u[2 * nxn + gi]};
    const OhmAdj r = ohm_adj_point(Bm, Bp, 1.0 / (double)a.n[gi], 0.0, u, lE[gi], lE[nxn + gi],
                                   lE[2 * nxn + gi], ph);
    P[0][k] = r.P[0] + lBb[nxn + gi];
    P[1][k] = r.P[1] + lBb[2 * nxn + gi];
    P[2][k] = r.P[2];
    P[3][k] = r.P[3];
  }
  __syncthreads();
  for (int k = t0; k < c1 - c0; k += nt) {
    const int gc = c0 + k;
    const double Pc[4] = {P[0][k], P[1][k], P[2][k], P[3][k]};
    const double Pc1[4] = {P[0][k + 1], P[1][k + 1], P[2][k + 1], P[3][k + 1]};
    double ly, lz;
    curl_adj_point(Pc, Pc1, gc == 0, gc == nx - 1, ph.idx, ly, lz);
    lB[nx + gc] += ly;
    lB[2 * nx + gc] += lz;
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Adjoint of one step for slot p < np1 (alive at the end of the step or born
// in it). In: lf, lv = adjoints of the state after the step;
// lNr, lJ = adjoints of the step's deposit; E, Bb = the node fields the
// step's gather used. Out: lf, lv = adjoints of the state before the step
// (zero for slots born or removed in it); the adjoints of E and Bbar
// at the particle and its offset in the cell c0 (out; returns c0, or -1 when it
// has none); its terms
// of grad[M] (u_cr, into gucr) and grad[M + 1] (u2, into gu2). The injection's
// and the faux-shock return's adjoints are taken in FP64; those of the deposit
// and the push (Boris, gather) in the run's precision, that of the per-slot
// adjoints lf, lv and of lNr, lJ. The caller sums E's and Bbar's over a piece of
// a cell's slots in the run's precision, pieces and the gradient in FP64.
template <typename T>
__device__ __forceinline__ int particle_adj_slot(int p, const Win<T>& w, const State<T>& a0,
                                                 const Slots<T>& t1, const uint8_t* ev,
                                                 const Geo& g, const Phys& ph,
                                                 const PushConst<T>& pc, long long step,
                                                 int np0, double& gu2, double& gucr, T out[7]) {
  using A = T;  // arithmetic of the push's adjoint
  const int nxn = g.nxn;
  const int cap = w.cap;
  const Slots<T>& t0 = a0.s;
  {
    const bool born = p >= np0;
    // every load of the slot before the first decision (a slot without a
    // particle reads values it does not use)
    const uint8_t e = born ? (uint8_t)kEvNone : ev[p];
    const int c1 = t1.ci[p], c0 = born ? -1 : t0.ci[p];
    const uint32_t id = w.s.id[p];
    const A f1 = t1.f[p];
    const A v1[3] = {t1.v[p], t1.v[cap + p], t1.v[2 * cap + p]};
    A lf1 = w.lf[p];
    A lv[3] = {w.lv[p], w.lv[cap + p], w.lv[2 * cap + p]};
    const T ft0 = born ? (T)0 : t0.f[p];
    T vxt = (T)0, vyt = (T)0, vzt = (T)0;
    if (!born) {
      vxt = t0.v[p];
      vyt = t0.v[cap + p];
      vzt = t0.v[2 * cap + p];
    }
    if (c1 < 0 || (!born && c0 < 0) || e == kEvRemoved) {
      w.lf[p] = (T)0;
      w.lv[p] = w.lv[cap + p] = w.lv[2 * cap + p] = (T)0;
      return -1;
    }
    // ---- deposit at the state after the step (in the run's precision)
    A wp;
    if constexpr (sizeof(T) == 4) wp = (id & kIdCR) ? pc.wcr : pc.wth;
    else wp = (id & kIdCR) ? ph.w_cr : ph.w_th;
    {
      A dj = w.lNr[c1 + 1] - w.lNr[c1];
      for (int c = 0; c < 3; ++c) {
        const A ja = w.lJ[c * nxn + c1], jb = w.lJ[c * nxn + c1 + 1];
        dj += (jb - ja) * v1[c];
        lv[c] += wp * (((A)1 - f1) * ja + f1 * jb);
      }
      lf1 += wp * dj;
    }
    if (born) {
      if (id & kIdCR) {  // v = p (mu, sn c, sn s) - u_cr x, mu = a + (1 - a) s1, a = u_cr / p
        double v[3], U[4];
        const double X = cr_draw(ph, id & kIdMask, step, v, U);
        const double pv = ph.p_iso_v, s1 = U[0], mu = (v[0] + ph.u_cr) / pv;
        const double sn = sqrt(fmax(1.0 - mu * mu, 0.0));
        const double dmu = (1.0 - s1) / pv;
        const double dsn = (sn > 0.0) ? -mu * dmu / sn : 0.0;
        const double dvx = pv * dmu - 1.0, dvy = pv * dsn * U[1], dvz = pv * dsn * U[2];
        gucr += (double)lv[0] * dvx + (double)lv[1] * dvy + (double)lv[2] * dvz;
        const double ix = floor(X);
        if (ix >= 0.0 && ix < (double)g.nx)  // placement not clamped
          gucr += (double)lf1 * U[3] * dvx * ph.dtdx;
      }
      w.lf[p] = (T)0;
      w.lv[p] = w.lv[cap + p] = w.lv[2 * cap + p] = (T)0;
      return -1;
    }
    // ---- recompute the push from the state before the step
    const A f0 = (A)ft0;
    const A v0[3] = {vxt, vyt, vzt};
    // (FP32: E at the particle rounded as in the forward, so that the gradient is
    // that of the trajectory it took; FP64: E0 + f (E1 - E0), the difference is
    // needed anyway)
    A Ep[3], Bp[3], Ed[3], Bd[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const A e0 = a0.E[c * nxn + c0], b0 = a0.Bb[c * nxn + c0];
      Ed[c] = a0.E[c * nxn + c0 + 1] - e0;
      Bd[c] = a0.Bb[c * nxn + c0 + 1] - b0;
      if constexpr (sizeof(T) == 4) {
        Ep[c] = fmaT(f0, a0.E[c * nxn + c0 + 1], ((A)1 - f0) * e0);
        Bp[c] = fmaT(f0, a0.Bb[c * nxn + c0 + 1], ((A)1 - f0) * b0);
      } else {
        Ep[c] = fmaT(f0, Ed[c], e0);
        Bp[c] = fmaT(f0, Bd[c], b0);
      }
    }
    // ---- Boris: v+ = q + em, q = vm + p x s, p = vm + vm x t,
    //      s = (2 / (1 + t.t)) t, t = hdt B, vm = v + em, em = hdt E
    const A hdt = pc.hdt;
    A em[3], vm[3], t[3], sv[3], pp[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      em[c] = hdt * Ep[c];
      vm[c] = v0[c] + em[c];
      t[c] = hdt * Bp[c];
    }
    const A fct = (A)2 * rcpT((A)1 + fmaT(t[2], t[2], fmaT(t[1], t[1], t[0] * t[0])));
    for (int c = 0; c < 3; ++c) sv[c] = fct * t[c];
    pp[0] = vm[0] + fmaT(vm[1], t[2], -(vm[2] * t[1]));
    pp[1] = vm[1] + fmaT(vm[2], t[0], -(vm[0] * t[2]));
    pp[2] = vm[2] + fmaT(vm[0], t[1], -(vm[1] * t[0]));
    A lvp[3];  // adjoint of vp
    A lf0;
    if (e == kEvReturned) {
      // vnew = R(vp; u2), f1 = clamp(gf * vnew_x * dtdx), gf = Xn/(Xn - Xo);
      // vp: the velocity before the return
      const A vp[3] = {fmaT(pp[1], sv[2], fmaT(-pp[2], sv[1], vm[0])) + em[0],
                       fmaT(pp[2], sv[0], fmaT(-pp[0], sv[2], vm[1])) + em[1],
                       fmaT(pp[0], sv[1], fmaT(-pp[1], sv[0], vm[2])) + em[2]};
      const Philox4 r = draw4(ph.seed, id & kIdMask, step, kPurposeFS);
      const double s1 = sqrt(u01(r.x[1]));
      double cs, sn2;
      fs_sincos2pi(u01(r.x[2]), &cs, &sn2);
      const double u2 = ph.u2;
      const double wx = (double)vp[0] + u2;
      const double wv = sqrt(wx * wx + (double)vp[1] * vp[1] + (double)vp[2] * vp[2]);
      const double a = u2 / wv;
      const double mu = a + (1.0 - a) * s1;
      const double snm = sqrt(fmax(1.0 - mu * mu, 0.0));
      const double vnx = wv * mu - u2;
      const double av = (double)vp[0] * ph.dtdx;  // Xn - Xo
      const double Xo = (double)c0 + (double)f0;
      const double gf = (Xo + av) / av;
      const double fraw = gf * vnx * ph.dtdx;
      double Lx = lv[0], Ly = lv[1], Lz = lv[2];
      const double lf1d = lf1;
      double lXo = 0.0, lav = 0.0;
      if (fraw >= 0.0 && fraw < 1.0) {
        Lx += lf1d * gf * ph.dtdx;
        const double lgf = lf1d * vnx * ph.dtdx;
        lXo = lgf / av;
        lav = -lgf * Xo / (av * av);
      }
      // through the return map R
      const double Lsn = (Ly * cs + Lz * sn2) * wv;
      double Lw = Lx * mu + (Ly * cs + Lz * sn2) * snm;
      const double Lmu = Lx * wv - ((snm > 0.0) ? Lsn * mu / snm : 0.0);
      const double La = Lmu * (1.0 - s1);
      Lw -= La * u2 / (wv * wv);
      double Lu2 = -Lx + La / wv;
      Lu2 += Lw * wx / wv;
      gu2 += Lu2;
      lvp[0] = (A)(Lw * wx / wv + lav * ph.dtdx);
      lvp[1] = (A)(Lw * vp[1] / wv);
      lvp[2] = (A)(Lw * vp[2] / wv);
      lf0 = (A)lXo;
    } else {
      lvp[0] = lv[0] + lf1 * pc.dtdx;
      lvp[1] = lv[1];
      lvp[2] = lv[2];
      lf0 = lf1;
    }
    // ---- Boris adjoint
    const A* Lq = lvp;
    A Lem[3] = {lvp[0], lvp[1], lvp[2]};
    A Lvm[3] = {Lq[0], Lq[1], Lq[2]};
    // q = vm + p x s: L_p = s x L_q, L_s = L_q x p
    const A Lp[3] = {sv[1] * Lq[2] - sv[2] * Lq[1], sv[2] * Lq[0] - sv[0] * Lq[2],
                          sv[0] * Lq[1] - sv[1] * Lq[0]};
    const A Ls[3] = {Lq[1] * pp[2] - Lq[2] * pp[1], Lq[2] * pp[0] - Lq[0] * pp[2],
                          Lq[0] * pp[1] - Lq[1] * pp[0]};
    // p = vm + vm x t: L_vm += L_p + t x L_p, L_t = L_p x vm
    Lvm[0] += Lp[0] + (t[1] * Lp[2] - t[2] * Lp[1]);
    Lvm[1] += Lp[1] + (t[2] * Lp[0] - t[0] * Lp[2]);
    Lvm[2] += Lp[2] + (t[0] * Lp[1] - t[1] * Lp[0]);
    A Lt[3] = {Lp[1] * vm[2] - Lp[2] * vm[1], Lp[2] * vm[0] - Lp[0] * vm[2],
                    Lp[0] * vm[1] - Lp[1] * vm[0]};
    // s = fct t, fct = 2 / (1 + tt)
    const A Lf = Ls[0] * t[0] + Ls[1] * t[1] + Ls[2] * t[2];
    const A Ltt = -Lf * fct * fct * (A)0.5;
    for (int c = 0; c < 3; ++c) {
      Lt[c] += fct * Ls[c] + (A)2 * Ltt * t[c];
      Lem[c] += Lvm[c];
    }
    const A LE[3] = {hdt * Lem[0], hdt * Lem[1], hdt * Lem[2]};
    const A LB[3] = {hdt * Lt[0], hdt * Lt[1], hdt * Lt[2]};
    // ---- gather adjoint at the state before the step: the adjoints of E and
    //      Bbar at the particle and its offset go to the caller, which
    //      shares them out to the nodes c0, c0 + 1
    A dlf = (A)0;  // summed on its own: one rounding at the size of lf0 a step
    for (int c = 0; c < 3; ++c) {
      out[c] = LE[c];
      out[3 + c] = LB[c];
      dlf = fmaT(LE[c], Ed[c], fmaT(LB[c], Bd[c], dlf));
    }
    lf0 += dlf;
    out[6] = f0;
    w.lf[p] = (T)lf0;
    w.lv[p] = (T)Lvm[0];
    w.lv[cap + p] = (T)Lvm[1];
    w.lv[2 * cap + p] = (T)Lvm[2];
    return c0;
  }
}

// Adjoint of one step for every slot p < np1 (slots alive at the end of the
// step or born in it): particle_adj_slot per slot; the shares of E and Bbar at
// a slot's two nodes (12 values) are sorted by cell over the block and added
// per cell by one warp, 12 lanes and two splits (cell_sort), then once per
// cell by FP64 atomics. (Before: per lane group by 60 shuffles a cell in
// FP32, 12 atomics per particle in FP64.) The last blocks hold the slots born
// in the step, whose FP64 draw chain is long: blocks are taken from both ends.
template <typename T>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 4 : 2)
    k_win_particle_adj(Win<T> w, State<T> a0, Slots<T> t1, const uint8_t* ev, double* lE,
                       double* lBb, Geo g, Phys ph, PushConst<T> pc, long long step, int np0,
                       int np1, int M) {
  __shared__ CellSort cs;
  __shared__ T rec[kBlock][8];  // adjoints of E, Bbar; the node weights 1 - f, f
  const int nxn = g.nxn;
  const int lane = threadIdx.x & 31;
  double gu2 = 0.0, gucr = 0.0;
  const int blk = (blockIdx.x & 1) ? gridDim.x - 1 - blockIdx.x / 2 : blockIdx.x / 2;
  const int p = blk * kBlock + threadIdx.x;
  T a[7];
  const int c0 =
      (p < np1) ? particle_adj_slot<T>(p, w, a0, t1, ev, g, ph, pc, step, np0, gu2, gucr, a) : -1;
  // value k of a cell's 12: component k / 2 (E, then Bbar), node k & 1
  auto target = [&](int k, int c) {
    return (k < 6 ? lE + (k >> 1) * nxn : lBb + ((k >> 1) - 3) * nxn) + c + (k & 1);
  };
  int base, range;
  const int pos = cell_sort(cs, c0, base, range);
  if (range > kSortKeys) {
    if (c0 >= 0)
#pragma unroll
      for (int k = 0; k < 12; ++k)
        atomicAdd(target(k, c0), wide_double(a[k >> 1] * ((k & 1) ? a[6] : (T)1 - a[6])));
  } else {
    if (c0 >= 0) {
#pragma unroll
      for (int k = 0; k < 6; ++k) rec[pos][k] = a[k];
      rec[pos][6] = (T)1 - a[6];
      rec[pos][7] = a[6];
    }
    __syncthreads();
    const int k = lane & 15, pieces = range ? cs.pieces : 0;
    for (int c = threadIdx.x >> 5; c < pieces; c += kBlock / 32) {
      const int b1 = cs.to[c];
      T s = (T)0;
      if (k < 12)
#pragma unroll 4
        for (int i = cs.from[c] + (lane >> 4); i < b1; i += 2)
          s = fmaT(rec[i][k >> 1], rec[i][6 + (k & 1)], s);
      s += __shfl_xor_sync(0xffffffffu, s, 16);
      if (lane < 12) atomicAdd(target(k, base + cs.cell[c]), wide_double(s));
    }
  }
  // only slots that were returned or injected add to these: most warps have
  // none (tested on the bit patterns, off the FP64 pipe)
  const bool any = __double_as_longlong(gu2) != 0 || __double_as_longlong(gucr) != 0;
  if (__any_sync(0xffffffffu, any)) {
    gu2 = warp_sum_d(gu2);
    gucr = warp_sum_d(gucr);
    if ((threadIdx.x & 31) == 0) {
      if (gucr != 0.0) atomicAdd(&w.grad[M], gucr);
      if (gu2 != 0.0) atomicAdd(&w.grad[M + 1], gu2);
    }
  }
}

// d loss / d a_m = sum_c lB_y(c) cos(arg) + lB_z(c) sin(arg), a CTA per mode
// and 256 cells (grad is zero before)
__global__ void k_win_mode_grad(const double* lB, double* grad, const double* phases, Geo g,
                                double dx) {
  const int m = blockIdx.x;
  const double L = (double)g.nx * dx;
  double s = 0.0;
  const int i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i < g.nx) {
    const double x = ((double)i + 0.5) * dx;
    const double arg = 2.0 * 3.14159265358979323846 * (double)(m + 1) * x / L + phases[m];
    double sn, cs;
    sincos(arg, &sn, &cs);
    s = lB[g.nx + i] * cs + lB[2 * g.nx + i] * sn;
  }
  s = warp_sum_d(s);
  if ((threadIdx.x & 31) == 0) atomicAdd(&grad[m], s);
}

}  // namespace win
}  // namespace fsx

// =====================================================================
// Host side and C ABI
// =====================================================================
using namespace fsx;
using namespace fsx::win;

namespace {
constexpr size_t kAl = 256;
inline size_t al(size_t x) { return (x + kAl - 1) / kAl * kAl; }
inline int blocks(long long n) { return (int)std::max<long long>(1, (n + kBlock - 1) / kBlock); }
inline int tiles(int nx) { return (nx + kTbCells - 1) / kTbCells; }
}  // namespace

struct fs_window {
  fs_params p;
  Geo g;
  Phys ph;
  int steps, ckpt, nseg, M, loss_i0;
  long long n_init;
  int cap;
  size_t tsz;  // sizeof(T)
  char* base;
  cudaStream_t st;
  // regions (byte offsets)
  size_t o_state, o_ckpt, o_tape, o_ev, o_tapeB, o_tapeM, o_tapeE, o_fields, o_q, o_ctr, o_adj,
      o_params, o_sched;
  // slot schedule: slots at the start of step n (n = 0..steps; also on the
  // device); a slot born in the window has its slot number as id
  std::vector<int> np_at;
  // the recompute of a segment beside the reversal of the one after it: its
  // stream and events (made by the first backward): a segment recomputed, and how
  // far the reversal is
  cudaStream_t side = nullptr;
  cudaEvent_t taped = nullptr, reversed = nullptr;
  bool have_forward = false;
  int qsel = 0;  // which of the two deposit sums the next step uses
  long long counts[5] = {0, 0, 0, 0, 0};  // of the last forward
};

namespace {

// bytes of one copy of the per-slot state (ci, f, v[3], id)
size_t slot_bytes(int cap, size_t tsz) {
  return al(4 * (size_t)cap) + al(tsz * cap) + al(3 * tsz * cap) + al(4 * (size_t)cap);
}
size_t tape_slot_bytes(int cap, size_t tsz) {  // ci, f, v
  return al(4 * (size_t)cap) + al(tsz * cap) + al(3 * tsz * cap);
}
size_t mom_bytes(int nxn, size_t tsz) { return 5 * al(tsz * nxn); }  // n, u[3], nraw

// per step the integer part of an accumulator advanced by ppc u_sh dt/dx
// (the engine's inflow count, one transverse row)
void injection_schedule(const Phys& ph, int steps, std::vector<int>* ninj) {
  double acc = 0.0;
  ninj->assign(steps, 0);
  for (int n = 0; n < steps; ++n) {
    acc = acc + ph.rate;
    const double fl = std::floor(acc);
    (*ninj)[n] = (int)fl;
    acc = acc - fl;
  }
}

// Entries of the tape for segments of up to K steps. A segment is recomputed while
// the one after it is reversed, into the entries that this has done with: the two
// run through the tape in opposite directions (tape_entry), one entry apart.
int tape_entries(int K, int nseg) { return K + (nseg > 1 ? 1 : 0); }

int window_sizes(const fs_params* p, int steps, int ckpt, long long n_init, int M, Geo* g,
                 Phys* ph, int* cap, size_t* total, size_t off[13]) {
  if (!p || steps < 1 || ckpt < 1 || n_init < 0 || M < 0 || M > 4096) return FS_EINVAL;
  if (p->dim != 1 || p->bc_x != FS_BC_FAUXSHOCK || p->c_light != 0.0) return FS_EINVAL;
  // the blocked field kernels keep a tile's RK4 stage inputs in shared memory
  const size_t tb = (p->precision == FS_FP64) ? 8 : 4;
  // (up to 10 substeps in FP32, 9 in FP64)
  if (p->n_sub < 1 || p->n_sub > (tb == 8 ? 9 : 10)) return FS_EINVAL;
  static_assert(rk4_adj_smem(10, 4) <= kMaxSmem && rk4_adj_smem(9, 8) <= kMaxSmem,
                "the reverse field kernel's tile fits a CTA");
  int rc = derive_geometry(p, g, ph);
  if (rc) return rc;
  std::vector<int> ninj;
  injection_schedule(*ph, steps, &ninj);
  long long c = n_init;
  const int kinds = (p->inject_thermal ? 1 : 0) + (p->cr_enable ? 1 : 0);
  for (int v : ninj) c += (long long)v * kinds;
  if (c > (1LL << 30)) return FS_EINVAL;
  *cap = (int)std::max<long long>(c, 1);
  const size_t tsz = (p->precision == FS_FP64) ? 8 : 4;
  const int nx = g->nx, nxn = g->nxn;
  const int nseg = (steps + ckpt - 1) / ckpt;
  const int K = std::min(ckpt, steps);
  size_t o = 0;
  off[0] = o; o += slot_bytes(*cap, tsz);                                  // state
  off[1] = o;                                                               // checkpoints
  o += (size_t)nseg * (slot_bytes(*cap, tsz) + al(3 * tsz * nx) + mom_bytes(nxn, tsz));
  const size_t KT = (size_t)tape_entries(K, nseg);                         // tape:
  off[2] = o; o += KT * tape_slot_bytes(*cap, tsz);                        // particles
  off[3] = o; o += KT * al((size_t)*cap);                                  // events
  off[4] = o; o += KT * al(3 * tsz * nx);                                  // B
  off[5] = o; o += KT * mom_bytes(nxn, tsz);                               // moments
  off[11] = o; o += (KT + 2) * 2 * al(3 * tsz * nxn);                      // E, Bbar (and of
                                                                            // two checkpoints)
  off[6] = o; o += 2 * al(3 * tsz * nxn) + 2 * al(3 * tsz * nx) + mom_bytes(nxn, tsz);
  off[7] = o; o += 2 * al(8 * 4 * (size_t)nxn);                            // fixed-point sums
  off[8] = o; o += al(8 * 8);                                              // counters
  off[9] = o;
  o += al(tsz * *cap) + al(3 * tsz * *cap);                                // lf, lv
  o += 8 * al(8 * 3 * (size_t)(nx + nxn));                                 // field adjoints
  off[10] = o; o += al(8 * (size_t)(3 * M + 2));                           // amps, phases, grad
  off[12] = o; o += al(4 * (size_t)(steps + 1));                           // slot schedule
  *total = o;
  return FS_OK;
}

template <typename T>
Slots<T> slots_at(char* b, int cap, bool with_id) {
  Slots<T> s;
  size_t o = 0;
  s.ci = (int*)(b + o); o += al(4 * (size_t)cap);
  s.f = (T*)(b + o); o += al(sizeof(T) * cap);
  s.v = (T*)(b + o); o += al(3 * sizeof(T) * cap);
  s.id = with_id ? (uint32_t*)(b + o) : nullptr;
  return s;
}

template <typename T>
Win<T> win_ptrs(fs_window* w) {
  Win<T> r;
  const int nx = w->g.nx, nxn = w->g.nxn;
  r.cap = w->cap;
  r.s = slots_at<T>(w->base + w->o_state, w->cap, true);
  char* f = w->base + w->o_fields;
  size_t o = 0;
  auto take = [&](size_t bytes) { char* q = f + o; o += al(bytes); return q; };
  r.E = (T*)take(3 * sizeof(T) * nxn);
  r.Bb = (T*)take(3 * sizeof(T) * nxn);
  r.B[0] = (T*)take(3 * sizeof(T) * nx);
  r.B[1] = (T*)take(3 * sizeof(T) * nx);
  r.n = (T*)take(sizeof(T) * nxn);
  r.u = (T*)take(3 * sizeof(T) * nxn);
  r.nraw = (T*)take(sizeof(T) * nxn);
  r.q[0] = (unsigned long long*)(w->base + w->o_q);
  r.q[1] = r.q[0] + al(8 * 4 * (size_t)nxn) / 8;
  r.ctr = (unsigned long long*)(w->base + w->o_ctr);
  char* a = w->base + w->o_adj;
  o = 0;
  auto tka = [&](size_t bytes) { char* q = a + o; o += al(bytes); return q; };
  r.lf = (T*)tka(sizeof(T) * w->cap);
  r.lv = (T*)tka(3 * sizeof(T) * w->cap);
  const size_t fb = 8 * 3 * (size_t)(nx + nxn);
  r.lB = (double*)tka(fb);
  r.lBx = (double*)tka(fb);
  for (int k = 0; k < 2; ++k) {
    r.lE[k] = (double*)tka(fb);
    r.lBb[k] = (double*)tka(fb);
  }
  r.lNr = (T*)tka(fb);
  r.lJ = (T*)tka(fb);
  r.grad = (double*)(w->base + w->o_params) + 2 * w->M;
  return r;
}

// dynamic shared memory of the blocked field kernels beyond the default 48 KB
template <typename T>
bool smem_opt_in(int n_sub) {
  return raise_smem<k_win_fields<T>>(fields_smem(n_sub, sizeof(T))) == cudaSuccess &&
         raise_smem<k_win_rk4_adj<T>>(rk4_adj_smem(n_sub, sizeof(T))) == cudaSuccess;
}

// checkpoint c: slots, B, moments
struct Ck {
  char* slots;
  char* B;
  char* mom;
};
Ck ckpt_at(fs_window* w, int c) {
  const size_t sb = slot_bytes(w->cap, w->tsz), bb = al(3 * w->tsz * w->g.nx);
  const size_t one = sb + bb + mom_bytes(w->g.nxn, w->tsz);
  char* b = w->base + w->o_ckpt + (size_t)c * one;
  return Ck{b, b + sb, b + sb + bb};
}
template <typename T>
void mom_ptrs(char* b, int nxn, T** n, T** u, T** r) {
  *n = (T*)b;
  *u = (T*)(b + al(sizeof(T) * nxn));
  *r = (T*)(b + 4 * al(sizeof(T) * nxn));
}
// where step k of a segment of parity t keeps its events and the state after it
size_t tape_entry(const fs_window* w, int t, int k) {
  return t ? tape_entries(std::min(w->ckpt, w->steps), w->nseg) - 1 - k : k;
}
uint8_t* ev_at(fs_window* w, int t, int k) {
  return (uint8_t*)(w->base + w->o_ev) + tape_entry(w, t, k) * al(w->cap);
}
// E, Bbar entry e (0 and 1: of the checkpoints of segments of either parity)
template <typename T>
void tape_E(fs_window* w, size_t e, State<T>* a) {
  const size_t b = al(3 * sizeof(T) * w->g.nxn);
  a->E = (T*)(w->base + w->o_tapeE + e * 2 * b);
  a->Bb = (T*)((char*)a->E + b);
}

// the state at the start of segment c: its checkpoint, with E, Bbar formed from it
template <typename T>
State<T> ckpt_state(fs_window* w, int c) {
  const Ck ck = ckpt_at(w, c);
  State<T> a;
  a.s = slots_at<T>(ck.slots, w->cap, false);
  a.B = (T*)ck.B;
  mom_ptrs<T>(ck.mom, w->g.nxn, &a.n, &a.u, &a.nraw);
  tape_E<T>(w, c & 1, &a);
  return a;
}
// state k of segment c (k >= 1: recomputed)
template <typename T>
State<T> seg_state(fs_window* w, int c, int k) {
  if (k == 0) return ckpt_state<T>(w, c);
  const size_t e = tape_entry(w, c & 1, k - 1);
  State<T> a;
  a.s = slots_at<T>(w->base + w->o_tape + e * tape_slot_bytes(w->cap, w->tsz), w->cap, false);
  a.B = (T*)(w->base + w->o_tapeB + e * al(3 * sizeof(T) * w->g.nx));
  mom_ptrs<T>(w->base + w->o_tapeM + e * mom_bytes(w->g.nxn, w->tsz), w->g.nxn, &a.n, &a.u,
              &a.nraw);
  tape_E<T>(w, 2 + e, &a);
  return a;
}

void cpy(void* d, const void* s, size_t n, cudaStream_t st) {
  cudaMemcpyAsync(d, s, n, cudaMemcpyDeviceToDevice, st);
}

// one forward step n from state a to state b; drawn: the slots that hold the
// ions born in it; ev: where the step's events go (or nullptr)
template <typename T>
void forward_step(fs_window* w, const Win<T>& r, int n, const State<T>& a, const State<T>& b,
                  const Slots<T>& drawn, uint8_t* ev, cudaStream_t st) {
  const int np = w->np_at[n], np1 = w->np_at[n + 1];
  unsigned long long *q = r.q[w->qsel], *qz = r.q[1 - w->qsel];
  if (np1 > 0)
    k_win_push_deposit<T><<<blocks(np1), kBlock, 0, st>>>(r, a, b.s, drawn, ev, q, w->g, w->ph,
                                                             push_const<T>(w->ph), n, np, np1);
  k_win_fields<T><<<tiles(w->g.nx), fields_threads(w->p.n_sub), fields_smem(w->p.n_sub, sizeof(T)), st>>>(
      a.B, b, q, qz, w->g, w->ph, field_const<T>(w->ph), w->p.n_sub);
  w->qsel ^= 1;
}

template <typename T>
void save_ckpt(fs_window* w, const State<T>& a, int c) {
  const Ck ck = ckpt_at(w, c);
  cpy(ck.slots, w->base + w->o_state, slot_bytes(w->cap, w->tsz), w->st);
  cpy(ck.B, a.B, 3 * sizeof(T) * w->g.nx, w->st);
  T *n, *u, *q;
  mom_ptrs<T>(ck.mom, w->g.nxn, &n, &u, &q);
  cpy(n, a.n, sizeof(T) * w->g.nxn, w->st);
  cpy(u, a.u, 3 * sizeof(T) * w->g.nxn, w->st);
  cpy(q, a.nraw, sizeof(T) * w->g.nxn, w->st);
}

template <typename T>
void ohm_of(fs_window* w, const State<T>& a, cudaStream_t st) {
  k_ohm<T, 1><<<blocks(w->g.nxn), kBlock, 0, st>>>(a.B, a.n, a.u, nullptr, a.E, a.Bb, nullptr,
                                                       w->g, w->ph);
}

template <typename T>
int do_forward(fs_window* w, const double* theta, double* loss) {
  Win<T> r = win_ptrs<T>(w);
  const int M = w->M;
  if (!(theta[M + 1] > 0.0) || !(theta[M] >= 0.0) || !(theta[M] < w->ph.p_iso_v))
    return FS_EINVAL;
  w->ph.u_cr = theta[M];
  w->ph.u2 = theta[M + 1];
  double* amps = (double*)(w->base + w->o_params);
  if (M > 0 && cudaMemcpyAsync(amps, theta, sizeof(double) * M, cudaMemcpyHostToDevice,
                               w->st) != cudaSuccess)
    return FS_ECUDA;
  cudaMemsetAsync(r.ctr, 0, 8 * 8, w->st);
  // initial state: the caller's particles (kept in checkpoint 0's slots
  // since fs_window_init), B0 + modes, moments, E
  Ck c0 = ckpt_at(w, 0);
  cpy(w->base + w->o_state, c0.slots, slot_bytes(w->cap, w->tsz), w->st);
  const int np0 = w->np_at[0], nborn = w->np_at[w->steps] - np0;
  if (nborn > 0)
    k_win_draw<T><<<blocks(nborn), kBlock, 0, w->st>>>(r, w->g, w->ph,
                                                       (const int*)(w->base + w->o_sched), w->steps);
  k_win_seed_B<T><<<(w->g.nx + kSeedCells - 1) / kSeedCells, kBlock, 0, w->st>>>(r.B[0], w->g, w->ph, w->p.dx, amps,
                                                          amps + M, M);
  const size_t qb = 8 * 4 * (size_t)w->g.nxn;
  cudaMemsetAsync(r.q[0], 0, qb, w->st);
  cudaMemsetAsync(r.q[1], 0, qb, w->st);
  State<T> a{r.s, r.B[0], r.n, r.u, r.nraw, r.E, r.Bb};
  // the initial moments: a deposit without a push (every slot taken as it is)
  if (np0 > 0)
    k_win_push_deposit<T><<<blocks(np0), kBlock, 0, w->st>>>(
        r, a, r.s, r.s, nullptr, r.q[1], w->g, w->ph, push_const<T>(w->ph), 0, 0, np0);
  k_win_moments<T><<<blocks(w->g.nxn), kBlock, 0, w->st>>>(r, r.q[1], w->g, w->ph);
  ohm_of<T>(w, a, w->st);
  w->qsel = 0;  // (the first step clears the other sums)
  for (int n = 0; n < w->steps; ++n) {
    if (n % w->ckpt == 0) save_ckpt<T>(w, a, n / w->ckpt);
    State<T> b = a;
    b.B = a.B == r.B[0] ? r.B[1] : r.B[0];
    forward_step<T>(w, r, n, a, b, r.s, nullptr, w->st);
    a = b;
  }
  double* dl = r.lBx;  // scratch for the loss (free outside the backward)
  k_win_loss<T><<<1, kBlock, 0, w->st>>>(a.B, w->g, w->ph, w->loss_i0, w->p.dx,
                                                       dl, nullptr, 1.0);
  unsigned long long c[4];
  if (cudaMemcpyAsync(loss, dl, 8, cudaMemcpyDeviceToHost, w->st) != cudaSuccess ||
      cudaMemcpyAsync(c, r.ctr, sizeof(c), cudaMemcpyDeviceToHost, w->st) != cudaSuccess ||
      cudaStreamSynchronize(w->st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return FS_ECUDA;
  for (int k = 0; k < 4; ++k) w->counts[k] = (long long)c[k];
  w->counts[4] = nborn;
  w->have_forward = true;
  return FS_OK;
}

// the side stream and its events; false if one cannot be made
bool make_side(fs_window* w) {
  if (!w->side && cudaStreamCreateWithFlags(&w->side, cudaStreamNonBlocking) != cudaSuccess)
    return false;
  for (cudaEvent_t* e : {&w->taped, &w->reversed})
    if (!*e && cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) return false;
  return true;
}

template <typename T>
int do_backward(fs_window* w, double dloss, double* grad) {
  if (!w->have_forward) return FS_EINVAL;
  if (!make_side(w)) return FS_ECUDA;
  // the recompute overwrites the forward's sums: a new forward is due
  w->have_forward = false;
  Win<T> r = win_ptrs<T>(w);
  const int nx = w->g.nx, nxn = w->g.nxn, M = w->M;
  const size_t fb = 8 * 3 * (size_t)(nx + nxn);
  cudaMemsetAsync(r.grad, 0, 8 * (M + 2), w->st);
  cudaMemsetAsync(r.lf, 0, sizeof(T) * w->cap, w->st);
  cudaMemsetAsync(r.lv, 0, 3 * sizeof(T) * w->cap, w->st);
  int esel = 0;  // lE, lBb of the state after the step being reversed (none at the end)
  cudaMemsetAsync(r.lE[0], 0, fb, w->st);
  cudaMemsetAsync(r.lBb[0], 0, fb, w->st);
  // d loss / d B at the end (the final field after the forward)
  k_win_loss<T><<<1, kBlock, 0, w->st>>>(r.B[w->steps & 1], w->g, w->ph, w->loss_i0, w->p.dx,
                                                  nullptr, r.lB, dloss);
  // Segment by segment from the end: recompute it, keeping every state, then
  // reverse it. The recompute of segment seg - 1 (it needs only its checkpoint)
  // runs on the side stream while segment seg is reversed: both are chains of
  // short kernels that leave most of the GPU idle. Its step k takes the tape
  // entry of step K - k of segment seg, so it follows the reversal of that step.
  const int K = std::min(w->ckpt, w->steps);
  auto follow = [](cudaEvent_t e, cudaStream_t from, cudaStream_t to) {
    return cudaEventRecord(e, from) == cudaSuccess && cudaStreamWaitEvent(to, e, 0) == cudaSuccess;
  };
  auto recompute = [&](int seg, int k) {
    const State<T> first = ckpt_state<T>(w, seg);
    if (k == 0) ohm_of<T>(w, first, w->side);
    forward_step<T>(w, r, seg * w->ckpt + k, seg_state<T>(w, seg, k), seg_state<T>(w, seg, k + 1),
                    first.s, ev_at(w, seg & 1, k), w->side);
  };
  if (!follow(w->reversed, w->st, w->side)) return FS_ECUDA;
  for (int k = 0; k < w->steps - (w->nseg - 1) * w->ckpt; ++k) recompute(w->nseg - 1, k);
  for (int seg = w->nseg - 1; seg >= 0; --seg) {
    const int n0 = seg * w->ckpt, n1 = std::min(w->steps, n0 + w->ckpt);
    // (st: after the segment's recompute; side: after the reversal of the segment
    // after it, which had the first entries and the checkpoint's E, Bbar)
    if (!follow(w->taped, w->side, w->st)) return FS_ECUDA;
    if (seg > 0)
      for (int k = 0; K - k >= n1 - n0; ++k) recompute(seg - 1, k);
    for (int n = n1 - 1; n >= n0; --n) {
      const int k = n - n0;
      const State<T> a = seg_state<T>(w, seg, k), b = seg_state<T>(w, seg, k + 1);
      // the step's field update and moments in reverse, with the Ohm's law
      // that followed it
      k_win_rk4_adj<T><<<tiles(nx), rk4_adj_threads(w->p.n_sub), rk4_adj_smem(w->p.n_sub, sizeof(T)), w->st>>>(
          w->g, w->ph, field_const<T>(w->ph), w->p.n_sub, a.B, b, r.lE[esel], r.lBb[esel],
          r.lE[1 - esel], r.lBb[1 - esel], r.lB, r.lBx, r.lNr, r.lJ);
      std::swap(r.lB, r.lBx);
      esel ^= 1;
      const int npa = w->np_at[n], npb = w->np_at[n + 1];
      if (npb > 0)
        k_win_particle_adj<T><<<blocks(npb), kBlock, 0, w->st>>>(
            r, a, b.s, ev_at(w, seg & 1, k), r.lE[esel], r.lBb[esel], w->g, w->ph,
            push_const<T>(w->ph), n, npa, npb, M);
      if (seg > 0) {
        if (!follow(w->reversed, w->st, w->side)) return FS_ECUDA;
        if (k > 0) recompute(seg - 1, K - k);
      }
    }
    if (seg == 0)
      k_win_ohm_adj_start<T><<<tiles(nx), 32, 0, w->st>>>(ckpt_state<T>(w, 0), w->g, w->ph, r.lE[esel],
                                                                  r.lBb[esel], r.lB);
  }
  double* phases = (double*)(w->base + w->o_params) + M;
  if (M > 0) k_win_mode_grad<<<dim3(M, blocks(nx)), kBlock, 0, w->st>>>(r.lB, r.grad, phases, w->g, w->p.dx);
  if (cudaMemcpyAsync(grad, r.grad, 8 * (M + 2), cudaMemcpyDeviceToHost, w->st) != cudaSuccess ||
      cudaStreamSynchronize(w->st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return FS_ECUDA;
  return FS_OK;
}

}  // namespace

extern "C" {

int fs_window_query(const fs_params* p, int steps, int ckpt_every, long long n_init,
                    int n_modes, size_t* bytes) {
  FS_GUARD_BEGIN
  if (!bytes) return FS_EINVAL;
  Geo g;
  Phys ph;
  int cap;
  size_t off[13];
  return window_sizes(p, steps, ckpt_every, n_init, n_modes, &g, &ph, &cap, bytes, off);
  FS_GUARD_END
}

int fs_window_init(const fs_params* p, int steps, int ckpt_every, long long n_init,
                   const double* x_init, const double* v_init, int n_modes,
                   const double* mode_phase, int loss_i0, void* dev_buf, size_t bytes,
                   void* cuda_stream, fs_window** out) {
  FS_GUARD_BEGIN
  if (!out || (n_init > 0 && (!x_init || !v_init)) || (n_modes > 0 && !mode_phase) || !dev_buf)
    return FS_EINVAL;
  *out = nullptr;
  Geo g;
  Phys ph;
  int cap;
  size_t need, off[13];
  int rc = window_sizes(p, steps, ckpt_every, n_init, n_modes, &g, &ph, &cap, &need, off);
  if (rc) return rc;
  if (bytes < need || ((uintptr_t)dev_buf % kAl) != 0) return FS_EINVAL;
  if (loss_i0 < 0 || loss_i0 > g.nx) return FS_EINVAL;
  for (long long k = 0; k < n_init; ++k)
    if (!(x_init[k] >= 0.0 && x_init[k] < (double)g.nx)) return FS_EINVAL;
  fs_window* w = new fs_window();
  w->p = *p;
  w->g = g;
  w->ph = ph;
  w->steps = steps;
  w->ckpt = ckpt_every;
  w->nseg = (steps + ckpt_every - 1) / ckpt_every;
  w->M = n_modes;
  w->loss_i0 = loss_i0;
  w->n_init = n_init;
  w->cap = cap;
  w->tsz = (p->precision == FS_FP64) ? 8 : 4;
  w->base = (char*)dev_buf;
  w->st = (cudaStream_t)cuda_stream;
  w->o_state = off[0]; w->o_ckpt = off[1]; w->o_tape = off[2]; w->o_ev = off[3];
  w->o_tapeB = off[4]; w->o_tapeM = off[5]; w->o_fields = off[6]; w->o_q = off[7];
  w->o_ctr = off[8]; w->o_adj = off[9]; w->o_params = off[10]; w->o_tapeE = off[11];
  w->o_sched = off[12];
  // slot schedule: initial particles, then per step the thermal and
  // cosmic-ray injections (ids continue from n_init)
  std::vector<int> ninj;
  injection_schedule(ph, steps, &ninj);
  const int kinds = (p->inject_thermal ? 1 : 0) + (p->cr_enable ? 1 : 0);
  w->np_at.assign(steps + 1, 0);
  long long np = n_init;
  for (int n = 0; n < steps; ++n) {
    w->np_at[n] = (int)np;
    np += (long long)ninj[n] * kinds;
  }
  w->np_at[steps] = (int)np;
  // initial particles into checkpoint 0's slots (cell + offset)
  const size_t tsz = w->tsz;
  std::vector<char> host(slot_bytes(cap, tsz), 0);
  int* hci = (int*)host.data();
  char* hf = host.data() + al(4 * (size_t)cap);
  char* hv = hf + al(tsz * cap);
  uint32_t* hid = (uint32_t*)(hv + al(3 * tsz * cap));
  for (int k = 0; k < cap; ++k) hci[k] = -1;
  for (long long k = 0; k < n_init; ++k) {
    const double X = x_init[k];
    const double ix = std::floor(X);
    hci[k] = (int)ix;
    const double fx = X - ix;
    hid[k] = (uint32_t)k;
    if (tsz == 8) {
      ((double*)hf)[k] = fx;
      for (int c = 0; c < 3; ++c) ((double*)hv)[(size_t)c * cap + k] = v_init[3 * k + c];
    } else {
      float ft = (float)fx;
      if (ft >= 1.0f) ft = 0x1.fffffep-1f;
      ((float*)hf)[k] = ft;
      for (int c = 0; c < 3; ++c) ((float*)hv)[(size_t)c * cap + k] = (float)v_init[3 * k + c];
    }
  }
  Ck c0 = ckpt_at(w, 0);
  bool ok = (tsz == 8 ? smem_opt_in<double>(p->n_sub) : smem_opt_in<float>(p->n_sub)) &&
            cudaMemcpyAsync(c0.slots, host.data(), host.size(), cudaMemcpyHostToDevice, w->st) ==
                cudaSuccess &&
            (n_modes == 0 ||
             cudaMemcpyAsync(w->base + w->o_params + 8 * (size_t)n_modes, mode_phase,
                             8 * (size_t)n_modes, cudaMemcpyHostToDevice, w->st) == cudaSuccess) &&
            cudaMemcpyAsync(w->base + w->o_sched, w->np_at.data(), 4 * ((size_t)steps + 1),
                            cudaMemcpyHostToDevice, w->st) == cudaSuccess &&
            cudaStreamSynchronize(w->st) == cudaSuccess;
  if (!ok) {
    delete w;
    return FS_ECUDA;
  }
  *out = w;
  return FS_OK;
  FS_GUARD_END
}

int fs_window_forward(fs_window* w, const double* theta, double* loss) {
  FS_GUARD_BEGIN
  if (!w || !theta || !loss) return FS_EINVAL;
  return w->tsz == 8 ? do_forward<double>(w, theta, loss) : do_forward<float>(w, theta, loss);
  FS_GUARD_END
}

int fs_window_backward(fs_window* w, double dloss, double* grad) {
  FS_GUARD_BEGIN
  if (!w || !grad) return FS_EINVAL;
  return w->tsz == 8 ? do_backward<double>(w, dloss, grad) : do_backward<float>(w, dloss, grad);
  FS_GUARD_END
}

int fs_window_counts(fs_window* w, long long* out5) {
  FS_GUARD_BEGIN
  if (!w || !out5) return FS_EINVAL;
  for (int k = 0; k < 5; ++k) out5[k] = w->counts[k];
  return FS_OK;
  FS_GUARD_END
}

int fs_window_destroy(fs_window* w) {
  FS_GUARD_BEGIN
  if (!w) return FS_OK;
  if (w->side) {
    cudaStreamSynchronize(w->side);
    cudaStreamDestroy(w->side);
  }
  for (cudaEvent_t e : {w->taped, w->reversed})
    if (e) cudaEventDestroy(e);
  delete w;
  return FS_OK;
  FS_GUARD_END
}

}  // extern "C"
