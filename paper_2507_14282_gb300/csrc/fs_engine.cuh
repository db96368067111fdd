// fs_engine.cuh -- the hot-path kernels of one hybrid step, templated on the
// arithmetic type T (float or double) and the dimension DIM (1 or 2).
//
// Step n -> n+1 (Sec. 2 boundary inside a textbook hybrid PIC step):
//   k_push     persistent CTAs, each over a group of tiles of cells
//              (fs_push.cuh): CIC gather of E^n and Bbar^n from a
//              shared-memory field tile, Boris push, move, open far wall,
//              faux-shock pass/return (Eq. 1), in-tile counting sort by new
//              cell, CIC deposit of n and J by runs of sorted particles with a
//              warp team reduction into a shared-memory node tile, then
//              stayers written back to the tile's bucket and leavers to the
//              mover list. Deposit partials per tile, no global atomics
//              (except rare far movers).
//   k_inject_* thermal inflow at x = L and the cosmic-ray source at x = 0, drawn
//              into records (in the captured step, beside the push).
//   k_movers   leavers and new particles appended to their tile's bucket (in the
//              captured step, beside the next two, which read no bucket).
//   k_moments  sum of the per-tile partials in a fixed order, wall
//              half-volume correction, density floor, u = J / n
//              (k_moments_ct: the same with the 2D tile shape compiled in).
//   k_ohm / k_faraday  RK4 substeps of dB/dt = -curl E(B), E from Ohm's law.
//   k_ohm (final) also packs E and Bbar per node for the next gather.
//
// The FP64 instantiation is compiled without FMA contraction and evaluates
// every expression in the same order as the written scheme, so that it agrees
// bit for bit with an implementation of the same scheme on the CPU. Node sums
// of the FP64 deposit are int64 fixed point (2^-40), independent of order.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fs_device.cuh"
#include "fs_internal.h"

namespace fsx {

constexpr int kBlock = 256;

template <typename T>
struct Num;
template <>
struct Num<float> {
  using acc = float;
  static constexpr float offmax = 0x1.fffffep-1f;
  __device__ static float fl(float x) { return floorf(x); }
  __device__ static float ab(float x) { return fabsf(x); }
};
template <>
struct Num<double> {
  using acc = unsigned long long;  // int64 fixed point, two's complement
  static constexpr double offmax = 0x1.fffffffffffffp-1;
  __device__ static double fl(double x) { return floor(x); }
  __device__ static double ab(double x) { return fabs(x); }
};

// A deposit contribution c (already scaled by 2^40 for FP64) in accumulator
// form. FP64: c rounded to the nearest integer, ties to even (llrint(c)),
// worked out on the bit pattern with integer shifts: the value is
// mant * 2^(e - 1075); the bits shifted out decide the rounding. Exact for
// every double; it keeps the addition off GB300's narrow FP64 pipe.
__device__ __forceinline__ float to_acc(float c, int = 0) { return c; }
// (exp: of c 2^exp)
__device__ __forceinline__ unsigned long long to_acc(double c, int exp = 0) {
  const long long b = __double_as_longlong(c);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long mant = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
  const int sh = 1075 - exp - e;  // right shift of the 53-bit significand
  long long r;
  if (e == 0 || sh > 53) {
    r = 0;  // zero, subnormal, or |c| < 1/2
  } else if (sh <= 0) {
    r = mant << (-sh);  // already an integer (|c| >= 2^52; a shift of at most 10 here)
  } else {
    const long long q = mant >> sh;
    const long long rem = mant - (q << sh);
    const long long half = 1LL << (sh - 1);
    r = q + ((rem > half || (rem == half && (q & 1))) ? 1 : 0);
  }
  return (unsigned long long)(b < 0 ? -r : r);
}
// a * b in accumulator form. FP64: rounded once from the exact product to
// the nearest integer (fma with 1.5 * 2^52), as the written scheme states.
// (An all-integer version with the 106-bit product measured 3 % slower in the
// push: the fused multiply-add is worth its FP64 pipe slot here.)
// (magic: 1.5 * 2^(52 - exp), for the product times 2^exp)
__device__ __forceinline__ float to_acc_prod(float a, float b, float = 0.0f) { return a * b; }
__device__ __forceinline__ unsigned long long to_acc_prod(double a, double b,
                                                          double magic = 0x1.8p52) {
  const double m = __fma_rn(a, b, magic);
  return (unsigned long long)(__double_as_longlong(m) - __double_as_longlong(magic));
}
__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float rcpT(float a) { return __frcp_rn(a); }
__device__ __forceinline__ double rcpT(double a) { return __drcp_rn(a); }
__device__ __forceinline__ float sqrtT(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ double sqrtT(double a) { return __dsqrt_rn(a); }
// an accumulator's value in the run's precision: FP32 sums as they are (no
// round trip through FP64, whose conversions use GB300's narrow FP64 pipe),
// FP64 fixed point scaled back by 2^-40
__device__ __forceinline__ float acc_value(float a) { return a; }
__device__ __forceinline__ double acc_value(unsigned long long a) {
  return (double)(long long)a * 0x1p-40;
}

template <typename T>
__device__ __forceinline__ T deposit_weight_scale() {
  return (T)1;
}
template <>
__device__ __forceinline__ double deposit_weight_scale<double>() {
  return 0x1p40;
}

__device__ __forceinline__ void atomic_acc(float* a, float v) { atomicAdd(a, v); }
__device__ __forceinline__ void atomic_acc(unsigned long long* a,
                                           unsigned long long v) {
  atomicAdd(a, v);
}

__device__ __forceinline__ float shfl_up(float v, int o) {
  return __shfl_up_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ unsigned long long shfl_up(unsigned long long v,
                                                      int o) {
  return __shfl_up_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ float shfl_xor(float v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ unsigned long long shfl_xor(unsigned long long v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}

__device__ __forceinline__ int wrap(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

// Kinetic energy of a macroparticle of weight wp: wp v^2 / 2 (v stored), or
// for relativistic ions (u = gamma v stored, c2inv = 1/c^2 > 0)
// wp (gamma - 1) c^2 = wp u.u / (gamma + 1).
__device__ __forceinline__ double kinetic(double wp, double vx, double vy,
                                          double vz, double vol, double c2inv = 0.0) {
  if (c2inv > 0.0) {
    const double uu = __fma_rn(vz, vz, __fma_rn(vy, vy, __dmul_rn(vx, vx)));
    const double gamma = __dsqrt_rn(__dadd_rn(1.0, __dmul_rn(uu, c2inv)));
    return __dmul_rn(__dmul_rn(wp, __ddiv_rn(uu, __dadd_rn(gamma, 1.0))), vol);
  }
  return __dmul_rn(
      __dmul_rn(__dmul_rn(wp, 0.5),
                __dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)),
                          __dmul_rn(vz, vz))),
      vol);
}

// 1/gamma of a stored u = gamma v: 1 / sqrt(1 + u.u / c^2)
template <typename T>
__device__ __forceinline__ T inv_gamma_u(T ux, T uy, T uz, T c2inv) {
  const T uu = fmaT(uz, uz, fmaT(uy, uy, ux * ux));
  return (T)1 / sqrtT((T)1 + uu * c2inv);
}
// gamma of a velocity: 1 / sqrt(1 - v.v / c^2)
__device__ __forceinline__ double gamma_v(double vx, double vy, double vz, double c2inv) {
  const double vv = __fma_rn(vz, vz, __fma_rn(vy, vy, __dmul_rn(vx, vx)));
  return __ddiv_rn(1.0, __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(vv, c2inv))));
}
// the velocity of a stored state (u for relativistic ions, v otherwise)
template <typename T>
__device__ __forceinline__ void velocity_of(T ux, T uy, T uz, T c2inv, T& vx, T& vy, T& vz) {
  if (c2inv > (T)0) {
    const T ig = inv_gamma_u(ux, uy, uz, c2inv);
    vx = ux * ig;
    vy = uy * ig;
    vz = uz * ig;
  } else {
    vx = ux;
    vy = uy;
    vz = uz;
  }
}

// ------------------------------------------------------------------------
// Boris rotation, the written order: half kick, t = B dt/2,
// s = 2 t / (1 + t.t), v' = v- + v- x t, v+ = v- + v' x s (each component as
// two fused multiply-adds), half kick.
// ------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void boris(T& vx, T& vy, T& vz, const T E[3],
                                      const T B[3], T hdt, T c2inv = (T)0) {
  const T emx = hdt * E[0], emy = hdt * E[1], emz = hdt * E[2];
  const T vmx = vx + emx, vmy = vy + emy, vmz = vz + emz;
  // relativistic ions (u = gamma v stored): t = B dt / (2 gamma-), gamma-
  // from the half-kicked u
  T hg = hdt;
  if (c2inv > (T)0) {
    const T uu = fmaT(vmz, vmz, fmaT(vmy, vmy, vmx * vmx));
    hg = hdt / sqrtT((T)1 + uu * c2inv);
  }
  const T tx = hg * B[0], ty = hg * B[1], tz = hg * B[2];
  const T tt = fmaT(tz, tz, fmaT(ty, ty, tx * tx));
  // 2 / (1 + t.t) as 2 * (correctly rounded reciprocal): doubling is exact,
  // so this is the same number as the rounded quotient
  const T f = (T)2 * rcpT((T)1 + tt);
  const T sx = f * tx, sy = f * ty, sz = f * tz;
  const T px = fmaT(vmy, tz, fmaT(-vmz, ty, vmx));
  const T py = fmaT(vmz, tx, fmaT(-vmx, tz, vmy));
  const T pz = fmaT(vmx, ty, fmaT(-vmy, tx, vmz));
  const T qx = fmaT(py, sz, fmaT(-pz, sy, vmx));
  const T qy = fmaT(pz, sx, fmaT(-px, sz, vmy));
  const T qz = fmaT(px, sy, fmaT(-py, sx, vmz));
  vx = qx + emx;
  vy = qy + emy;
  vz = qz + emz;
}

// ------------------------------------------------------------------------
// Faux-shock decision (Sec. 2, Eq. 1) in FP64. Returns true and overwrites v
// when the particle is returned: P = ((1 - u2/v)/(1 + u2/v))^2 with v the
// speed in the chosen frame (0 when v <= u2); returned iff U0 < P and the
// downstream-frame speed |v'| = |v + u2 x| exceeds u2; the new direction has
// mu' = a + (1 - a) sqrt(U1), a = u2/|v'| (flux-weighted, isotropic in the
// downstream), azimuth 2 pi U2; |v'| is kept.
// ------------------------------------------------------------------------
__device__ __forceinline__ bool fs_return(double& vx, double& vy, double& vz,
                                          double u2, int frame,
                                          unsigned long long seed,
                                          uint32_t pid, long long step) {
  const double sp = __dsqrt_rn(__dadd_rn(
      __dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz)));
  const double wx = __dadd_rn(vx, u2);
  const double w = __dsqrt_rn(__dadd_rn(
      __dadd_rn(__dmul_rn(wx, wx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz)));
  const double vp = (frame == FS_FRAME_SHOCK) ? sp : w;
  double prob = 0.0;
  if (vp > u2) {
    const double a = __ddiv_rn(u2, vp);
    const double q = __ddiv_rn(__dsub_rn(1.0, a), __dadd_rn(1.0, a));
    prob = __dmul_rn(q, q);
  }
  const Philox4 r = draw4(seed, pid, step, kPurposeFS);
  const double U0 = u01(r.x[0]), U1 = u01(r.x[1]), U2 = u01(r.x[2]);
  if (!(U0 < prob && w > u2)) return false;
  const double a = __ddiv_rn(u2, w);
  const double mu = __dadd_rn(a, __dmul_rn(__dsub_rn(1.0, a), __dsqrt_rn(U1)));
  const double sn = __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(mu, mu)));
  double c, s;
  fs_sincos2pi(U2, &c, &s);
  const double ws = __dmul_rn(w, sn);
  vx = __dsub_rn(__dmul_rn(w, mu), u2);
  vy = __dmul_rn(ws, c);
  vz = __dmul_rn(ws, s);
  return true;
}

// ------------------------------------------------------------------------
// k_movers: append each leaver to its destination tile's bucket.
// ------------------------------------------------------------------------
// Block blk of nblk: one warp per source tile, its leavers go to their
// destination tiles.
// One leaver record of the mover list.
template <typename T>
struct MoverRec {
  int cell;
  T ox, oy, vx, vy, vz;
  uint32_t id;
};
template <typename T, int DIM>
__device__ __forceinline__ MoverRec<T> mover_load(const DevPtrs<T>& d, bool act, int src) {
  MoverRec<T> r;
  r.cell = act ? d.M.cell[src] : 0;
  r.ox = act ? d.M.ox[src] : (T)0;
  r.oy = (DIM == 2 && act) ? d.M.oy[src] : (T)0;
  r.vx = act ? d.M.vx[src] : (T)0;
  r.vy = act ? d.M.vy[src] : (T)0;
  r.vz = act ? d.M.vz[src] : (T)0;
  r.id = act ? d.M.id[src] : 0u;
  return r;
}
// destination tile of an active record (-1: none)
template <typename T>
__device__ __forceinline__ int mover_dest(const Geo& g, bool act, const MoverRec<T>& r) {
  const int i = r.cell & 0xFFFF, j = r.cell >> 16;
  return act ? (j / g.TY) * g.ntx + i / g.TX : -1;
}
template <typename T, int DIM>
__device__ __forceinline__ void mover_store(const DevPtrs<T>& d, const Geo& g, int out, bool act,
                                            int dt, int slot, const MoverRec<T>& r) {
  if (!act) return;
  if (slot >= g.tile_cap) {
    atomicSub(&d.cnt[out][dt], 1);
    atomicOr(&d.ctr->status, kStatusCapacity);
    return;
  }
  const Parts<T> PO = d.P[out];
  const int gi = dt * g.tile_cap + slot;  // a tile's bucket starts at tile x capacity
  PO.cell[gi] = r.cell;
  PO.ox[gi] = r.ox;
  if (DIM == 2) PO.oy[gi] = r.oy;
  PO.vx[gi] = r.vx;
  PO.vy[gi] = r.vy;
  PO.vz[gi] = r.vz;
  PO.id[gi] = r.id;
}

// Block blk of nblk: one warp per source tile, its leavers go to their
// destination tiles; each warp works on two source tiles at a time (their
// loads and slot atomics in flight together). Lanes bound for the same tile
// take consecutive slots after one atomic by the lowest of them.
template <typename T, int DIM>
__device__ __forceinline__ void movers_body(const DevPtrs<T>& d, const Geo& g, int out, int blk,
                                            int nblk) {
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  const int stride = nblk * wpb;
  const unsigned below = (1u << lane) - 1u;
  for (int t = blk * wpb + (threadIdx.x >> 5); t < g.ntiles; t += 2 * stride) {
    const int t2 = t + stride;
    const int nm1 = d.mcnt[t];
    const int nm2 = t2 < g.ntiles ? d.mcnt[t2] : 0;
    const int mb1 = t * g.mover_per_tile, mb2 = t2 * g.mover_per_tile;
    for (int k0 = 0; k0 < nm1 || k0 < nm2; k0 += 32) {  // counts are warp-uniform
      const int k = k0 + lane;
      const bool a1 = k < nm1, a2 = k < nm2;
      const MoverRec<T> r1 = mover_load<T, DIM>(d, a1, mb1 + k);
      const MoverRec<T> r2 = mover_load<T, DIM>(d, a2, mb2 + k);
      const int dt1 = mover_dest(g, a1, r1), dt2 = mover_dest(g, a2, r2);
      const unsigned p1 = __match_any_sync(0xffffffffu, dt1);
      const unsigned p2 = __match_any_sync(0xffffffffu, dt2);
      const int l1 = __ffs(p1) - 1, l2 = __ffs(p2) - 1;
      int b1 = 0, b2 = 0;
      if (a1 && lane == l1) b1 = atomicAdd(&d.cnt[out][dt1], __popc(p1));
      if (a2 && lane == l2) b2 = atomicAdd(&d.cnt[out][dt2], __popc(p2));
      b1 = __shfl_sync(0xffffffffu, b1, l1);
      b2 = __shfl_sync(0xffffffffu, b2, l2);
      mover_store<T, DIM>(d, g, out, a1, dt1, b1 + __popc(p1 & below), r1);
      mover_store<T, DIM>(d, g, out, a2, dt2, b2 + __popc(p2 & below), r2);
    }
  }
}

// The step's new particles (drawn by inject_draw into d.I, cell -1: none) into
// their tiles' buckets.
template <typename T, int DIM>
__device__ __forceinline__ void place_injected(const DevPtrs<T>& d, const Geo& g, int out, int blk,
                                               int nblk) {
  const Parts<T> I = d.I;
  for (int k = blk * blockDim.x + threadIdx.x; k < g.ninj; k += nblk * blockDim.x) {
    const int cell = I.cell[k];
    if (cell < 0) continue;
    const MoverRec<T> r{cell, I.ox[k], DIM == 2 ? I.oy[k] : (T)0, I.vx[k], I.vy[k], I.vz[k],
                        I.id[k]};
    const int dt = mover_dest(g, true, r);
    mover_store<T, DIM>(d, g, out, true, dt, atomicAdd(&d.cnt[out][dt], 1), r);
  }
}

// what: 1 the leavers of every tile, 2 the injected particles, 3 both
template <typename T, int DIM>
__global__ void k_movers(DevPtrs<T> d, Geo g, int out, int what) {
  if (what & 1) movers_body<T, DIM>(d, g, out, blockIdx.x, gridDim.x);
  if (what & 2) place_injected<T, DIM>(d, g, out, blockIdx.x, gridDim.x);
}

// Deposit of one particle into the far accumulators (global atomics).
template <typename T, int DIM>
__device__ __forceinline__ void deposit_far(const DevPtrs<T>& d, const Geo& g,
                                            int i, int j, T fx, T fy, T wp,
                                            T vx, T vy, T vz) {
  using A = typename Num<T>::acc;
  A* far = (A*)d.far;
  const size_t nn = (size_t)g.nxn * g.ny;
  const int i1 = (g.bc_x == FS_BC_PERIODIC && i + 1 == g.nx) ? 0 : i + 1;
  if (DIM == 1) {
    const T c0 = wp * ((T)1 - fx), c1 = wp * fx;
    atomic_acc(&far[0 * nn + i], to_acc(c0));
    atomic_acc(&far[1 * nn + i], to_acc_prod(c0, vx));
    atomic_acc(&far[2 * nn + i], to_acc_prod(c0, vy));
    atomic_acc(&far[3 * nn + i], to_acc_prod(c0, vz));
    atomic_acc(&far[0 * nn + i1], to_acc(c1));
    atomic_acc(&far[1 * nn + i1], to_acc_prod(c1, vx));
    atomic_acc(&far[2 * nn + i1], to_acc_prod(c1, vy));
    atomic_acc(&far[3 * nn + i1], to_acc_prod(c1, vz));
  } else {
    const int j1 = (j + 1 == g.ny) ? 0 : j + 1;
    const T gx0 = (T)1 - fx, gy0 = (T)1 - fy;
    const int nd[4] = {j * g.nxn + i, j * g.nxn + i1, j1 * g.nxn + i,
                       j1 * g.nxn + i1};
    const T cw[4] = {wp * (gx0 * gy0), wp * (fx * gy0), wp * (gx0 * fy),
                     wp * (fx * fy)};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      atomic_acc(&far[0 * nn + nd[c]], to_acc(cw[c]));
      atomic_acc(&far[1 * nn + nd[c]], to_acc_prod(cw[c], vx));
      atomic_acc(&far[2 * nn + nd[c]], to_acc_prod(cw[c], vy));
      atomic_acc(&far[3 * nn + nd[c]], to_acc_prod(cw[c], vz));
    }
  }
}

// One new particle as record k of d.I (placed into its tile's bucket after the
// push, place_injected), deposited into the far accumulators now.
template <typename T, int DIM>
__device__ __forceinline__ void record_new(const DevPtrs<T>& d, const Geo& g, const Phys& ph,
                                           int k, int i, int j, T fx, T fy, T vx, T vy, T vz,
                                           uint32_t id) {
  const Parts<T> I = d.I;
  I.cell[k] = (j << 16) | i;
  I.ox[k] = fx;
  if (DIM == 2) I.oy[k] = fy;
  I.vx[k] = vx;
  I.vy[k] = vy;
  I.vz[k] = vz;
  I.id[k] = id;
  const double ws = deposit_weight_scale<T>();
  const T wp = (T)(((id & kIdCR) ? ph.w_cr : ph.w_th) * ws);
  T dvx, dvy, dvz;  // the current uses the velocity
  velocity_of<T>(vx, vy, vz, (T)ph.c2inv, dvx, dvy, dvz);
  deposit_far<T, DIM>(d, g, i, j, fx, fy, wp, dvx, dvy, dvz);
}

// ------------------------------------------------------------------------
// Injection (Sec. 2). k_inject_count (one CTA): per transverse row the
// accumulator advances by ppc u_sh dt/dx, its integer part is this step's
// count; a scan over rows gives each row's first id. k_inject_draw: one thread
// per (row, slot, species) draws the particle into its record and deposits it.
// The draws need nothing of the step's push (a long chain of FP64 operations:
// 17 us, 35 us for both species in one thread), so the captured step runs
// them beside it; k_movers puts the records into the buckets.
// ------------------------------------------------------------------------
// The whole block (any multiple of 32 threads up to 1024) counts every row.
__device__ __forceinline__ void inject_count_body(double* acc, int* rowcnt, int* rowoff, int ny,
                                                  double rate, int per_row_mult) {
  __shared__ int wsum[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int b = 0; b < ny; b += blockDim.x) {
    const int j = b + threadIdx.x;
    int n = 0;
    if (j < ny) {
      double v = __dadd_rn(acc[j], rate);
      const double fl = floor(v);
      n = (int)fl;
      acc[j] = __dsub_rn(v, fl);
      rowcnt[j] = n;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int inc = n * per_row_mult;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
      int s = (lane < (int)(blockDim.x >> 5)) ? wsum[lane] : 0;
      int si = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, si, o);
        if (lane >= o) si += v;
      }
      if (lane < (int)(blockDim.x >> 5)) wsum[lane] = si - s;
    }
    __syncthreads();
    if (j < ny) rowoff[j] = carry + wsum[w] + inc - n * per_row_mult;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry += wsum[w] + inc;
    __syncthreads();
  }
  if (threadIdx.x == 0) rowoff[ny] = carry;
}

static __global__ void k_inject_count(double* acc, int* rowcnt, int* rowoff, int ny,
                                      double rate, int per_row_mult) {
  inject_count_body(acc, rowcnt, rowoff, ny, rate, per_row_mult);
}

// New particle k of row j of one species (cr: a cosmic ray at x = 0, else
// thermal at x = L) into record rec (cell -1 when the row has fewer), ids from
// `first` (next_id before this step's injection) in (row, thermal, cosmic ray)
// order; counts and energy added to the caller's l_inj, l_e.
template <typename T, int DIM>
__device__ __forceinline__ void inject_draw(const DevPtrs<T>& d, const Geo& g, const Phys& ph,
                                            const int* rowcnt, const int* rowoff, int j, int k,
                                            bool cr, int rec, unsigned long long first,
                                            long long step, long long& l_inj, double& l_e) {
  const int n = rowcnt[j], nx = g.nx;
  const unsigned long long num = first + rowoff[j] + k + (cr && ph.inject_thermal ? n : 0);
  if (k >= n || num > kIdMask) {
    if (k < n) atomicOr(&d.ctr->status, kStatusIdOverflow);
    d.I.cell[rec] = -1;
    return;
  }
  const uint32_t pid = (uint32_t)num;
  double vx, vy, vz, X, fy;
  if (!cr) {
    const Philox4 ra = draw4(ph.seed, pid, step, kPurposeInjA);
    const Philox4 rb = draw4(ph.seed, pid, step, kPurposeInjB);
    double g0, g1, g2, g3;
    gauss2(u01(ra.x[0]), u01(ra.x[1]), &g0, &g1);
    gauss2(u01(ra.x[2]), u01(ra.x[3]), &g2, &g3);
    vx = __dsub_rn(__dmul_rn(ph.vth, g0), ph.mach_a);
    vy = __dmul_rn(ph.vth, g1);
    vz = __dmul_rn(ph.vth, g2);
    X = __dsub_rn((double)nx, __dmul_rn(__dmul_rn(u01(rb.x[0]), fabs(vx)), ph.dtdx));
    fy = u01(rb.x[1]);
  } else {
    const Philox4 rc = draw4(ph.seed, pid, step, kPurposeInjCR);
    // speed p_iso / gamma(p_iso) in the downstream frame (p_iso without c)
    const double a = __ddiv_rn(ph.u_cr, ph.p_iso_v);
    const double mu = __dadd_rn(a, __dmul_rn(__dsub_rn(1.0, a), __dsqrt_rn(u01(rc.x[0]))));
    const double sn = __dsqrt_rn(__dsub_rn(1.0, __dmul_rn(mu, mu)));
    double c, s;
    fs_sincos2pi(u01(rc.x[1]), &c, &s);
    const double ws = __dmul_rn(ph.p_iso_v, sn);
    vx = __dsub_rn(__dmul_rn(ph.p_iso_v, mu), ph.u_cr);
    vy = __dmul_rn(ws, c);
    vz = __dmul_rn(ws, s);
    X = __dmul_rn(__dmul_rn(u01(rc.x[2]), vx), ph.dtdx);
    fy = u01(rc.x[3]);
  }
  const double ix = floor(X);
  int i = (int)ix;
  double fx = __dsub_rn(X, ix);
  if (i >= nx) { i = nx - 1; fx = Num<double>::offmax; }
  if (i < 0) { i = 0; fx = 0.0; }
  if (fx >= 1.0) fx = Num<double>::offmax;
  T ft = (T)fx;
  if (ft >= (T)1) ft = Num<T>::offmax;
  T fyt = (DIM == 2) ? (T)fy : (T)0;
  if (fyt >= (T)1) fyt = Num<T>::offmax;
  if (ph.c2inv > 0.0) {  // stored as u = gamma v
    const double gv = gamma_v(vx, vy, vz, ph.c2inv);
    vx = __dmul_rn(vx, gv); vy = __dmul_rn(vy, gv); vz = __dmul_rn(vz, gv);
  }
  record_new<T, DIM>(d, g, ph, rec, i, j, ft, fyt, (T)vx, (T)vy, (T)vz, cr ? pid | kIdCR : pid);
  ++l_inj;
  l_e = __dadd_rn(l_e, kinetic(cr ? ph.w_cr : ph.w_th, vx, vy, vz, ph.cellvol, ph.c2inv));
}

// Draws of thread `id` of `nthreads`: record rec = (row j, slot k, species)
template <typename T, int DIM>
__device__ __forceinline__ void inject_draws(const DevPtrs<T>& d, const Geo& g, const Phys& ph,
                                             int id, int nthreads) {
  const long long step = d.ctr->step;
  const unsigned long long first = d.ctr->next_id;
  const int* rowcnt = d.inj;
  const int* rowoff = rowcnt + g.ny;
  const int both = ph.inject_thermal && ph.cr_enable;
  const int per = g.ninj / g.ny, maxk = both ? per / 2 : per;
  long long l_inj = 0;
  double l_e = 0.0;
  for (int r = id; r < g.ninj; r += nthreads) {
    const int j = r / per, q = r - j * per;
    const bool cr = both ? q >= maxk : !ph.inject_thermal;
    inject_draw<T, DIM>(d, g, ph, rowcnt, rowoff, j, both && cr ? q - maxk : q, cr, r, first, step,
                        l_inj, l_e);
  }
  if (l_inj) {
    atomicAdd(&d.ctr->injected, (unsigned long long)l_inj);
    atomicAdd(&d.ctr->injected_energy, l_e);
  }
}

template <typename T, int DIM>
__global__ void __launch_bounds__(64) k_inject_draw(DevPtrs<T> d, Geo g, Phys ph) {
  inject_draws<T, DIM>(d, g, ph, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// The row counts and the draws of one run by one block.
template <typename T, int DIM>
__device__ __forceinline__ void inject_run_block(const DevPtrs<T>& d, const Geo& g,
                                                 const Phys& ph) {
  inject_count_body(d.acc, d.inj, d.inj + g.ny, g.ny, ph.rate,
                    (ph.inject_thermal ? 1 : 0) + (ph.cr_enable ? 1 : 0));
  __syncthreads();
  inject_draws<T, DIM>(d, g, ph, threadIdx.x, blockDim.x);
}
template <typename T, int DIM>
__global__ void __launch_bounds__(kBlock) k_inject_run(DevPtrs<T> d, Geo g, Phys ph) {
  inject_run_block<T, DIM>(d, g, ph);
}

// end of a step: advance the device step counter and next_id (past the step's
// injected particles)
__device__ __forceinline__ void step_end(Counters* ctr, const int* inj, const Geo& g) {
  ctr->step += 1;
  if (g.ninj) ctr->next_id += inj[2 * g.ny];
}
static __global__ void k_step_end(Counters* ctr, const int* inj, Geo g) {
  if (threadIdx.x == 0 && blockIdx.x == 0) step_end(ctr, inj, g);
}

// ------------------------------------------------------------------------
// k_moments: per node, the deposit partials of every tile whose accumulator
// covers it (tiles in increasing row, then column order; within a tile every
// accumulator slot that maps to the node), plus the far accumulator; then the
// wall half-volume correction (x2 at i = 0 and i = nx in the faux-shock box),
// the density floor and u = J / n.
// ------------------------------------------------------------------------
// The node's moments from its sums s (n, Jx, Jy, Jz); clears its far sums.
template <typename T, int DIM>
__device__ __forceinline__ void moments_finish(const DevPtrs<T>& d, const Geo& g, const Phys& ph,
                                               int q, int i, const typename Num<T>::acc (&s)[4]) {
  using A = typename Num<T>::acc;
  const int nn = g.nxn * g.ny;
  T nt = acc_value(s[0]), jxt = acc_value(s[1]), jyt = acc_value(s[2]), jzt = acc_value(s[3]);
  if (g.bc_x == FS_BC_FAUXSHOCK && (i == 0 || i == g.nx)) {
    nt = nt * (T)2; jxt = jxt * (T)2; jyt = jyt * (T)2; jzt = jzt * (T)2;
  }
  d.J[q] = jxt;
  d.J[(size_t)nn + q] = jyt;
  d.J[(size_t)2 * nn + q] = jzt;
  const T nf = (T)ph.n_floor;
  if (nt < nf) nt = nf;
  d.n[q] = nt;
  d.u[q] = jxt / nt;
  d.u[(size_t)nn + q] = jyt / nt;
  d.u[(size_t)2 * nn + q] = jzt / nt;
  A* farw = (A*)d.far;
#pragma unroll
  for (int c = 0; c < 4; ++c) farw[(size_t)c * nn + q] = (A)0;
}

template <typename T, int DIM>
__device__ __forceinline__ void moments_body(const DevPtrs<T>& d, const Geo& g, const Phys& ph,
                                             int blk, int nblk) {
  using A = typename Num<T>::acc;
  const int nn = g.nxn * g.ny;
  const int AX = g.TX + 3, AY = (DIM == 2) ? g.TY + 3 : 1, NA = AX * AY;
  for (int q = blk * blockDim.x + threadIdx.x; q < nn; q += nblk * blockDim.x) {
    const int i = q % g.nxn, j = q / g.nxn;
    // candidate tile columns / rows (distinct): a tile's accumulator spans
    // nodes i0 - 1 .. i0 + TX + 1, so tiles home - 2 .. home + 1 can cover i
    int tcx[4], ncx = 0, tcy[4], ncy = 0;
    {
      const int home = min(i / g.TX, g.ntx - 1);
      for (int dd = -2; dd <= 1; ++dd) {
        int c = home + dd;
        if (g.bc_x == FS_BC_PERIODIC) c = wrap(c, g.ntx);
        else if (c < 0 || c >= g.ntx) continue;
        bool dup = false;
        for (int k = 0; k < ncx; ++k) dup |= (tcx[k] == c);
        if (!dup) tcx[ncx++] = c;
      }
    }
    if (DIM == 2) {
      const int home = j / g.TY;
      for (int dd = -2; dd <= 1; ++dd) {
        const int c = wrap(home + dd, g.nty);
        bool dup = false;
        for (int k = 0; k < ncy; ++k) dup |= (tcy[k] == c);
        if (!dup) tcy[ncy++] = c;
      }
    } else {
      tcy[0] = 0;
      ncy = 1;
    }
    // sort candidates ascending (fixed summation order)
    for (int a = 0; a < ncx; ++a)
      for (int b = a + 1; b < ncx; ++b)
        if (tcx[b] < tcx[a]) { int t = tcx[a]; tcx[a] = tcx[b]; tcx[b] = t; }
    for (int a = 0; a < ncy; ++a)
      for (int b = a + 1; b < ncy; ++b)
        if (tcy[b] < tcy[a]) { int t = tcy[a]; tcy[a] = tcy[b]; tcy[b] = t; }
    A s[4];
    const A* far = (const A*)d.far;
#pragma unroll
    for (int c = 0; c < 4; ++c) s[c] = far[(size_t)c * nn + q];
    for (int yy = 0; yy < ncy; ++yy) {
      const int ty = tcy[yy];
      // accumulator rows of node row j (more than one only when the box is
      // narrower than a tile's accumulator)
      int ay0 = 0;
      if (DIM == 2) ay0 = wrap(j - (ty * g.TY - 1), g.ny);
      for (int ay = ay0; ay < AY; ay += (DIM == 2 ? g.ny : AY)) {
        for (int xx = 0; xx < ncx; ++xx) {
          const int tx = tcx[xx];
          const int t = ty * g.ntx + tx;
          const A* part = (const A*)d.partial + (size_t)t * 4 * NA;
          int ax0 = i - (tx * g.TX - 1);
          int step = AX;
          if (g.bc_x == FS_BC_PERIODIC) {
            ax0 = wrap(ax0, g.nx);
            step = g.nx;
          }
          for (int ax = ax0; ax >= 0 && ax < AX; ax += step) {
            const int k = ax + ay * AX;
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] += part[c * NA + k];
          }
        }
      }
    }
    moments_finish<T, DIM>(d, g, ph, q, i, s);
  }
}

template <typename T, int DIM>
__global__ void k_moments(DevPtrs<T> d, Geo g, Phys ph) {
  moments_body<T, DIM>(d, g, ph, blockIdx.x, gridDim.x);
}

// The same sums for a 2D box with x walls (whose rows hold more than one tile's
// accumulator rows and more tile rows than cover a node): the candidate tiles
// of a node are a fixed, small set (MX columns by MY rows), so every load is
// issued without a data-dependent loop; rows are taken in increasing wrapped
// order, columns in increasing order, as in moments_body. The tile shape is
// compiled in (TXC x TYC) or the run's (0). Bound by the loads in flight:
// 3000 x 250 cells, FP32, 39 -> 25 us against moments_body's loops.
template <typename T, int TXC, int TYC, int MX, int MY>
__global__ void k_moments_ct(DevPtrs<T> d, Geo g, Phys ph) {
  using A = typename Num<T>::acc;
  const int TX = TXC ? TXC : g.TX, TY = TYC ? TYC : g.TY;
  const int AX = TX + 3, AY = TY + 3, NA = AX * AY;
  const int nn = g.nxn * g.ny;
  const A* far = (const A*)d.far;
  const A* partial = (const A*)d.partial;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += gridDim.x * blockDim.x) {
    const int i = q % g.nxn, j = q / g.nxn;
    // candidate rows: ty with 0 <= j - (ty TY - 1) < AY, wrapped, ascending
    int tyw[MY], ayv[MY];
    const int tyh = (j + 1) / TY;
#pragma unroll
    for (int u = 0; u < MY; ++u) {
      const int ty = tyh - (MY - 1) + u;
      const int ay = j - (ty * TY - 1);
      const bool ok = ay >= 0 && ay < AY;
      tyw[u] = ok ? (ty < 0 ? ty + g.nty : (ty >= g.nty ? ty - g.nty : ty)) : 0x7fffffff;
      ayv[u] = ay;
    }
#pragma unroll
    for (int a = 0; a < MY; ++a)
#pragma unroll
      for (int b = a + 1; b < MY; ++b)
        if (tyw[b] < tyw[a]) {
          const int t0 = tyw[a], t1 = ayv[a];
          tyw[a] = tyw[b]; ayv[a] = ayv[b];
          tyw[b] = t0; ayv[b] = t1;
        }
    A s[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) s[c] = far[(size_t)c * nn + q];
    const int txh = (i + 1) / TX;
#pragma unroll
    for (int u = 0; u < MY; ++u) {
      if (tyw[u] == 0x7fffffff) continue;
#pragma unroll
      for (int x = 0; x < MX; ++x) {
        const int tx = txh - (MX - 1) + x;
        const int ax = i - (tx * TX - 1);
        if (tx < 0 || tx >= g.ntx || ax < 0 || ax >= AX) continue;
        const A* part = partial + (size_t)(tyw[u] * g.ntx + tx) * 4 * NA + ax + ayv[u] * AX;
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] += part[c * NA];
      }
    }
    moments_finish<T, 2>(d, g, ph, q, i, s);
  }
}

// ------------------------------------------------------------------------
// Ohm's law at the nodes (massless isothermal electrons, J = curl B), the
// cross products and the 1/n scaling written as fused multiply-adds:
//   E = ((curl B - j_ext x) x Bbar)/n - u x Bbar - T_e grad n / n (+ eta curl B)
// Bbar is B averaged onto the nodes; derivatives are two-point differences
// averaged across the transverse direction; x walls use zero-gradient ghost
// cells (and a mirrored density gradient), periodic boxes wrap.
// With G != nullptr also packs (E, Bbar) per node, plus a ghost row ny
// (copy of row 0) and, in a periodic box, a ghost column nx (copy of 0).
// With pre != nullptr the density terms come from k_ohm_pre (same values).
// ------------------------------------------------------------------------
// The density terms of Ohm's law at node (i, j), fixed while n is: 1/n and
// the pressure terms -(T_e dn/dx), -(T_e dn/dy) (two-point differences, a
// mirrored density gradient at the x walls, periodic wrap).
template <typename T, int DIM>
__device__ __forceinline__ void density_terms(const T* __restrict__ nN, int i, int j,
                                              const Geo& g, const Phys& ph, T& inv_n,
                                              T& pgx, T& pgy) {
  const int nx = g.nx, ny = g.ny, nxn = g.nxn;
  const bool per = (g.bc_x == FS_BC_PERIODIC);
  const T te = (T)ph.te;
  auto nxo = [&](int c) {
    if (per) return wrap(c, nx);
    if (c < 0) return -c;
    if (c > nx) return 2 * nx - c;
    return c;
  };
  T dnx, dny;
  if (DIM == 1) {
    dnx = (nN[nxo(i + 1)] - nN[nxo(i - 1)]) * (T)ph.hdx;
    dny = (T)0;
  } else {
    dnx = (nN[j * nxn + nxo(i + 1)] - nN[j * nxn + nxo(i - 1)]) * (T)ph.hdx;
    dny = (nN[wrap(j + 1, ny) * nxn + i] - nN[wrap(j - 1, ny) * nxn + i]) * (T)ph.hdy;
  }
  inv_n = (T)1 / nN[j * nxn + i];
  pgx = -(te * dnx);
  pgy = -(te * dny);
}

// Writes density_terms for every node once per step (n is fixed during the
// field substeps): pre = [1/n][-(T_e dn/dx)][-(T_e dn/dy)] planes.
template <typename T, int DIM>
__global__ void k_ohm_pre(const T* __restrict__ nN, T* __restrict__ pre, Geo g, Phys ph) {
  const int nxn = g.nxn;
  const int nn = nxn * g.ny;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += gridDim.x * blockDim.x) {
    const int i = q % nxn, j = q / nxn;
    T inv_n, pgx, pgy;
    density_terms<T, DIM>(nN, i, j, g, ph, inv_n, pgx, pgy);
    pre[q] = inv_n;
    pre[nn + q] = pgx;
    pre[2 * nn + q] = pgy;
  }
}

// The node value of Ohm's law from curl B (cxv, cyv, czv), Bbar, 1/n, the
// pressure terms and u.
template <typename T>
__device__ __forceinline__ void ohm_e(T cxv, T cyv, T czv, T bbx, T bby, T bbz, T inv_n, T pgx,
                                      T pgy, T ux, T uy, T uz, T jcr, T eta, bool resist,
                                      T& ex, T& ey, T& ez) {
  const T ax = cxv - jcr, ay = cyv, az = czv;
  const T cax = fmaT(ay, bbz, -(az * bby));
  const T cay = fmaT(az, bbx, -(ax * bbz));
  const T caz = fmaT(ax, bby, -(ay * bbx));
  const T cux = fmaT(uy, bbz, -(uz * bby));
  const T cuy = fmaT(uz, bbx, -(ux * bbz));
  const T cuz = fmaT(ux, bby, -(uy * bbx));
  ex = fmaT(pgx, inv_n, fmaT(cax, inv_n, -cux));
  ey = fmaT(pgy, inv_n, fmaT(cay, inv_n, -cuy));
  ez = fmaT(caz, inv_n, -cuz);
  if (resist) {
    ex = ex + eta * cxv;
    ey = ey + eta * cyv;
    ez = ez + eta * czv;
  }
}

// The RK4 stage update of one B component from K = -curl E:
//   stage 1: Bsum = K;            Bs = B + (h/2) K
//   stage 2: Bsum = Bsum + 2 K;   Bs = B + (h/2) K
//   stage 3: Bsum = Bsum + 2 K;   Bs = B + h K
//   stage 4: Bsum = Bsum + K;     B  = B + (h/6) Bsum
template <typename T>
__device__ __forceinline__ void rk4_stage(int stage, T K, T& bsum, T& bs, T& b, T h, T hh,
                                          T h6) {
  if (stage == 1) {
    bsum = K;
    bs = fmaT(hh, K, b);
  } else if (stage == 2) {
    bsum = fmaT((T)2, K, bsum);
    bs = fmaT(hh, K, b);
  } else if (stage == 3) {
    bsum = fmaT((T)2, K, bsum);
    bs = fmaT(h, K, b);
  } else {
    const T sum = bsum + K;
    b = fmaT(h6, sum, b);
  }
}

// Ohm's law at node q = j * nxn + i (the body of k_ohm).
template <typename T, int DIM>
__device__ __forceinline__ void ohm_node(int q, const T* Bc, const T* nN, const T* uN,
                                         const T* pre, T* Eo, T* Bbo, T* G, const Geo& g,
                                         const Phys& ph, T* preo = nullptr) {
  const int nx = g.nx, ny = g.ny, nxn = g.nxn;
  const int nc = nx * ny, nn = nxn * ny;
  const T hdx = (T)ph.hdx, hdy = (T)ph.hdy, idx = (T)ph.idx;
  const T jcr = (T)ph.jcr, eta = (T)ph.eta;
  const bool per = (g.bc_x == FS_BC_PERIODIC);
  {
    const int i = q % nxn, j = q / nxn;
    auto cxo = [&](int c) { return per ? wrap(c, nx) : min(max(c, 0), nx - 1); };
    T bbx, bby, bbz, cxv, cyv, czv;
    if (DIM == 1) {
      const int im = cxo(i - 1), ip = cxo(i);
      const T bmx = Bc[im], bpx = Bc[ip];
      const T bmy = Bc[nc + im], bpy = Bc[nc + ip];
      const T bmz = Bc[2 * nc + im], bpz = Bc[2 * nc + ip];
      bbx = (T)0.5 * (bmx + bpx);
      bby = (T)0.5 * (bmy + bpy);
      bbz = (T)0.5 * (bmz + bpz);
      const T dby = (bpy - bmy) * idx;
      const T dbz = (bpz - bmz) * idx;
      cxv = (T)0;
      cyv = -dbz;
      czv = dby;
    } else {
      const int im = cxo(i - 1), ip = cxo(i);
      const int jm = wrap(j - 1, ny), jp = j;
      const int cmm = jm * nx + im, cpm = jm * nx + ip;
      const int cmp = jp * nx + im, cpp = jp * nx + ip;
      T b[3][4];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        b[c][0] = Bc[c * nc + cmm];
        b[c][1] = Bc[c * nc + cpm];
        b[c][2] = Bc[c * nc + cmp];
        b[c][3] = Bc[c * nc + cpp];
      }
      bbx = (T)0.25 * ((b[0][0] + b[0][1]) + (b[0][2] + b[0][3]));
      bby = (T)0.25 * ((b[1][0] + b[1][1]) + (b[1][2] + b[1][3]));
      bbz = (T)0.25 * ((b[2][0] + b[2][1]) + (b[2][2] + b[2][3]));
      const T dxby = ((b[1][3] + b[1][1]) - (b[1][2] + b[1][0])) * hdx;
      const T dxbz = ((b[2][3] + b[2][1]) - (b[2][2] + b[2][0])) * hdx;
      const T dybx = ((b[0][3] + b[0][2]) - (b[0][1] + b[0][0])) * hdy;
      const T dybz = ((b[2][3] + b[2][2]) - (b[2][1] + b[2][0])) * hdy;
      cxv = dybz;
      cyv = -dxbz;
      czv = dxby - dybx;
    }
    T inv_n, pgx, pgy;
    if (pre) {
      inv_n = pre[q];
      pgx = pre[nn + q];
      pgy = pre[2 * nn + q];
    } else {
      density_terms<T, DIM>(nN, i, j, g, ph, inv_n, pgx, pgy);
      if (preo) {
        preo[q] = inv_n;
        preo[nn + q] = pgx;
        preo[2 * nn + q] = pgy;
      }
    }
    T ex, ey, ez;
    ohm_e<T>(cxv, cyv, czv, bbx, bby, bbz, inv_n, pgx, pgy, uN[q], uN[nn + q], uN[2 * nn + q],
             jcr, eta, ph.eta != 0.0, ex, ey, ez);
    Eo[q] = ex;
    Eo[nn + q] = ey;
    Eo[2 * nn + q] = ez;
    if (Bbo) {
      Bbo[q] = bbx;
      Bbo[nn + q] = bby;
      Bbo[2 * nn + q] = bbz;
    }
    if (G) {
      const T v[8] = {ex, ey, ez, bbx, bby, bbz, (T)0, (T)0};
      const int gx = nx + 1;
      auto put = [&](int gi, int gj) {
        T* dst = G + ((size_t)gj * gx + gi) * 8;
#pragma unroll
        for (int c = 0; c < 8; ++c) dst[c] = v[c];
      };
      put(i, j);
      if (j == 0) put(i, ny);
      if (per && i == 0) {
        put(nx, j);
        if (j == 0) put(nx, ny);
      }
    }
  }
}

template <typename T, int DIM>
__global__ void k_ohm(const T* __restrict__ Bc, const T* __restrict__ nN,
                      const T* __restrict__ uN, const T* __restrict__ pre,
                      T* __restrict__ Eo, T* __restrict__ Bbo, T* __restrict__ G, Geo g,
                      Phys ph) {
  const int nn = g.nxn * g.ny;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += gridDim.x * blockDim.x)
    ohm_node<T, DIM>(q, Bc, nN, uN, pre, Eo, Bbo, G, g, ph);
}

// Faraday at centre c = j * nx + i, K = -curl E from the four corner nodes
// (two in 1D), and the RK4 stage update (rk4_stage): the body of k_faraday.
template <typename T, int DIM>
__device__ __forceinline__ void faraday_cell(int c, const T* En, T* B, T* Bs, T* Bsum,
                                             int stage, const Geo& g, const Phys& ph) {
  const int nx = g.nx, ny = g.ny, nxn = g.nxn;
  const int nc = nx * ny, nn = nxn * ny;
  const T hdx = (T)ph.hdx, hdy = (T)ph.hdy, idx = (T)ph.idx;
  const T h = (T)ph.h, hh = (T)ph.hh, h6 = (T)ph.h6;
  const bool per = (g.bc_x == FS_BC_PERIODIC);
  {
    const int i = c % nx, j = c / nx;
    const int i1 = (per && i + 1 == nx) ? 0 : i + 1;
    T K[3];
    if (DIM == 1) {
      const T dxey = (En[nn + i1] - En[nn + i]) * idx;
      const T dxez = (En[2 * nn + i1] - En[2 * nn + i]) * idx;
      K[0] = (T)0;
      K[1] = dxez;
      K[2] = -dxey;
    } else {
      const int j1 = (j + 1 == ny) ? 0 : j + 1;
      const int q00 = j * nxn + i, q10 = j * nxn + i1;
      const int q01 = j1 * nxn + i, q11 = j1 * nxn + i1;
      const T dxey = ((En[nn + q10] + En[nn + q11]) - (En[nn + q00] + En[nn + q01])) * hdx;
      const T dxez = ((En[2 * nn + q10] + En[2 * nn + q11]) -
                      (En[2 * nn + q00] + En[2 * nn + q01])) * hdx;
      const T dyex = ((En[q01] + En[q11]) - (En[q00] + En[q10])) * hdy;
      const T dyez = ((En[2 * nn + q01] + En[2 * nn + q11]) -
                      (En[2 * nn + q00] + En[2 * nn + q10])) * hdy;
      K[0] = -dyez;
      K[1] = dxez;
      K[2] = dyex - dxey;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const size_t k = (size_t)q * nc + c;
      rk4_stage<T>(stage, K[q], Bsum[k], Bs[k], B[k], h, hh, h6);
    }
  }
}

template <typename T, int DIM>
__global__ void k_faraday(const T* __restrict__ En, T* __restrict__ B,
                          T* __restrict__ Bs, T* __restrict__ Bsum, int stage,
                          Geo g, Phys ph) {
  const int nc = g.nx * g.ny;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x)
    faraday_cell<T, DIM>(c, En, B, Bs, Bsum, stage, g, ph);
}

// The field kernels' constants in the run's precision, formed on the host
// (kernel parameters of that type need no FP64 conversion on the device).
template <typename T>
struct FieldConst {
  T idx, hdx, hdy, te, jcr, eta;  // 1/dx, 1/(2dx), 1/(2dy), T_e, j_cr, eta
  T h, hh, h6;                    // RK4 substep h, h/2, h/6
  int resist;                     // eta != 0
};
template <typename T>
inline FieldConst<T> field_const(const Phys& ph) {
  return FieldConst<T>{(T)ph.idx, (T)ph.hdx, (T)ph.hdy, (T)ph.te, (T)ph.jcr,
                       (T)ph.eta, (T)ph.h,   (T)ph.hh,  (T)ph.h6, ph.eta != 0.0 ? 1 : 0};
}
// the same on the device (IEEE conversions round alike on host and device)
template <typename T>
__device__ __forceinline__ FieldConst<T> field_const_dev(const Phys& ph) {
  return FieldConst<T>{(T)ph.idx, (T)ph.hdx, (T)ph.hdy, (T)ph.te, (T)ph.jcr,
                       (T)ph.eta, (T)ph.h,   (T)ph.hh,  (T)ph.h6, ph.eta != 0.0 ? 1 : 0};
}

// Ohm's law from B at every node with the density terms formed here and kept in
// preo ([1/n][-(T_e dn/dx)][-(T_e dn/dy)]) for the stages that follow: the
// start of the 2D field advance.
template <typename T, int DIM>
__global__ void k_ohm_start(const T* __restrict__ Bc, const T* __restrict__ nN,
                            const T* __restrict__ uN, T* __restrict__ Eo, T* __restrict__ preo,
                            Geo g, Phys ph) {
  const int nn = g.nxn * g.ny;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nn; q += gridDim.x * blockDim.x)
    ohm_node<T, DIM>(q, Bc, nN, uN, nullptr, Eo, nullptr, nullptr, g, ph, preo);
}

// ------------------------------------------------------------------------
// One RK4 stage of the 2D field advance in one pass: Faraday from Ei and the
// stage update of B (stages 1-3: the stage field, kept in registers; stage 4:
// the new B, into Bnew), then Ohm's E of that field at the nodes into Eo; with
// FIN also Bbar and the packed gather block G. A warp marches down the rows
// of a strip of 32 columns (lane = column i: its node and the cell to its
// right): a row's E, B, RK4 sum, u and density terms are read once, the
// neighbour columns come by shuffles, the previous row's sums stay in
// registers, and nothing is shared between warps. Cell i needs node i + 1 (the
// lane above), node i needs cell i - 1 (the lane below), so lanes 1 .. 30 are
// the strip's own 30 columns; the cell row above the chunk is formed again.
// Same expressions as ohm_node and faraday_cell. Used in FP64, where the narrow
// FP64 pipe binds (80 % busy): against a pass per operator the row and column
// sums that neighbours share are formed once, 53 operations per node and stage
// instead of 65, and the stage field never goes to memory. 4096 x 256 cells,
// two substeps: 1345 -> 1175 us. (In FP32, 8192 x 512 cells: 612 us against
// k_field_substep's 340.)
// One warp per block: the marches are few and long, so that blocks of several
// would leave SMs uneven.
constexpr int kMarchCols = 30;
template <typename T, int STAGE, bool FIN>
__global__ void __launch_bounds__(32)
    k_field_march(const T* __restrict__ Ei, T* __restrict__ Eo, const T* __restrict__ B,
                  T* __restrict__ Bsum, T* __restrict__ Bnew, const T* __restrict__ uN,
                  const T* __restrict__ pre, T* __restrict__ Bbo, T* __restrict__ G, Geo g,
                  FieldConst<T> fc, int rows, int strips) {
  const int nx = g.nx, ny = g.ny, nxn = g.nxn;
  const int nc = nx * ny, nn = nxn * ny;
  const int lane = threadIdx.x & 31;
  const int strip = blockIdx.x % strips, j0 = (blockIdx.x / strips) * rows;
  const int j1 = min(ny, j0 + rows);
  const bool per = g.bc_x == FS_BC_PERIODIC;
  const int i = strip * kMarchCols - 1 + lane;
  // this lane's node and cell columns (clamped or wrapped into the box)
  const int ni = per ? wrap(i, nx) : min(max(i, 0), nx);
  const int ci = per ? ni : min(max(i, 0), nx - 1);
  const bool own = lane >= 1 && lane <= kMarchCols;
  const bool own_node = own && i < nxn, own_cell = own && i < nx;
  const bool wall0 = !per && i == 0, wall1 = !per && i == nx;
  const T hdx = fc.hdx, hdy = fc.hdy;
  const unsigned full = 0xffffffffu;
  struct Row {  // what a row needs from memory; e: the node row below it
    T e[3], b[3], s[3], u[3], p[3];
  };
  auto load = [&](int j, bool node, Row& r) {
    const int jp = j + 1 == ny ? 0 : j + 1;
    const int qe = jp * nxn + ni, qc = j * nx + ci, qn = j * nxn + ni;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r.e[c] = Ei[c * nn + qe];
      r.b[c] = B[c * nc + qc];
      if (STAGE != 1) r.s[c] = Bsum[c * nc + qc];
      if (node) {
        r.u[c] = uN[c * nn + qn];
        r.p[c] = pre[c * nn + qn];
      }
    }
  };
  T ea[3];        // E of the node row of the current cell row
  T rx, rz;       // its sums of Ex, Ez over a cell's two nodes
  T bs[3], bp[3]; // stage field of the current and the previous cell row
  T pp[3];        // the previous row's sums over a node's two cells
  auto right_sum = [&](T v) { return v + __shfl_down_sync(full, v, 1); };
  // the stage field of a cell row from its loads; st: store the cell's values
  auto cell_row = [&](int j, const Row& r, bool st) {
    const T cy = ea[1] + r.e[1], cz = ea[2] + r.e[2];
    const T dxey = (__shfl_down_sync(full, cy, 1) - cy) * hdx;
    const T dxez = (__shfl_down_sync(full, cz, 1) - cz) * hdx;
    const T nx_ = right_sum(r.e[0]), nz_ = right_sum(r.e[2]);
    const T dyex = (nx_ - rx) * hdy;
    const T dyez = (nz_ - rz) * hdy;
    rx = nx_;
    rz = nz_;
    const T K[3] = {-dyez, dxez, dyex - dxey};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T sum = STAGE != 1 ? r.s[c] : (T)0, b = r.b[c];
      rk4_stage<T>(STAGE, K[c], sum, bs[c], b, fc.h, fc.hh, fc.h6);
      if (STAGE == 4) bs[c] = b;
      if (st) {
        const size_t k = (size_t)c * nc + (size_t)j * nx + i;
        if (STAGE == 4) Bnew[k] = b;
        else Bsum[k] = sum;
      }
      ea[c] = r.e[c];
    }
  };
  // a node's two cells of the current row: lb the left one
  auto pair_sums = [&](T (&p)[3], T (&lb)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      lb[c] = __shfl_up_sync(full, bs[c], 1);
      if (wall1) bs[c] = lb[c];
      if (wall0) lb[c] = bs[c];
      p[c] = lb[c] + bs[c];
    }
  };
  {
    const int jm = j0 == 0 ? ny - 1 : j0 - 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) ea[c] = Ei[c * nn + jm * nxn + ni];
    rx = right_sum(ea[0]);
    rz = right_sum(ea[2]);
    Row r;
    load(jm, false, r);
    cell_row(jm, r, false);
    T lb[3];
    pair_sums(pp, lb);
#pragma unroll
    for (int c = 0; c < 3; ++c) bp[c] = bs[c];
  }
  Row cur;
  load(j0, true, cur);
  for (int j = j0; j < j1; ++j) {
    Row nxt;
    if (j + 1 < j1) load(j + 1, true, nxt);  // in flight while this row is worked on
    cell_row(j, cur, own_cell);
    T p[3], lb[3];
    pair_sums(p, lb);
    T bb[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) bb[c] = (T)0.25 * (pp[c] + p[c]);
    const T cy = bs[1] + bp[1], cz = bs[2] + bp[2];  // right column's sums
    T ly = __shfl_up_sync(full, cy, 1), lz = __shfl_up_sync(full, cz, 1);
    if (wall0) {
      ly = cy;
      lz = cz;
    }
    const T dxby = (cy - ly) * hdx, dxbz = (cz - lz) * hdx;
    const T dybx = (p[0] - pp[0]) * hdy, dybz = (p[2] - pp[2]) * hdy;
    T E[3];
    ohm_e<T>(dybz, -dxbz, dxby - dybx, bb[0], bb[1], bb[2], cur.p[0], cur.p[1], cur.p[2], cur.u[0],
             cur.u[1], cur.u[2], fc.jcr, fc.eta, fc.resist != 0, E[0], E[1], E[2]);
    if (own_node) {
      const size_t q = (size_t)j * nxn + i;
#pragma unroll
      for (int c = 0; c < 3; ++c) Eo[(size_t)c * nn + q] = E[c];
      if (FIN) {
#pragma unroll
        for (int c = 0; c < 3; ++c) Bbo[(size_t)c * nn + q] = bb[c];
        const T v[8] = {E[0], E[1], E[2], bb[0], bb[1], bb[2], (T)0, (T)0};
        auto put = [&](int gi, int gj) {
          T* dst = G + ((size_t)gj * (nx + 1) + gi) * 8;
#pragma unroll
          for (int c = 0; c < 8; ++c) dst[c] = v[c];
        };
        put(i, j);
        if (j == 0) put(i, ny);
        if (per && i == 0) {
          put(nx, j);
          if (j == 0) put(nx, ny);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      pp[c] = p[c];
      bp[c] = bs[c];
    }
    cur = nxt;
  }
}

// ------------------------------------------------------------------------
// One RK4 substep of the 2D FP32 field advance in one launch: the four stages
// follow each other down the rows of a warp's strip of columns (lane = column),
// each a row behind the one before. At row t the warp reads B, n and u of the
// row once; Ohm's E of B at node row t, stage 1 at cell row t - 1, its E at node
// row t - 1, stage 2 at cell row t - 2, ... stage 4 (the new B) at cell row
// t - 4; with FIN also E, Bbar and the packed gather block G of the new B. What
// a stage needs of earlier rows (B, the RK4 sum, node terms, E and sums of the
// previous row) is kept in registers, neighbour columns come by shuffles: no
// shared memory and no barrier. Each stage spoils one column at either end of
// the warp, the density differences one more at the right: 23 of 32 lanes are
// the strip's own (22 with FIN), and a march starts 4 (5) rows early. At an x
// wall the wall's node reads its one cell on both sides and the density is
// mirrored; y wraps. Same expressions as ohm_node and faraday_cell.
// Bound by instruction issue: 465 per row of 23 columns (556 of 22 with FIN). The tiles of
// 32 x 16 cells before recomputed a halo of 4 to 5 cells, 2.1 times their
// cells, through shared memory and 8 barriers: 8192 x 512 cells, two substeps,
// 571 -> 340 us; 3000 x 250 172 -> 90; 256 x 64 59 -> 34; 512 x 512 periodic
// (a pass per operator before) 141 -> 51.
template <typename T>
struct NodeRow {  // 1/n, the pressure terms and u at a node
  T inv, pgx, pgy, ux, uy, uz;
};
template <typename T>
struct CellSums {  // of the previous cell row: a node's two-cell sums, B_y, B_z
  T p[3], by, bz;
};
template <typename T>
struct NodeSums {  // of the previous node row: E, a cell's two-node sums of Ex, Ez
  T e[3], rx, rz;
};
template <typename T, bool FIN>
__global__ void __launch_bounds__(32)
    k_field_substep(const T* __restrict__ B, T* __restrict__ Bn, const T* __restrict__ nN,
                    const T* __restrict__ uN, T* __restrict__ Eo, T* __restrict__ Bbo,
                    T* __restrict__ G, Geo g, FieldConst<T> fc, int rows, int strips) {
  constexpr int OFF = FIN ? 5 : 4, COLS = FIN ? 22 : 23;
  const int nx = g.nx, ny = g.ny, nxn = g.nxn;
  const int nc = nx * ny, nn = nxn * ny;
  const int lane = threadIdx.x;
  const int strip = blockIdx.x % strips, j0 = (blockIdx.x / strips) * rows;
  const int j1 = min(ny, j0 + rows);
  const bool per = g.bc_x == FS_BC_PERIODIC;
  const int i = strip * COLS - OFF + lane;
  const int ni = per ? wrap(i, nx) : min(max(i, 0), nx);
  const int ci = per ? ni : min(max(i, 0), nx - 1);
  const bool own = lane >= OFF && lane < OFF + COLS;
  const bool own_node = own && i < nxn, own_cell = own && i < nx;
  const bool wall0 = !per && i == 0, wall1 = !per && i == nx;
  const bool edge = __any_sync(0xffffffffu, wall0 || wall1);
  const T hdx = fc.hdx, hdy = fc.hdy, te = fc.te;
  const unsigned full = 0xffffffffu;
  auto up1 = [&](T v) { return __shfl_up_sync(full, v, 1); };
  auto down1 = [&](T v) { return __shfl_down_sync(full, v, 1); };
  // Ohm's law at a node row from the cell row f below it and the sums of the
  // cell row above (kept up to date)
  auto ohm_row = [&](CellSums<T>& s, T (&f)[3], const NodeRow<T>& d, T (&E)[3], T (&bb)[3]) {
    T lb[3], p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) lb[c] = up1(f[c]);
    if (edge) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (wall1) f[c] = lb[c];
        if (wall0) lb[c] = f[c];
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p[c] = lb[c] + f[c];
      bb[c] = (T)0.25 * (s.p[c] + p[c]);
    }
    const T cy = f[1] + s.by, cz = f[2] + s.bz;
    T ly = up1(cy), lz = up1(cz);
    if (edge && wall0) {
      ly = cy;
      lz = cz;
    }
    const T dxby = (cy - ly) * hdx, dxbz = (cz - lz) * hdx;
    const T dybx = (p[0] - s.p[0]) * hdy, dybz = (p[2] - s.p[2]) * hdy;
    ohm_e<T>(dybz, -dxbz, dxby - dybx, bb[0], bb[1], bb[2], d.inv, d.pgx, d.pgy, d.ux, d.uy, d.uz,
             fc.jcr, fc.eta, fc.resist != 0, E[0], E[1], E[2]);
    s = CellSums<T>{{p[0], p[1], p[2]}, f[1], f[2]};
  };
  // K = -curl E at the cell row between the node row in s and the row E
  auto faraday_row = [&](NodeSums<T>& s, const T (&E)[3], T (&K)[3]) {
    const T cy = s.e[1] + E[1], cz = s.e[2] + E[2];
    const T dxey = (down1(cy) - cy) * hdx, dxez = (down1(cz) - cz) * hdx;
    const T rx = E[0] + down1(E[0]), rz = E[2] + down1(E[2]);
    const T dyex = (rx - s.rx) * hdy, dyez = (rz - s.rz) * hdy;
    K[0] = -dyez;
    K[1] = dxez;
    K[2] = dyex - dxey;
    s = NodeSums<T>{{E[0], E[1], E[2]}, rx, rz};
  };
  CellSums<T> cs[5] = {};
  NodeSums<T> ns[4] = {};
  NodeRow<T> nd[5] = {};  // node rows t, t - 1, ...
  T bq[4][3] = {};        // B of cell rows t - 1, t - 2, ...
  T sq[3][3] = {};        // RK4 sums of cell rows t - 2, t - 3, t - 4
  int t = j0 - OFF;
  int r = wrap(t, ny);  // row t in the box
  T nm = nN[wrap(t - 1, ny) * nxn + ni], n0 = nN[r * nxn + ni];
  struct In {
    T b[3], u[3], np;
  };
  auto load = [&](int row, In& x) {
    const int rp = row + 1 == ny ? 0 : row + 1;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x.b[c] = B[c * nc + row * nx + ci];
      x.u[c] = uN[c * nn + row * nxn + ni];
    }
    x.np = nN[rp * nxn + ni];
  };
  In cur;
  load(r, cur);
  for (; t < j1 + 4; ++t) {
    In nxt;
    r = r + 1 == ny ? 0 : r + 1;
    load(r, nxt);  // in flight while this row is worked on
    {
      T nl = up1(n0), nr = down1(n0);
      if (edge) {
        if (wall0) nl = nr;
        if (wall1) nr = nl;
      }
      const T dnx = (nr - nl) * hdx, dny = (cur.np - nm) * hdy;
      nd[0] = NodeRow<T>{(T)1 / n0, -(te * dnx), -(te * dny), cur.u[0], cur.u[1], cur.u[2]};
      nm = n0;
      n0 = cur.np;
    }
    T E[3], bb[3], K[3], f[3], s1[3], s2[3], s3[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] = cur.b[c];
    ohm_row(cs[0], f, nd[0], E, bb);
    faraday_row(ns[0], E, K);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T b = bq[0][c];
      rk4_stage<T>(1, K[c], s1[c], f[c], b, fc.h, fc.hh, fc.h6);
    }
    ohm_row(cs[1], f, nd[1], E, bb);
    faraday_row(ns[1], E, K);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T b = bq[1][c];
      s2[c] = sq[0][c];
      rk4_stage<T>(2, K[c], s2[c], f[c], b, fc.h, fc.hh, fc.h6);
    }
    ohm_row(cs[2], f, nd[2], E, bb);
    faraday_row(ns[2], E, K);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T b = bq[2][c];
      s3[c] = sq[1][c];
      rk4_stage<T>(3, K[c], s3[c], f[c], b, fc.h, fc.hh, fc.h6);
    }
    ohm_row(cs[3], f, nd[3], E, bb);
    faraday_row(ns[3], E, K);
    const int j = t - 4;
    const bool mine = j >= j0;  // (the rows before are the march's start)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T b = bq[3][c], sum = sq[2][c], none;
      rk4_stage<T>(4, K[c], sum, none, b, fc.h, fc.hh, fc.h6);
      f[c] = b;
      if (mine && own_cell) Bn[(size_t)c * nc + (size_t)j * nx + i] = b;
    }
    if (FIN) {
      ohm_row(cs[4], f, nd[4], E, bb);
      if (mine && own_node) {
        const size_t q = (size_t)j * nxn + i;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          Eo[(size_t)c * nn + q] = E[c];
          Bbo[(size_t)c * nn + q] = bb[c];
        }
        auto put = [&](int gi, int gj) {
          float4* dst = (float4*)(G + ((size_t)gj * (nx + 1) + gi) * 8);
          dst[0] = make_float4(E[0], E[1], E[2], bb[0]);
          dst[1] = make_float4(bb[1], bb[2], 0.0f, 0.0f);
        };
        put(i, j);
        if (j == 0) put(i, ny);
        if (per && i == 0) {
          put(nx, j);
          if (j == 0) put(nx, ny);
        }
      }
    }
#pragma unroll
    for (int k = 3; k > 0; --k)
#pragma unroll
      for (int c = 0; c < 3; ++c) bq[k][c] = bq[k - 1][c];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      bq[0][c] = cur.b[c];
      sq[2][c] = s3[c];
      sq[1][c] = s2[c];
      sq[0][c] = s1[c];
    }
#pragma unroll
    for (int k = 4; k > 0; --k) nd[k] = nd[k - 1];
    cur = nxt;
  }
}

// Quantity c (n, Jx, Jy, Jz) at node i of a 1D box with x walls: the far sum,
// then the partials of the tiles whose accumulators cover the node (tile tx:
// nodes tx TX - 1 .. tx TX + TX + 1) in increasing order, wall nodes x2: the
// sums of moments_body.
template <typename T>
__device__ __forceinline__ T moment1(const DevPtrs<T>& d, const Geo& g, int i, int c) {
  using A = typename Num<T>::acc;
  const int TX = g.TX, NA = TX + 3;
  A s = ((const A*)d.far)[(size_t)c * g.nxn + i];
  const int hi = min((i + 1) / TX, g.ntx - 1);
  for (int tx = i >= 2 ? (i - 2) / TX : 0; tx <= hi; ++tx)
    s += ((const A*)d.partial)[((size_t)tx * 4 + c) * NA + i - (tx * TX - 1)];
  T v = acc_value(s);
  if (i == 0 || i == g.nx) v = v * (T)2;
  return v;
}

// E_y (comp 0) or E_z (comp 1) at a node of a 1D grid: the values ohm_e gives
// there (no y differences; with j_ext = 0 its zero products drop out). bm, bp:
// B_y, B_z of the node's left and right cells; bbx: B_x at the node. E_x is
// not needed within a step: Faraday's law has no use for it in 1D and B_x
// stays as it is.
template <typename T>
__device__ __forceinline__ T ohm1_comp(int comp, T bmy, T bpy, T bmz, T bpz, T bbx, T inv_n, T ux,
                                       T uy, T uz, const FieldConst<T>& fc) {
  const T ax = (T)0 - fc.jcr;
  if (comp == 0) {
    const T dby = (bpy - bmy) * fc.idx;
    const T bbz = (T)0.5 * (bmz + bpz);
    const T cay = fc.jcr != (T)0 ? fmaT(dby, bbx, -(ax * bbz)) : dby * bbx;
    const T cuy = fmaT(uz, bbx, -(ux * bbz));
    T ey = fmaT(cay, inv_n, -cuy);
    if (fc.resist) {
      const T cyv = -((bpz - bmz) * fc.idx);
      ey = ey + fc.eta * cyv;
    }
    return ey;
  }
  const T dbz = (bpz - bmz) * fc.idx;
  const T bby = (T)0.5 * (bmy + bpy);
  const T caz = fc.jcr != (T)0 ? fmaT(ax, bby, dbz * bbx) : dbz * bbx;
  const T cuz = fmaT(ux, bby, -(uy * bbx));
  T ez = fmaT(caz, inv_n, -cuz);
  if (fc.resist) {
    const T czv = (bpy - bmy) * fc.idx;
    ez = ez + fc.eta * czv;
  }
  return ez;
}

// A 1D tile: L cells, L + 1 nodes; the block's two halves (half >= L + 1
// threads each, a multiple of the warp) take one transverse component each,
// a thread one cell and one node. What stays fixed over the stages and the
// thread's own B and RK4 sum are in registers; the stage field S and, in FP64,
// E_y and E_z at the nodes are in shared memory.
template <typename T>
struct Node1 {  // 1/n, B_x and u at a node
  T inv, bbx, ux, uy, uz;
};
template <typename T>
struct Tile1 {
  int L, half, comp, a;
  T* S;  // stage field: FP32 [2 buffers][2][L], FP64 [2][L]
  T* E;  // FP64 only: E_y, E_z [2][L + 1]
  Node1<T> n0, n1;  // the thread's node a, and (FP32) node a + 1
  T b, k;           // B of the thread's component at cell a, the RK4 sum
};
// values of T a tile keeps in shared memory
__host__ __device__ constexpr size_t tile1_words(size_t L, size_t tsz) {
  return tsz == 4 ? 4 * L : 2 * L + 2 * (L + 1);
}
// threads of a block of two halves for a tile of L cells
__host__ __device__ constexpr int tile1_threads(int L) { return 2 * ((L + 1 + 31) / 32 * 32); }

// One RK4 substep (four stages of Ohm and Faraday) of a tile with n, u
// frozen, K_y = dE_z/dx, K_z = -dE_y/dx. At the tile's ends a node reads its
// end cell on both sides. Stage s's input field goes to keep[s] ([2][L]) if
// given. FP32, latency-bound: a thread forms the E of both nodes of its cell,
// so that a stage is one pass and one barrier on alternating buffers. FP64,
// bound by its instruction count (an FP64 instruction holds an SM quarter's
// pipe for 64 cycles): E once per node, in a pass of its own.
template <typename T>
__device__ __forceinline__ void tile1_substep(Tile1<T>& t, const FieldConst<T>& fc, T* keep) {
  const int L = t.L, Ln = L + 1, a = t.a;
  const bool cell = a < L;
  T bs = t.b;
  if constexpr (sizeof(T) == 4) {
    const int m = max(a - 1, 0), p = min(a + 1, L - 1);
#pragma unroll
    for (int stage = 1; stage <= 4; ++stage) {
      const T* y = t.S + ((stage - 1) & 1) * 2 * L;
      T* d = t.S + (stage & 1) * 2 * L;
      if (cell) {
        const T ym = y[m], yc = y[a], yp = y[p];
        const T zm = y[L + m], zc = y[L + a], zp = y[L + p];
        if (keep) keep[(2 * (stage - 1) + t.comp) * L + a] = t.comp ? zc : yc;
        const int oc = 1 - t.comp;  // B_y needs E_z, B_z needs E_y
        const T e0 = ohm1_comp<T>(oc, ym, yc, zm, zc, t.n0.bbx, t.n0.inv, t.n0.ux, t.n0.uy,
                                  t.n0.uz, fc);
        const T e1 = ohm1_comp<T>(oc, yc, yp, zc, zp, t.n1.bbx, t.n1.inv, t.n1.ux, t.n1.uy,
                                  t.n1.uz, fc);
        const T dx = (e1 - e0) * fc.idx;
        rk4_stage<T>(stage, t.comp ? -dx : dx, t.k, bs, t.b, fc.h, fc.hh, fc.h6);
        d[t.comp * L + a] = stage == 4 ? t.b : bs;
      }
      __syncthreads();
    }
  } else {
    const int m = max(a - 1, 0), p = min(a, L - 1);
    T* own = t.S + t.comp * L + a;
    const T* eo = t.E + (t.comp ? 0 : Ln) + a;
#pragma unroll
    for (int stage = 1; stage <= 4; ++stage) {
      const T* y = t.S;
      if (keep && cell) keep[(2 * (stage - 1) + t.comp) * L + a] = *own;
      if (a < Ln)
        t.E[t.comp * Ln + a] = ohm1_comp<T>(t.comp, y[m], y[p], y[L + m], y[L + p], t.n0.bbx,
                                            t.n0.inv, t.n0.ux, t.n0.uy, t.n0.uz, fc);
      __syncthreads();
      if (cell) {
        const T dx = (eo[1] - eo[0]) * fc.idx;
        rk4_stage<T>(stage, t.comp ? -dx : dx, t.k, bs, t.b, fc.h, fc.hh, fc.h6);
        *own = stage == 4 ? t.b : bs;
      }
      __syncthreads();
    }
  }
}

// The full Ohm's law at a tile's node from its field y ([2][L]), the node's
// cells m and p and its pressure term.
template <typename T>
__device__ __forceinline__ void tile1_ohm(const T* y, int L, int m, int p, const Node1<T>& n,
                                          T pg, const FieldConst<T>& fc, T (&E)[3], T (&Bb)[3]) {
  const T bmy = y[m], bpy = y[p], bmz = y[L + m], bpz = y[L + p];
  Bb[0] = n.bbx;
  Bb[1] = (T)0.5 * (bmy + bpy);
  Bb[2] = (T)0.5 * (bmz + bpz);
  const T dby = (bpy - bmy) * fc.idx, dbz = (bpz - bmz) * fc.idx;
  ohm_e<T>((T)0, -dbz, dby, Bb[0], Bb[1], Bb[2], n.inv, pg, -(fc.te * (T)0), n.ux, n.uy, n.uz,
           fc.jcr, fc.eta, fc.resist != 0, E[0], E[1], E[2]);
}

// ------------------------------------------------------------------------
// The moments and the whole field advance of a 1D step with x walls (n, J, u
// from the deposit, n_sub RK4 substeps, then Ohm's E and Bbar for the next
// gather) in one launch: on a 1D grid the separate passes are tens of tiny
// launches per step. Neighbouring tiles read the same B and far sums, so the
// new B goes to the other buffer and the other far sums, of the step before,
// are cleared for the next (Sim::swaps_fields); the first block counts the
// step. (With a launch of its own for that, twenty FP64 steps of 512 cells 758
// us, ten FP32 steps of 8100 cells 524; now 719 and 509.) A CTA owns TILE cells
// (and their left nodes; the last tile also node nx) and runs every pass in
// shared memory over its cells plus field1_halo(n_sub) cells around
// them, which it recomputes: each pass's stencil reaches one cell, so
// values made wrong at a tile's inner edges (read with indices clamped to
// the tile) move in by one cell per pass and stay outside the owned cells;
// at a wall the clamped indices are the wall's ghost cells and the density
// is mirrored as in density_terms. Reads B from Bin, writes the new B to
// Bout (neighbouring tiles read Bin's cells), E, Bbar and the packed gather
// block G at the owned nodes. Same per-element arithmetic as ohm_node /
// faraday_cell (1D), so FP64 results are those of the separate passes.
// A chain of dependent passes (tile1_substep): 1/n and the pressure term are
// formed once, B_x and E_x are left out of the stages, the y and z components
// go to different warps, and a thread keeps its node's terms in registers.
// TILE 32 while that leaves SMs free (tile and halo fill two warps a
// component), 64 beyond (less halo to recompute). 512 cells FP64: 14.4 us with
// the moments, which took 8.6 us beside the fields' 21.5 before.
__host__ __device__ constexpr int field1_halo(int n_sub) { return 4 * n_sub + 2; }
constexpr int kF1 = 64, kF1Small = 32;
constexpr int kF1MaxSub = 16;
constexpr int field1_threads(int tile, int n_sub) {
  return tile1_threads(tile + 2 * field1_halo(n_sub));
}
inline int field1_tile(int nx) { return nx <= 152 * kF1 ? kF1Small : kF1; }
template <typename T>
inline size_t field1_smem(int n_sub, int tile) {
  const size_t L = tile + 2 * (size_t)field1_halo(n_sub);
  return sizeof(T) * (tile1_words(L, sizeof(T)) + 6 * (L + 1));
}

// Tile blk of the 1D field advance (the body of k_field_step1); smem is the
// block's dynamic shared memory (field1_smem(n_sub, TILE) bytes); at least
// field1_threads(TILE, n_sub) threads.
template <typename T, int TILE>
__device__ __forceinline__ void field_step1_body(const DevPtrs<T>& d, const Geo& g, T n_floor,
                                                 const FieldConst<T>& fc, int n_sub, int blk,
                                                 unsigned char* smem) {
  const int nx = g.nx, nxn = g.nxn, t0 = threadIdx.x, nt = blockDim.x;
  const int H = field1_halo(n_sub);
  const int c0 = blk * TILE, c1 = min(nx, c0 + TILE);
  const int lo = max(0, c0 - H), L = min(nx, c1 + H) - lo, Ln = L + 1;
  auto owns_node = [&](int i) { return i >= c0 && (i < c1 || (i == nx && c1 == nx)); };
  Tile1<T> t;
  t.L = L;
  t.half = blockDim.x / 2;
  t.comp = (int)threadIdx.x >= t.half;
  const int a = t.a = threadIdx.x - t.comp * t.half;
  t.S = (T*)smem;
  t.E = t.S + 2 * L;
  T* sn = t.S + tile1_words(L, sizeof(T));  // [Ln] n
  T* sinv = sn + Ln;                        // [Ln] 1/n
  T* spg = sinv + Ln;                       // [Ln] the pressure term -(T_e dn/dx)
  T* su = spg + Ln;                         // [3][Ln] J, then u
  const int gi = lo + a;                    // this thread's cell and node
  T bxm = (T)0, bxc = (T)0, bxp = (T)0;
  t.b = (T)0;
  if (a < L) {
    t.b = d.B[(t.comp + 1) * nx + gi];
    t.S[t.comp * L + a] = t.b;
    bxp = d.B[lo + min(a + 1, L - 1)];
  }
  if (a < Ln) {
    bxm = d.B[lo + max(a - 1, 0)];
    bxc = d.B[lo + min(a, L - 1)];
  }
  for (int k = t0; k < 4 * Ln; k += nt) {
    const int c = k / Ln, i = k - c * Ln;
    const T v = moment1<T>(d, g, lo + i, c);
    if (owns_node(lo + i)) ((typename Num<T>::acc*)d.far_next)[c * nxn + lo + i] = 0;
    if (c == 0) {
      const T n = v < n_floor ? n_floor : v;
      sn[i] = n;
      if (owns_node(lo + i)) d.n[lo + i] = n;
    } else {
      su[k - Ln] = v;
      if (owns_node(lo + i)) d.J[(c - 1) * nxn + lo + i] = v;
    }
  }
  __syncthreads();
  for (int k = t0; k < 5 * Ln; k += nt) {
    const int c = k / Ln, i = k - c * Ln;
    if (c < 4) {  // u = J / n, then 1/n
      const T v = (c < 3 ? su[k] : (T)1) / sn[i];
      if (c == 3) {
        sinv[i] = v;
      } else {
        su[k] = v;
        if (owns_node(lo + i)) d.u[c * nxn + lo + i] = v;
      }
    } else {
      const int q = lo + i;
      const int xp = ((q + 1 > nx) ? 2 * nx - (q + 1) : q + 1) - lo;
      const int xm = ((q - 1 < 0) ? -(q - 1) : q - 1) - lo;
      const T dnx = (sn[min(max(xp, 0), L)] - sn[min(max(xm, 0), L)]) * fc.hdx;
      spg[i] = -(fc.te * dnx);
    }
  }
  __syncthreads();
  auto node = [&](int i, T bm, T bp) {
    return Node1<T>{sinv[i], (T)0.5 * (bm + bp), su[i], su[Ln + i], su[2 * Ln + i]};
  };
  if (a < Ln) t.n0 = node(a, bxm, bxc);
  if (sizeof(T) == 4 && a < L) t.n1 = node(a + 1, bxc, bxp);
  for (int sub = 0; sub < n_sub; ++sub) tile1_substep<T>(t, fc, nullptr);
  if (t.comp == 0 && a < Ln && owns_node(gi)) {
    T E[3], Bb[3];
    tile1_ohm<T>(t.S, L, max(a - 1, 0), min(a, L - 1), t.n0, spg[a], fc, E, Bb);
    const T v[8] = {E[0], E[1], E[2], Bb[0], Bb[1], Bb[2], (T)0, (T)0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      d.E[c * nxn + gi] = E[c];
      d.Bb[c * nxn + gi] = Bb[c];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      d.G[(size_t)gi * 8 + c] = v[c];                  // row 0
      d.G[((size_t)(nx + 1) + gi) * 8 + c] = v[c];     // its ghost copy (row ny = 1)
    }
  }
  if (a < L && gi >= c0 && gi < c1) {
    d.Bs[(t.comp + 1) * nx + gi] = t.b;
    if (t.comp == 0) d.Bs[gi] = bxc;
  }
  if (blk == 0 && t0 == 0) step_end(d.ctr, d.inj, g);
}

template <typename T, int TILE>
__global__ void __launch_bounds__(field1_threads(TILE, kF1MaxSub))
    k_field_step1(DevPtrs<T> d, Geo g, T n_floor, FieldConst<T> fc, int n_sub) {
  extern __shared__ __align__(16) unsigned char smem[];
  field_step1_body<T, TILE>(d, g, n_floor, fc, n_sub, blockIdx.x, smem);
}

// ------------------------------------------------------------------------
// Initial load (Sec. 2 set-up): ppc particles per cell, ids in cell-major
// order, position uniform in the cell, velocity a Maxwellian of thermal speed
// sqrt(beta_i/2) drifting at -u_sh x.
// ------------------------------------------------------------------------
template <typename T, int DIM>
__global__ void k_init_particles(DevPtrs<T> d, Geo g, Phys ph, int buf, int ppc) {
  const long long total = (long long)g.nx * g.ny * ppc;
  const Parts<T> P = d.P[buf];
  for (long long pidl = blockIdx.x * (long long)blockDim.x + threadIdx.x;
       pidl < total; pidl += (long long)gridDim.x * blockDim.x) {
    const uint32_t pid = (uint32_t)pidl;
    const long long cidx = pidl / ppc;
    const int k = (int)(pidl % ppc);
    const int i = (int)(cidx % g.nx), j = (int)(cidx / g.nx);
    const int tx = i / g.TX, ty = j / g.TY;
    const int t = ty * g.ntx + tx;
    const int lc = (i - tx * g.TX) + (j - ty * g.TY) * g.TX;
    const int gi = d.tile_base[t] + lc * ppc + k;
    const Philox4 ra = draw4(ph.seed, pid, 0, kPurposeInitA);
    const Philox4 rb = draw4(ph.seed, pid, 0, kPurposeInitB);
    const double fx = u01(ra.x[0]);
    const double fy = (DIM == 2) ? u01(ra.x[1]) : 0.0;
    double g0, g1, g2, g3;
    gauss2(u01(ra.x[2]), u01(ra.x[3]), &g0, &g1);
    gauss2(u01(rb.x[0]), u01(rb.x[1]), &g2, &g3);
    double vx = __dsub_rn(__dmul_rn(ph.vth, g0), ph.mach_a);
    double vy = __dmul_rn(ph.vth, g1);
    double vz = __dmul_rn(ph.vth, g2);
    if (ph.c2inv > 0.0) {  // stored as u = gamma v
      const double gv = gamma_v(vx, vy, vz, ph.c2inv);
      vx = __dmul_rn(vx, gv); vy = __dmul_rn(vy, gv); vz = __dmul_rn(vz, gv);
    }
    T ft = (T)fx, fyt = (T)fy;
    if (ft >= (T)1) ft = Num<T>::offmax;
    if (fyt >= (T)1) fyt = Num<T>::offmax;
    P.cell[gi] = (j << 16) | i;
    P.ox[gi] = ft;
    if (DIM == 2) P.oy[gi] = fyt;
    P.vx[gi] = (T)vx;
    P.vy[gi] = (T)vy;
    P.vz[gi] = (T)vz;
    P.id[gi] = pid;
  }
}

// Deposit every particle of buffer buf into the far accumulators (set-up and
// after a host injection; the per-tile partials are zero then).
template <typename T, int DIM>
__global__ void k_deposit_all(DevPtrs<T> d, Geo g, Phys ph, int buf) {
  const int t = blockIdx.x;
  const int cnt = min(d.cnt[buf][t], g.tile_cap);
  const int base = d.tile_base[t];
  const Parts<T> P = d.P[buf];
  const double ws = deposit_weight_scale<T>();
  const T wth = (T)(ph.w_th * ws), wcr = (T)(ph.w_cr * ws);
  for (int p = threadIdx.x; p < cnt; p += blockDim.x) {
    const int gi = base + p;
    const int cell = P.cell[gi];
    const uint32_t id = P.id[gi];
    T vx, vy, vz;  // the current uses the velocity
    velocity_of<T>(P.vx[gi], P.vy[gi], P.vz[gi], (T)ph.c2inv, vx, vy, vz);
    deposit_far<T, DIM>(d, g, cell & 0xFFFF, cell >> 16, P.ox[gi],
                        DIM == 2 ? P.oy[gi] : (T)0, (id & kIdCR) ? wcr : wth, vx, vy, vz);
  }
}

// Insert n particles given as FP64 columns (validated on the host, copied to
// the device as they are) into buffer buf: ids NULL gives first, first + 1, ...
template <typename T, int DIM>
__global__ void k_insert_columns(DevPtrs<T> d, Columns src, Geo g, int buf, int n,
                                 const uint32_t* __restrict__ ids, unsigned long long first) {
  const Parts<T> P = d.P[buf];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += gridDim.x * blockDim.x) {
    const int i = src.ci[k], j = (DIM == 2) ? src.cj[k] : 0;
    const int t = (j / g.TY) * g.ntx + i / g.TX;
    const int slot = atomicAdd(&d.cnt[buf][t], 1);
    if (slot >= g.tile_cap) {
      atomicSub(&d.cnt[buf][t], 1);
      atomicOr(&d.ctr->status, kStatusCapacity);
      continue;
    }
    const int gi = t * g.tile_cap + slot;
    T fx = (T)src.col[0][k], fy = (DIM == 2) ? (T)src.col[1][k] : (T)0;
    if (fx >= (T)1) fx = Num<T>::offmax;
    if (fy >= (T)1) fy = Num<T>::offmax;
    P.cell[gi] = (j << 16) | i;
    P.ox[gi] = fx;
    if (DIM == 2) P.oy[gi] = fy;
    P.vx[gi] = (T)src.col[2][k];
    P.vy[gi] = (T)src.col[3][k];
    P.vz[gi] = (T)src.col[4][k];
    P.id[gi] = ids ? ids[k] : (uint32_t)(first + (unsigned long long)k);
  }
}

// Exclusive prefix sums of the tiles' particle counts (clamped to the
// capacity) into off, their total into *total. One CTA.
static __global__ void __launch_bounds__(1024)
    k_scan_counts(const int* __restrict__ cnt, int ntiles, int cap, int* __restrict__ off,
                  unsigned long long* __restrict__ total) {
  __shared__ int wsum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int per = (ntiles + blockDim.x - 1) / blockDim.x;
  const int b = min(ntiles, (int)threadIdx.x * per), e = min(ntiles, b + per);
  int s = 0;
  for (int t = b; t < e; ++t) s += min(cnt[t], cap);
  int inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    int x = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += v;
    }
    wsum[lane] = x;
  }
  __syncthreads();
  int run = (w ? wsum[w - 1] : 0) + inc - s;
  for (int t = b; t < e; ++t) {
    off[t] = run;
    run += min(cnt[t], cap);
  }
  if (threadIdx.x == 0) *total = (unsigned long long)wsum[31];
}

// ------------------------------------------------------------------------
// Diagnostics (FP64 sums; order of the block partial sums is not fixed).
// ------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// A value as FP32, correct to one unit in the last place: FP64 values are cut
// by integer operations (the conversion instruction runs on GB300's narrow
// FP64 pipe); below FP32's range 0, above it an infinity.
__device__ __forceinline__ float near_float(float x) { return x; }
__device__ __forceinline__ float near_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7FFu) - 896;
  const unsigned m = e <= 0 ? 0u
                     : e >= 255 ? 0x7F800000u
                                : ((unsigned)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  return __uint_as_float((hi & 0x80000000u) | m);
}
// An FP32 value as FP64 (exact) by integer operations, for the same reason;
// subnormals are brought into the normal range first (x 2^64, exact);
// infinities and NaN stay so.
__device__ __forceinline__ double wide_double(double x) { return x; }
__device__ __forceinline__ double wide_double(float x) {
  const bool low = fabsf(x) < 0x1p-126f;
  const unsigned b = __float_as_uint(low ? x * 0x1p64f : x), e = (b >> 23) & 0xFFu;
  const unsigned hi = (b & 0x80000000u) |
                      (e == 0 ? 0u
                              : (((e == 0xFFu ? 0x7FFu : e + (low ? 832u : 896u)) << 20) |
                                 ((b & 0x7FFFFFu) >> 3)));
  return __hiloint2double((int)hi, (int)((b & 7u) << 29));
}

constexpr int kWarpsPerBlock = kBlock / 32;

// Adds 1 to cnt[k] for every lane of the warp with k >= 0 (all lanes call).
// Lanes on the counter of the lowest remaining lane are added as one, twice
// over; the rest add their own: a drifting thermal plasma puts most lanes
// on one or two counters, and shared atomics on one word are serialised lane
// by lane.
__device__ __forceinline__ void count_shared(unsigned* cnt, int k) {
  unsigned todo = __ballot_sync(0xffffffffu, k >= 0);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (!todo) return;
    const int l = __ffs(todo) - 1;
    const int k0 = __shfl_sync(0xffffffffu, k, l);
    const unsigned same = __ballot_sync(0xffffffffu, k == k0);
    if (lane == l) atomicAdd(&cnt[k0], (unsigned)__popc(same));
    todo &= ~same;
  }
  if ((todo >> lane) & 1u) atomicAdd(&cnt[k], 1u);
}

// Kinetic energy and momentum sums of buffer buf. One warp per tile, a grid
// of a few CTAs per SM that strides over the tiles. Bound by the FP64 pipe: 7
// operations per particle without relativistic terms (its weight and the cell
// volume come as one factor), against 19 and a block reduction per tile
// before; one set of sums for both species (two, chosen per lane, ran both
// sides of the choice: 449 us). 17.8 M particles FP64: 990 -> 290 us.
template <typename T, int DIM>
__global__ void __launch_bounds__(kBlock) k_diag_particles(DevPtrs<T> d, Geo g, Phys ph, int buf) {
  const Parts<T> P = d.P[buf];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s[4] = {0, 0, 0, 0};  // w v.v / 2 (or energy), w v
  unsigned long long live = 0;
  const bool rel = ph.c2inv > 0.0;
  const double wt = ph.w_th * ph.cellvol, wc = ph.w_cr * ph.cellvol;
  for (int t = blockIdx.x * kWarpsPerBlock + warp; t < g.ntiles;
       t += gridDim.x * kWarpsPerBlock) {
    const int cnt = min(d.cnt[buf][t], g.tile_cap), base = t * g.tile_cap;
    live += (unsigned)cnt;
#pragma unroll 4
    for (int p = lane; p < cnt; p += 32) {
      const int gi = base + p;
      const double w = (P.id[gi] & kIdCR) ? wc : wt;
      const double vx = wide_double(P.vx[gi]), vy = wide_double(P.vy[gi]),
                   vz = wide_double(P.vz[gi]);
      if (rel) s[0] += kinetic(w, vx, vy, vz, 1.0, ph.c2inv);
      else s[0] = __fma_rn(w, __fma_rn(vz, vz, __fma_rn(vy, vy, __dmul_rn(vx, vx))), s[0]);
      s[1] = __fma_rn(w, vx, s[1]);
      s[2] = __fma_rn(w, vy, s[2]);
      s[3] = __fma_rn(w, vz, s[3]);
    }
  }
  if (lane == 0 && live) atomicAdd(&d.ctr->live, live);
  __shared__ double red[4][kWarpsPerBlock];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double v = warp_sum((q == 0 && !rel) ? 0.5 * s[q] : s[q]);
    if (lane == 0) red[q][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double v = 0;
    for (int w = 0; w < kWarpsPerBlock; ++w) v += red[threadIdx.x][w];
    atomicAdd(&d.ctr->sums[threadIdx.x], v);
  }
}

template <typename T>
__global__ void k_diag_field(DevPtrs<T> d, Geo g, Phys ph) {
  const int nc = g.nx * g.ny;
  double s = 0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc;
       c += gridDim.x * blockDim.x) {
    const double bx = d.B[c], by = d.B[nc + c], bz = d.B[2 * nc + c];
    s += (0.5 * ((bx * bx + by * by) + bz * bz)) * ph.cellvol;
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) atomicAdd(&d.ctr->sums[4], s);
  // Stability number of the field integrator, z = h omega_max with h the
  // RK4 substep: the fastest discrete mode is bounded by the grid-scale
  // whistler, k^2 |Bbar| / n with k^2 <= 4/dx^2 + 4/dy^2 for the staggered
  // differences, plus advection, k |u| with k <= 2/dx + 2/dy. Kept as the
  // maximum over nodes in sums[5] (non-negative doubles order like their
  // bit patterns).
  // Two square roots and a division per node in FP64 would bind this kernel to
  // the FP64 pipe, so a node's z is first bounded in FP32 and only nodes whose
  // upper bound reaches the block's largest lower bound take the FP64 expression.
  const double kk = 16.0 * (ph.hdx * ph.hdx + ph.hdy * ph.hdy);
  const double ka = 4.0 * (ph.hdx + ph.hdy);
  const int nn = g.nxn * g.ny;
  const float kkf = (float)kk, kaf = (float)ka;
  // side -1: a lower, 1: an upper bound of z / h but for rounding (below 1e-5):
  // what the squares of B or u lose below FP32's normal range is far less than
  // the 1e-30 that is taken off or added, which changes |B| or |u| by 1e-15 at
  // most (from 1e-12 on by less than 1e-6 of it)
  auto bound = [&](int c, float side) {
    const float bx = near_float(d.Bb[c]), by = near_float(d.Bb[nn + c]),
                bz = near_float(d.Bb[2 * nn + c]);
    const float ux = near_float(d.u[c]), uy = near_float(d.u[nn + c]),
                uz = near_float(d.u[2 * nn + c]);
    const float b2 = bx * bx + by * by + bz * bz + side * 1e-30f;
    const float u2 = ux * ux + uy * uy + uz * uz + side * 1e-30f;
    return kkf * sqrtf(b2 < 0.0f ? 0.0f : b2) / near_float(d.n[c]) +
           kaf * sqrtf(u2 < 0.0f ? 0.0f : u2);  // (NaN stays NaN)
  };
  float zf = 0.0f;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nn; c += gridDim.x * blockDim.x) {
    const float z = bound(c, -1.0f);
    // beyond FP32's range (or NaN): every node takes the FP64 expression
    zf = (z < 1e30f) ? fmaxf(zf, z) : INFINITY;
  }
  __shared__ unsigned zblk;
  if (threadIdx.x == 0) zblk = 0u;
  __syncthreads();
  atomicMax(&zblk, __reduce_max_sync(0xffffffffu, __float_as_uint(zf)));
  __syncthreads();
  const float lim = __uint_as_float(zblk);
  // the bounds hold while their factors' products stay in FP32's normal range:
  // factors and densities within 1e-15 .. 1e15 (n >= n_floor), and a largest z
  // to which a product below that range adds nothing
  const bool plain = kkf > 1e-15f && kkf < 1e15f && kaf > 1e-15f && kaf < 1e15f &&
                     ph.n_floor > 1e-15;
  const float from = (plain && lim < 1e30f && lim > 1e-6f) ? lim * (1.0f - 1e-4f) : -1.0f;
  double zmax = 0.0;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nn;
       c += gridDim.x * blockDim.x) {
    if (from >= 0.0f && !(bound(c, 1.0f) >= from)) continue;
    const double bx = d.Bb[c], by = d.Bb[nn + c], bz = d.Bb[2 * nn + c];
    const double ux = d.u[c], uy = d.u[nn + c], uz = d.u[2 * nn + c];
    const double b = sqrt(bx * bx + by * by + bz * bz);
    const double um = sqrt(ux * ux + uy * uy + uz * uz);
    const double z = ph.h * (kk * b / (double)d.n[c] + ka * um);
    zmax = z > zmax ? z : zmax;  // a NaN z leaves zmax; NaN is caught elsewhere
  }
  if (zmax > 0.0)
    atomicMax((unsigned long long*)&d.ctr->sums[5], (unsigned long long)__double_as_longlong(zmax));
}

// x - p_x histogram of buffer buf. A CTA takes gx x gy tiles (a warp per
// tile); their particles reach only a few x bins, so the counts are kept in
// shared memory (nbx x hist_np counters; nbx = 0: too many, straight to
// global memory) and added to the histogram once. The bins are formed in FP32
// relative to the CTA's first cell; only values within eps of a bin edge
// take the written FP64 expressions (GB300's FP64 pipe is narrow).
// 17.8 M particles FP64: 505 -> 91 us.
constexpr int kHistShared = 8192;  // counters
template <typename T, int DIM>
__global__ void __launch_bounds__(kBlock)
    k_hist(DevPtrs<T> d, Geo g, Phys ph, int buf, int species, int gx, int gy, int nbx) {
  extern __shared__ unsigned sh[];
  const Parts<T> P = d.P[buf];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double hsx = (double)ph.hist_nx / (double)g.nx;
  const double hsp = (double)ph.hist_np / (ph.hist_pmax - ph.hist_pmin);
  const int tx0 = blockIdx.x * gx, ty0 = blockIdx.y * gy;
  const int ntx = min(gx, g.ntx - tx0), nty = min(gy, g.nty - ty0);
  const int i0 = tx0 * g.TX, np = ph.hist_np;
  const double xb = (double)i0 * hsx;
  const int bx0 = min((int)floor(xb), ph.hist_nx - 1);
  for (int k = threadIdx.x; k < nbx * np; k += kBlock) sh[k] = 0u;
  __syncthreads();
  const float fsx = (float)hsx, fsp = (float)hsp, fx0 = (float)(xb - (double)bx0);
  const float pmin = (float)ph.hist_pmin;
  const float epx = 2e-6f * ((float)(gx * g.TX) * fsx + 2.0f);
  const float epp = 2e-6f * ((fabsf(pmin) + fabsf((float)ph.hist_pmax)) * fsp + (float)np);
  const bool fast = epx < 0.25f && epp < 0.25f;
  constexpr int U = 4;  // particles of a lane whose loads are in flight together
  for (int w = warp; w < ntx * nty; w += kWarpsPerBlock) {
    const int t = (ty0 + w / ntx) * g.ntx + tx0 + w % ntx;
    const int cnt = min(d.cnt[buf][t], g.tile_cap), base = t * g.tile_cap;
    for (int p0 = lane; p0 - lane < cnt; p0 += 32 * U) {
      int cell[U];
      T ox[U], vx[U];
      bool take[U];
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int gi = base + p0 + 32 * r;
        take[r] = p0 + 32 * r < cnt;
        if (take[r] && species >= 0) take[r] = ((P.id[gi] & kIdCR) ? 1 : 0) == species;
        cell[r] = take[r] ? P.cell[gi] : 0;
        ox[r] = take[r] ? P.ox[gi] : (T)0;
        vx[r] = take[r] ? P.vx[gi] : (T)0;
      }
#pragma unroll
      for (int r = 0; r < U; ++r) {
        if (!__any_sync(0xffffffffu, take[r])) continue;
        const int i = cell[r] & 0xFFFF;
        const float tx = fmaf((float)(i - i0) + near_float(ox[r]), fsx, fx0);
        const float tp = (near_float(vx[r]) - pmin) * fsp;
        const float bxf = floorf(tx), bpf = floorf(tp);
        const float rx = tx - bxf, rp = tp - bpf;
        int bx = 0, bp = -1;
        if (fast && fabsf(tp) < 1e6f && rx > epx && rx < 1.0f - epx && rp > epp &&
            rp < 1.0f - epp) {
          bp = (int)bpf;
          bx = bx0 + (int)bxf;
        } else if (take[r]) {
          bx = (int)floor(((double)i + (double)ox[r]) * hsx);
          const double bpd = floor(((double)vx[r] - ph.hist_pmin) * hsp);
          if (bpd >= 0.0 && bpd < (double)np) bp = (int)bpd;
        }
        bx = min(max(bx, 0), ph.hist_nx - 1);
        const bool ok = take[r] && bp >= 0 && bp < np;
        const bool here = (unsigned)(bx - bx0) < (unsigned)nbx;
        count_shared(sh, ok && here ? (bx - bx0) * np + bp : -1);
        if (ok && !here) atomicAdd(&d.hist[(size_t)bx * np + bp], 1ull);
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nbx * np; k += kBlock)
    if (sh[k]) atomicAdd(&d.hist[(size_t)(bx0 + k / np) * np + k % np], (unsigned long long)sh[k]);
}

// Grid export / import in FP64 host layout ([row][col][component]), points
// q0 .. q0 + n - 1 of a grid of npts; nothing is exported from a run with an
// error.
template <typename T>
__global__ void k_export_grid(const T* src, int planes, int npts, int q0, int n, double* dst,
                              const Counters* ctr) {
  if (ctr->status) return;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n;
       q += gridDim.x * blockDim.x)
    for (int c = 0; c < planes; ++c)
      dst[(size_t)q * planes + c] = (double)src[(size_t)c * npts + q0 + q];
}

template <typename T>
__global__ void k_import_B(T* B, const double* src, int nc, int q0, int n) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n;
       q += gridDim.x * blockDim.x)
    for (int c = 0; c < 3; ++c) B[(size_t)c * nc + q0 + q] = (T)src[(size_t)q * 3 + c];
}

// The live particles k0 .. k0 + m - 1 of buffer buf, numbered in tile order
// (off: the tiles' first numbers), as contiguous FP64 columns: one warp per
// tile. Bound by HBM; it replaces seven small device-to-host copies per tile
// (1 M particles in 2458 tiles: the checkpoint's read-back, 138 ms in all
// with its restart, was almost all of them): 61 us.
template <typename T, int DIM>
__global__ void __launch_bounds__(kBlock)
    k_pack_columns(DevPtrs<T> d, Geo g, int buf, const int* __restrict__ off, int k0, int m,
                   Columns dst) {
  const Parts<T> P = d.P[buf];
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5); t < g.ntiles;
       t += gridDim.x * kWarpsPerBlock) {
    const int cnt = min(d.cnt[buf][t], g.tile_cap), base = t * g.tile_cap;
    const int o = off[t] - k0;
    for (int p = max(0, -o) + lane; p < cnt && o + p < m; p += 32) {
      const int gi = base + p, q = o + p;
      const int cell = P.cell[gi];
      dst.ci[q] = cell & 0xFFFF;
      dst.cj[q] = cell >> 16;
      dst.id[q] = P.id[gi];
      dst.col[0][q] = (double)P.ox[gi];
      dst.col[1][q] = DIM == 2 ? (double)P.oy[gi] : 0.0;
      dst.col[2][q] = (double)P.vx[gi];
      dst.col[3][q] = (double)P.vy[gi];
      dst.col[4][q] = (double)P.vz[gi];
    }
  }
}

}  // namespace fsx
