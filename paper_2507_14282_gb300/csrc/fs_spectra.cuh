// fs_spectra.cuh -- diagnostics of the paper's Sec. 3: transversely averaged
// lineouts of Bx, By, Bz and the perpendicular power spectrum
// < |F_perp(k_x, y)|^2 > = |F[By]|^2 + |F[Bz]|^2 averaged over y (Sec. 3.1,
// Fig. 3 caption), F the DFT along x normalised by 1/nx; and the momentum
// spectrum n(p) of the particles (the CR spectra of Sec. 3). FP64 in every
// precision; not on the per-step path.
//
// The spectrum packs each row into one complex sequence z = By + i Bz: for
// real By, Bz, F[By](k) = (Z(k) + conj Z(-k)) / 2 and F[Bz](k) =
// (Z(k) - conj Z(-k)) / 2i, so |F[By]|^2 + |F[Bz]|^2 = (|Z(k)|^2 +
// |Z(-k)|^2) / 2 with Z = F[z]. Rows of up to kFftMax cells are transformed
// in shared memory by a mixed-radix Cooley-Tukey FFT (one CTA per row); rows
// that are longer, or whose large prime factors would make that slower, by a
// direct DFT.
#pragma once
#include <algorithm>

#include "fs_engine.cuh"

namespace fsx {

constexpr int kFftMax = 14400;    // complex doubles in shared memory: 225 KB
constexpr int kFftThreads = 512;
constexpr int kFftPasses = 16;

// The passes of a row of n cells: n = r0 * rad[0] * ... * rad[np - 1]. The
// first pass (r0 points, no twiddles) reads the row from global memory; r0 is
// the product of the prime factors above 7 when there are any (summed term by
// term), else one of the radices 4, 2, 3, 5, 7.
struct FftPlan {
  int n, r0, np;
  int rad[kFftPasses];
};
// false: the row is left to the direct DFT
inline bool fft_plan(int n, int ny, FftPlan* f) {
  f->n = n;
  f->np = 0;
  if (n > kFftMax) return false;
  int m = n;
  const int radices[5] = {4, 2, 3, 5, 7};
  int list[kFftPasses], c = 0;
  for (int r : radices)
    while (m % r == 0) {
      m /= r;
      list[c++] = r;
    }
  int first = 0;
  f->r0 = m;
  if (m == 1) {
    f->r0 = list[0];
    first = 1;
  } else if (m > 64) {
    // FP64 operations per SM: the term-by-term first pass, one CTA per row
    // (4 per term), against the DFT's 14 per term spread over every SM as far
    // as it has threads. 1002 x 150 cells (r0 = 167): FFT 4 x fewer.
    const double t_fft = (double)((ny + 151) / 152) * 4.0 * n * (m + 16.0);
    const double dft_threads = 0.5 * n * ny;
    const double t_dft = 7.0 * n * n * ny / 152.0 * std::max(1.0, 152.0 * 512.0 / dft_threads);
    if (t_fft > t_dft) return false;
  }
  for (int k = first; k < c; ++k) f->rad[f->np++] = list[k];
  return true;
}

// y-averaged B: out[i * 3 + c] = (1/ny) sum_j B_c(i, j), rows in order. One
// warp per block (a column block per SM) with 16 rows' loads in flight:
// latency-bound at a few rows in flight, 17 blocks: 4096 x 256 cells 191 us
// before, 20 us now.
constexpr int kProfThreads = 32;
template <typename T>
__global__ void __launch_bounds__(kProfThreads)
    k_profile_B(const T* __restrict__ B, int nx, int ny, double* __restrict__ out) {
  const size_t nc = (size_t)nx * ny;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= 3 * nx) return;
  const int c = q / nx, i = q - c * nx;
  const T* src = B + c * nc + i;
  double a = 0.0;
#pragma unroll 16
  for (int j = 0; j < ny; ++j) a += (double)src[(size_t)j * nx];
  out[3 * i + c] = a / (double)ny;
}

// y-averaged n at nodes, rows summed in order
template <typename T>
__global__ void __launch_bounds__(kProfThreads)
    k_profile_n(const T* __restrict__ n, int nxn, int ny, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nxn) return;
  double acc = 0.0;
#pragma unroll 16
  for (int j = 0; j < ny; ++j) acc = acc + (double)n[(size_t)j * nxn + i];
  out[i] = acc / (double)ny;
}

// y-averaged |B - B0|^2 at centres, rows summed in order. A CTA takes 32
// columns: its warps form the terms of 64 rows in shared memory, then the
// first adds them in row order (an FP64 instruction holds an SM quarter's
// pipe for some 64 cycles, so one warp doing both is bound by its own
// chain: 4096 x 256 cells 108 us).
constexpr int kDb2Rows = 64;
template <typename T>
__global__ void __launch_bounds__(kBlock)
    k_profile_db2(const T* __restrict__ B, int nx, int ny, double b0x, double b0y, double b0z,
                  double* __restrict__ out) {
  __shared__ double term[kDb2Rows][32];
  const size_t nc = (size_t)nx * ny;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  double a2 = 0.0;
  for (int j0 = 0; j0 < ny; j0 += kDb2Rows) {
    const int nr = min(kDb2Rows, ny - j0);
    if (i < nx) {
#pragma unroll 4
      for (int r = warp; r < nr; r += kWarpsPerBlock) {
        const size_t c = (size_t)(j0 + r) * nx + i;
        const double dbx = (double)B[c] - b0x;
        const double dby = (double)B[nc + c] - b0y;
        const double dbz = (double)B[2 * nc + c] - b0z;
        term[r][lane] = (dbx * dbx + dby * dby) + dbz * dbz;
      }
    }
    __syncthreads();
    if (warp == 0)
      for (int r = 0; r < nr; ++r) a2 = a2 + term[r][lane];
    __syncthreads();
  }
  if (warp == 0 && i < nx) out[i] = a2 / (double)ny;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ double2 cmul_f(double2 a, double2 b) {
  return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)),
                      __fma_rn(a.x, b.y, __dmul_rn(a.y, b.x)));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}

// the row's contribution to P[k] from Z(k) and Z(nx - k); P is pre-zeroed,
// scale = 1 / (2 nx^2 ny)
__device__ __forceinline__ void add_power(double* P, int k, double2 zk, double2 zm,
                                          double scale) {
  const double s = (zk.x * zk.x + zk.y * zk.y) + (zm.x * zm.x + zm.y * zm.y);
  atomicAdd(&P[k], s * scale);
}

// W[j] = exp(-2 pi i j / n): every pass's twiddles are entries of it
static __global__ void k_fft_twiddles(double2* __restrict__ W, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  double2 w;
  sincospi(-2.0 * (double)j / (double)n, &w.y, &w.x);
  W[j] = w;
}

// R-point DFT in registers, R in {2, 3, 4, 5, 7}; the odd radices pair x_s
// with x_{R-s}, cs[k - 1] = exp(-2 pi i k / R) for k = 1 .. (R - 1) / 2
template <int R>
__device__ __forceinline__ void dft_small(double2 (&x)[R], const double2* cs) {
  if constexpr (R == 2) {
    const double2 a = x[0], b = x[1];
    x[0] = cadd(a, b);
    x[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const double2 a = cadd(x[0], x[2]), b = csub(x[0], x[2]);
    const double2 c = cadd(x[1], x[3]), d = csub(x[1], x[3]);
    x[0] = cadd(a, c);
    x[2] = csub(a, c);
    x[1] = make_double2(b.x + d.y, b.y - d.x);  // b - i d
    x[3] = make_double2(b.x - d.y, b.y + d.x);
  } else {
    constexpr int H = (R - 1) / 2;
    double2 p[H], m[H];
    double2 sum = x[0];
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      p[s - 1] = cadd(x[s], x[R - s]);
      m[s - 1] = csub(x[s], x[R - s]);
      sum = cadd(sum, p[s - 1]);
    }
    const double2 x0 = x[0];
    x[0] = sum;
#pragma unroll
    for (int q = 1; q <= H; ++q) {
      double2 a = x0, b = make_double2(0.0, 0.0);
#pragma unroll
      for (int s = 1; s <= H; ++s) {
        const int k = (q * s) % R;
        const double co = cs[(k <= H ? k : R - k) - 1].x;
        const double si = k <= H ? cs[k - 1].y : -cs[R - k - 1].y;  // -sin
        a.x = __fma_rn(co, p[s - 1].x, a.x);
        a.y = __fma_rn(co, p[s - 1].y, a.y);
        b.x = __fma_rn(si, m[s - 1].x, b.x);
        b.y = __fma_rn(si, m[s - 1].y, b.y);
      }
      // X_q = a + i b (b holds the -sin sums), X_{R-q} = a - i b
      x[q] = make_double2(a.x - b.y, a.y + b.x);
      x[R - q] = make_double2(a.x + b.y, a.y - b.x);
    }
  }
}

template <int R>
__device__ __forceinline__ void fft_roots(const double2* __restrict__ W, int n, double2 (&cs)[3]) {
  if constexpr (R == 3 || R == 5 || R == 7) {
#pragma unroll
    for (int k = 1; k <= (R - 1) / 2; ++k) cs[k - 1] = W[k * (n / R)];
  }
}

// One pass of radix R over transforms of length m already in z (in place)
template <int R>
__device__ __forceinline__ void fft_pass(double2* z, const double2* __restrict__ W, int n, int m) {
  double2 cs[3];
  fft_roots<R>(W, n, cs);
  const int tw = n / (m * R);
  for (int t = threadIdx.x; t < n / R; t += blockDim.x) {
    const int blk = t / m, j = t - blk * m;
    double2* p = z + (size_t)blk * m * R + j;
    double2 x[R];
    x[0] = p[0];
#pragma unroll
    for (int q = 1; q < R; ++q) x[q] = cmul_f(p[q * m], W[j * q * tw]);
    dft_small<R>(x, cs);
#pragma unroll
    for (int q = 0; q < R; ++q) p[q * m] = x[q];
  }
}

// position (in blocks of r0) of the first-pass transform of the points
// i, i + n / r0, i + 2 n / r0, ...: the digits of i in the later radices, reversed
__device__ __forceinline__ int fft_block(const FftPlan& f, int i) {
  int size = f.n / f.r0, b = 0;
  for (int k = f.np - 1; k >= 0; --k) {
    const int r = f.rad[k], d = i / r, q = i - d * r;
    i = d;
    size /= r;
    b += q * size;
  }
  return b;
}

template <typename T, int R>
__device__ __forceinline__ void fft_first(double2* z, const double2* __restrict__ W,
                                          const FftPlan& f, const T* by, const T* bz) {
  double2 cs[3];
  fft_roots<R>(W, f.n, cs);
  const int m = f.n / R;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double2 x[R];
#pragma unroll
    for (int s = 0; s < R; ++s)
      x[s] = make_double2((double)by[i + s * m], (double)bz[i + s * m]);
    dft_small<R>(x, cs);
    double2* p = z + (size_t)fft_block(f, i) * R;
#pragma unroll
    for (int s = 0; s < R; ++s) p[s] = x[s];
  }
}

// One CTA per row j; dynamic shared memory n double2; W: n twiddles.
// Bound by the FP64 pipe (about 170 K operations for 4096 cells) and the
// barriers of its passes; twiddles come from one table per call instead of a
// sincospi per radix-2 butterfly, and radix 4 does two levels per pass.
// 4096 x 256 cells FP64: 759 -> 126 us; 3000 x 250 cells (a direct DFT before):
// 34.9 ms -> 116 us.
template <typename T>
__global__ void __launch_bounds__(kFftThreads)
    k_bperp_fft(const T* __restrict__ B, int ny, FftPlan f, const double2* __restrict__ W,
                double* __restrict__ P) {
  extern __shared__ double2 z[];
  const int n = f.n;
  const size_t nc = (size_t)n * ny;
  const T* by = B + nc + (size_t)blockIdx.x * n;
  const T* bz = B + 2 * nc + (size_t)blockIdx.x * n;
  if (f.r0 == 4) {
    fft_first<T, 4>(z, W, f, by, bz);
  } else if (f.r0 == 2) {
    fft_first<T, 2>(z, W, f, by, bz);
  } else if (f.r0 == 3) {
    fft_first<T, 3>(z, W, f, by, bz);
  } else if (f.r0 == 5) {
    fft_first<T, 5>(z, W, f, by, bz);
  } else if (f.r0 == 7) {
    fft_first<T, 7>(z, W, f, by, bz);
  } else {  // term by term: point q of the r0-point transform of block b
    const int m = n / f.r0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const int i = t / f.r0, q = t - i * f.r0;
      double2 a = make_double2(0.0, 0.0);
      int k = 0;  // (q s) mod r0
      for (int s = 0; s < f.r0; ++s) {
        const double2 w = W[k * m];
        const double vy = (double)by[i + s * m], vz = (double)bz[i + s * m];
        a.x = __fma_rn(vy, w.x, __fma_rn(-vz, w.y, a.x));
        a.y = __fma_rn(vy, w.y, __fma_rn(vz, w.x, a.y));
        k += q;
        if (k >= f.r0) k -= f.r0;
      }
      z[(size_t)fft_block(f, i) * f.r0 + q] = a;
    }
  }
  __syncthreads();
  int m = f.r0;
  for (int k = 0; k < f.np; ++k) {
    const int r = f.rad[k];
    if (r == 4) fft_pass<4>(z, W, n, m);
    else if (r == 2) fft_pass<2>(z, W, n, m);
    else if (r == 3) fft_pass<3>(z, W, n, m);
    else if (r == 5) fft_pass<5>(z, W, n, m);
    else fft_pass<7>(z, W, n, m);
    m *= r;
    __syncthreads();
  }
  const double scale = 0.5 / ((double)n * (double)n * (double)ny);
  for (int k = threadIdx.x; k <= n / 2; k += blockDim.x)
    add_power(P, k, z[k], z[k == 0 ? 0 : n - k], scale);
}

// Direct DFT, one thread per (k, row): Z(k) and Z(nx - k) as sums over x
// with the phase step multiplied in and re-anchored every 64 terms.
template <typename T>
__global__ void k_bperp_dft(const T* __restrict__ B, int nx, int ny, double* __restrict__ P) {
  const int nk = nx / 2 + 1;
  const size_t nc = (size_t)nx * ny;
  const double scale = 0.5 / ((double)nx * (double)nx * (double)ny);
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (long long)nk * ny;
       q += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(q % nk), j = (int)(q / nk);
    const T* by = B + nc + (size_t)j * nx;
    const T* bz = B + 2 * nc + (size_t)j * nx;
    double2 zk = make_double2(0.0, 0.0), zm = make_double2(0.0, 0.0);
    double2 w = make_double2(1.0, 0.0), step;
    sincospi(-2.0 * (double)k / (double)nx, &step.y, &step.x);
    for (int x = 0; x < nx; ++x) {
      if ((x & 63) == 0) {  // exact phase exp(-2 pi i k x / nx) from the integer k x mod nx
        const long long kx = ((long long)k * x) % nx;
        sincospi(-2.0 * (double)kx / (double)nx, &w.y, &w.x);
      }
      const double2 v = make_double2((double)by[x], (double)bz[x]);
      const double2 a = cmul(v, w);                              // v exp(-i theta)
      const double2 b = cmul(v, make_double2(w.x, -w.y));        // v exp(+i theta): Z(-k)
      zk.x += a.x; zk.y += a.y;
      zm.x += b.x; zm.y += b.y;
      w = cmul(w, step);
    }
    add_power(P, k, zk, zm, scale);
  }
}

// Momentum spectrum n(p): counts of |u| between the log-spaced edges
// e[0..np] (e[k] <= |u| < e[k+1]); species -1 all, 1 cosmic rays only.
// Integer counts. The bin is first formed in FP32 from log2(u.u) with
// l2min = log2 e[0], per = np / log2(e[np]/e[0]); only a value within eps
// of a bin edge (or beyond FP32's range) takes the exact comparisons with
// |u| = sqrt(u.u) in FP64, which the narrow FP64 pipe makes expensive. Counts
// are kept per warp in shared memory (sh: bins * copies words, copies =
// warps or 1; 0: no shared counts, very many bins): a drifting thermal plasma
// puts most particles in a few bins, whose global atomics serialise.
// 17.8 M particles FP64: 4089 -> 69 us.
constexpr int kSpecShared = 8192;  // shared counters at most
template <typename T>
__global__ void __launch_bounds__(kBlock)
    k_spectrum_p(DevPtrs<T> d, Geo g, int buf, int species, int np, int copies, float l2min,
                 float per, float eps, const double* __restrict__ e,
                 unsigned long long* __restrict__ out) {
  extern __shared__ unsigned sh[];
  const Parts<T> P = d.P[buf];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < np * copies; k += kBlock) sh[k] = 0u;
  __syncthreads();
  unsigned* mine = sh + (copies > 1 ? warp * np : 0);
  for (int t = blockIdx.x * kWarpsPerBlock + warp; t < g.ntiles;
       t += gridDim.x * kWarpsPerBlock) {
    const int cnt = min(d.cnt[buf][t], g.tile_cap), base = t * g.tile_cap;
    constexpr int U = 4;  // particles of a lane whose loads are in flight together
    for (int p0 = lane; p0 - lane < cnt; p0 += 32 * U) {
      T vx[U], vy[U], vz[U];
      bool take[U];
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int gi = base + p0 + 32 * r;
        take[r] = p0 + 32 * r < cnt;
        if (take[r] && species == 1) take[r] = (P.id[gi] & kIdCR) != 0;
        vx[r] = take[r] ? P.vx[gi] : (T)0;
        vy[r] = take[r] ? P.vy[gi] : (T)0;
        vz[r] = take[r] ? P.vz[gi] : (T)0;
      }
#pragma unroll
      for (int r = 0; r < U; ++r) {
        if (!__any_sync(0xffffffffu, take[r])) continue;
        const float fx = near_float(vx[r]), fy = near_float(vy[r]), fz = near_float(vz[r]);
        const float p2 = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
        const float tb = (0.5f * __log2f(p2) - l2min) * per;
        const float fb = floorf(tb), fr = tb - fb;
        int bin = -1;
        if (p2 > 1e-30f && p2 < 1e30f && fr > eps && fr < 1.0f - eps) {
          if (fb >= 0.0f && fb < (float)np) bin = (int)fb;
        } else if (take[r]) {
          const double ux = vx[r], uy = vy[r], uz = vz[r];
          const double p = __dsqrt_rn(__fma_rn(uz, uz, __fma_rn(uy, uy, __dmul_rn(ux, ux))));
          if (p >= e[0] && p < e[np]) {
            int lo = 0, hi = np;  // e[lo] <= p < e[hi]
            while (hi - lo > 1) {
              const int mid = (lo + hi) >> 1;
              if (p >= e[mid]) lo = mid; else hi = mid;
            }
            bin = lo;
          }
        }
        if (!take[r] || bin < 0) continue;
        if (copies) atomicAdd(&mine[bin], 1u);
        else atomicAdd(&out[bin], 1ull);
      }
    }
  }
  __syncthreads();
  if (!copies) return;
  for (int k = threadIdx.x; k < np; k += kBlock) {
    unsigned s = 0;
    for (int w = 0; w < copies; ++w) s += sh[w * np + k];
    if (s) atomicAdd(&out[k], (unsigned long long)s);
  }
}

}  // namespace fsx
