// fs_ops.cuh -- launch side of the kernels for one arithmetic type T:
// fills the Ops table used by the C ABI. Instantiated by fs_f32.cu and
// fs_f64.cu (the latter compiled with -fmad=false).
#pragma once
#include <algorithm>
#include <cstring>
#include <mutex>

#include "fs_push.cuh"
#include "fs_spectra.cuh"

namespace fsx {

// one thread per element up to 64 blocks per SM (every kernel launched with
// it strides over the rest)
inline int grid_for(long long n, int block = kBlock) {
  long long g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > 152LL * 64) g = 152LL * 64;
  return (int)g;
}

template <typename T, int DIM, int CH, int NS, bool REL, int TXC = 0, int TYC = 0>
cudaError_t launch_push(Sim* s, int in) {
  const PushLayout<T, DIM> L(s->g.TX, s->g.TY, CH, NS);
  // per kernel instance: the occupancy at the last size asked for (host threads
  // may share it)
  static std::mutex mu;
  static size_t occ_bytes = 0;
  static int occ_blocks_c = 1, n_sm_c = 0;
  int occ_blocks, n_sm;
  {
    std::lock_guard<std::mutex> lock(mu);
    const cudaError_t er = raise_smem<k_push<T, DIM, CH, NS, REL, TXC, TYC>>(L.bytes);
    if (er != cudaSuccess) return er;
    if (L.bytes != occ_bytes) {
      int dev = 0, nsm = 0, occ = 0;
      cudaError_t e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_push<T, DIM, CH, NS, REL, TXC, TYC>,
                                                          kBlock, L.bytes);
      if (e != cudaSuccess) return e;
      if (occ < 1) return cudaErrorInvalidConfiguration;
      n_sm_c = nsm;
      occ_blocks_c = occ;
      occ_bytes = L.bytes;
    }
    occ_blocks = occ_blocks_c;
    n_sm = n_sm_c;
  }
  StepArgs a;
  a.g = s->g;
  a.ph = s->ph;
  a.in = in;
  a.out = 1 - in;
  const int per_sm = s->g.push_ctas > 0 ? std::min(occ_blocks, s->g.push_ctas) : occ_blocks;
  const long long want = (long long)n_sm * per_sm;
  const int grid = (int)std::min<long long>(want, s->g.ntiles);
  k_push<T, DIM, CH, NS, REL, TXC, TYC><<<grid, kBlock, L.bytes, s->stream>>>(
      s->ptrs<T>(in), a, push_const<T>(s->ph));
  return cudaGetLastError();
}

// shared-memory chunk (particles) and pipeline stages per precision
template <typename T>
struct PushShape;
template <>
struct PushShape<float> {
  static constexpr int kChunkSmall = 512, kStagesSmall = 3;
  static constexpr int kChunkLarge = 576, kStagesLarge = 2;
};
template <>
struct PushShape<double> {
  static constexpr int kChunkSmall = 512, kStagesSmall = 2;
  static constexpr int kChunkLarge = 512, kStagesLarge = 2;
};

template <typename T, int DIM>
cudaError_t push_dispatch(Sim* s, int in) {
  using S = PushShape<T>;
  // the relativistic terms are compiled in only for runs with a finite c
  if (s->ph.c2inv > 0.0) {
    if (s->g.chunk == S::kChunkSmall)
      return launch_push<T, DIM, S::kChunkSmall, S::kStagesSmall, true>(s, in);
    return launch_push<T, DIM, S::kChunkLarge, S::kStagesLarge, true>(s, in);
  }
  if (s->g.chunk == S::kChunkSmall)
    return launch_push<T, DIM, S::kChunkSmall, S::kStagesSmall, false>(s, in);
  // The 2D FP32 tile shape the library picks at 64 ppc (4 x 2 cells), compiled
  // in: every layout offset and tile constant of the push becomes an
  // immediate (7.11 -> 6.67 ms on the 268 M-particle precision form; the
  // FP64 push, bound by its FP64 pipe, gains nothing from the same).
  if constexpr (DIM == 2 && sizeof(T) == 4) {
    if (s->g.TX == 4 && s->g.TY == 2)
      return launch_push<T, DIM, S::kChunkLarge, S::kStagesLarge, false, 4, 2>(s, in);
  }
  return launch_push<T, DIM, S::kChunkLarge, S::kStagesLarge, false>(s, in);
}

template <typename T>
struct OpsImpl {
  static DevPtrs<T> P(Sim* s) { return s->ptrs<T>(); }

  static cudaError_t init_particles(Sim* s) {
    const long long total = (long long)s->g.nx * s->g.ny * s->p.ppc;
    if (s->g.dim == 1)
      k_init_particles<T, 1><<<grid_for(total), kBlock, 0, s->stream>>>(P(s), s->g, s->ph, s->cur, s->p.ppc);
    else
      k_init_particles<T, 2><<<grid_for(total), kBlock, 0, s->stream>>>(P(s), s->g, s->ph, s->cur, s->p.ppc);
    return cudaGetLastError();
  }

  static cudaError_t deposit_all(Sim* s, int buf) {
    using A = typename Num<T>::acc;
    const size_t na = (size_t)s->g.ntiles * 4 * s->g.na;
    cudaError_t e = cudaMemsetAsync(s->base + s->L.partial, 0, na * sizeof(A), s->stream);
    if (e != cudaSuccess) return e;
    if (s->g.dim == 1)
      k_deposit_all<T, 1><<<s->g.ntiles, kBlock, 0, s->stream>>>(P(s), s->g, s->ph, buf);
    else
      k_deposit_all<T, 2><<<s->g.ntiles, kBlock, 0, s->stream>>>(P(s), s->g, s->ph, buf);
    return cudaGetLastError();
  }

  static cudaError_t moments(Sim* s) {
    const long long nn = (long long)s->g.nxn * s->g.ny;
    const Geo& g = s->g;
    // boxes with x walls that are more than a tile's accumulator high and more
    // than three tile rows: a fixed set of candidate tiles per node; the shapes
    // the library picks for the benchmark's 2D workloads (FP32 4 x 2 at 64 ppc,
    // FP64 8 x 4 at 16 ppc) compiled in
    const bool ct = g.dim == 2 && g.bc_x != FS_BC_PERIODIC && g.ny >= 2 * (g.TY + 3) && g.nty > 3;
    auto run = [&](auto kern) {
      kern<<<grid_for(nn), kBlock, 0, s->stream>>>(P(s), g, s->ph);
    };
    if (g.dim == 1) run(k_moments<T, 1>);
    else if (!ct) run(k_moments<T, 2>);
    else if (g.TX == 4 && g.TY == 2) run(k_moments_ct<T, 4, 2, 2, 3>);
    else if (g.TX == 8 && g.TY == 4) run(k_moments_ct<T, 8, 4, 2, 2>);
    // tiles that can cover a node: (TX + 3) / TX columns rounded up, rows alike
    else if (g.TX == 2 && g.TY == 1) run(k_moments_ct<T, 0, 0, 3, 4>);
    else if (g.TX == 2 && g.TY == 2) run(k_moments_ct<T, 0, 0, 3, 3>);
    else if (g.TX == 2) run(k_moments_ct<T, 0, 0, 3, 2>);
    else if (g.TY == 1) run(k_moments_ct<T, 0, 0, 2, 4>);
    else if (g.TY == 2) run(k_moments_ct<T, 0, 0, 2, 3>);
    else run(k_moments_ct<T, 0, 0, 2, 2>);
    return cudaGetLastError();
  }

  // Ohm's law at every node, one thread per node (pre: the per-step density
  // terms of k_ohm_pre, or nullptr to form them here)
  template <int DIM>
  static void ohm(Sim* s, const T* Bc, T* Eo, T* Bbo, T* G, const T* pre = nullptr) {
    DevPtrs<T> d = P(s);
    const long long nn = (long long)s->g.nxn * s->g.ny;
    k_ohm<T, DIM><<<grid_for(nn), kBlock, 0, s->stream>>>(Bc, d.n, d.u, pre, Eo, Bbo, G, s->g,
                                                          s->ph);
  }

  static cudaError_t ohm_final(Sim* s) {
    DevPtrs<T> d = P(s);
    if (s->g.dim == 1) ohm<1>(s, d.B, d.E, d.Bb, d.G);
    else ohm<2>(s, d.B, d.E, d.Bb, d.G);
    return cudaGetLastError();
  }

  // 1D boxes with x walls: moments, the whole field advance and the step's end
  // in one tiled launch (k_field_step1).
  static_assert(kF1MaxSub == 16, "Sim::swaps_fields");
  template <int TILE>
  static cudaError_t field_step1(Sim* s, int in) {
    DevPtrs<T> d = s->ptrs<T>(in);
    const size_t smem = field1_smem<T>(s->p.n_sub, TILE);
    const cudaError_t e = raise_smem<k_field_step1<T, TILE>>(smem);
    if (e != cudaSuccess) return e;
    k_field_step1<T, TILE><<<(s->g.nx + TILE - 1) / TILE,
                             field1_threads(TILE, s->p.n_sub), smem, s->stream>>>(
        d, s->g, (T)s->ph.n_floor, field_const<T>(s->ph), s->p.n_sub);
    return cudaGetLastError();
  }
  static cudaError_t fields_tiled1(Sim* s, int in) {
    return field1_tile(s->g.nx) == kF1Small ? field_step1<kF1Small>(s, in)
                                            : field_step1<kF1>(s, in);
  }

  // Rows of a warp's march over ny rows in `strips` strips, each march
  // re-forming `extra` rows: the least work on the fullest SM, among the lengths
  // that give an SM at least `lo` warps (where there are that many rows) and
  // at most the `hi` it holds at once.
  static int march_rows(int strips, int ny, int extra, int lo, int hi) {
    int rows = 1;
    long long best = -1;
    for (int r = 1; r <= 128 && r <= ny; ++r) {
      const long long per_sm = ((long long)strips * ((ny + r - 1) / r) + 151) / 152;
      if (best >= 0 && per_sm < lo) break;
      const long long cost = per_sm * (r + extra);
      if (best >= 0 && cost >= best && per_sm <= hi) continue;
      best = per_sm > hi ? -1 : cost;
      rows = r;
    }
    return rows;
  }

  // FP32 2D: one launch per substep (k_field_substep), B alternating with the
  // stage buffer Bs.
  static cudaError_t fields_substeps(Sim* s) {
    DevPtrs<T> d = P(s);
    const Geo& g = s->g;
    const FieldConst<T> fc = field_const<T>(s->ph);
    T *b = d.B, *bn = d.Bs;
    for (int sub = 0; sub < s->p.n_sub; ++sub) {
      const bool fin = sub + 1 == s->p.n_sub;
      const int strips = fin ? (g.nxn + 21) / 22 : (g.nxn + 22) / 23;
      const int rows = march_rows(strips, g.ny, fin ? 10 : 9, 8, 16);
      const int grid = strips * ((g.ny + rows - 1) / rows);
      if (fin)
        k_field_substep<T, true><<<grid, 32, 0, s->stream>>>(b, bn, d.n, d.u, d.E, d.Bb, d.G, g, fc,
                                                             rows, strips);
      else
        k_field_substep<T, false><<<grid, 32, 0, s->stream>>>(b, bn, d.n, d.u, d.E, d.Bb, d.G, g,
                                                              fc, rows, strips);
      std::swap(b, bn);
    }
    if (b != d.B)  // odd n_sub: the field ended in the stage buffer
      return cudaMemcpyAsync(d.B, b, 3 * sizeof(T) * (size_t)g.nx * g.ny,
                             cudaMemcpyDeviceToDevice, s->stream);
    return cudaGetLastError();
  }

  // FP64 2D: Ohm's E of B, then a marching pass per RK4 stage (k_field_march); E
  // alternates with Es, B with Bs from one substep to the next.
  static cudaError_t fields_march(Sim* s) {
    DevPtrs<T> d = P(s);
    const Geo& g = s->g;
    const FieldConst<T> fc = field_const<T>(s->ph);
    k_ohm_start<T, 2><<<grid_for((long long)g.nxn * g.ny), kBlock, 0, s->stream>>>(
        d.B, d.n, d.u, d.E, d.pre, g, s->ph);
    const int strips = (g.nxn + kMarchCols - 1) / kMarchCols;
    const int rows = march_rows(strips, g.ny, 2, 11, 16);
    const int grid = strips * ((g.ny + rows - 1) / rows);
    T *b = d.B, *bn = d.Bs;
    auto pass = [&](auto kern, const T* ei, T* eo) {
      kern<<<grid, 32, 0, s->stream>>>(ei, eo, b, d.Bsum, bn, d.u, d.pre, d.Bb, d.G, g,
                                                  fc, rows, strips);
    };
    for (int sub = 0; sub < s->p.n_sub; ++sub) {
      pass(k_field_march<T, 1, false>, d.E, d.Es);
      pass(k_field_march<T, 2, false>, d.Es, d.E);
      pass(k_field_march<T, 3, false>, d.E, d.Es);
      if (sub + 1 == s->p.n_sub) pass(k_field_march<T, 4, true>, d.Es, d.E);
      else pass(k_field_march<T, 4, false>, d.Es, d.E);
      std::swap(b, bn);
    }
    if (b != d.B)  // odd n_sub: the field ended in the stage buffer
      return cudaMemcpyAsync(d.B, b, 3 * sizeof(T) * (size_t)g.nx * g.ny,
                             cudaMemcpyDeviceToDevice, s->stream);
    return cudaGetLastError();
  }

  // The field advance of boxes that k_field_step1 does not take: 2D, and 1D
  // periodic ones, whose passes stay one launch each.
  static cudaError_t fields(Sim* s) {
    if (s->g.dim == 2) {
      if constexpr (sizeof(T) == 4) return fields_substeps(s);
      else return fields_march(s);
    }
    DevPtrs<T> d = P(s);
    // FP64 (bound by the FP64 pipe): 1/n and the pressure terms once per step
    const T* pre = nullptr;
    if (sizeof(T) == 8) {
      k_ohm_pre<T, 1><<<grid_for(s->g.nxn), kBlock, 0, s->stream>>>(d.n, d.pre, s->g, s->ph);
      pre = d.pre;
    }
    auto faraday = [&](int stage) {
      k_faraday<T, 1><<<grid_for(s->g.nx), kBlock, 0, s->stream>>>(d.Es, d.B, d.Bs, d.Bsum, stage,
                                                                   s->g, s->ph);
    };
    for (int sub = 0; sub < s->p.n_sub; ++sub)
      for (int stage = 1; stage <= 4; ++stage) {
        ohm<1>(s, stage == 1 ? d.B : d.Bs, d.Es, nullptr, nullptr, pre);
        faraday(stage);
      }
    ohm<1>(s, d.B, d.E, d.Bb, d.G, pre);
    return cudaGetLastError();
  }

  // The draws of the step's injected particles, on st: one block counts and
  // draws when it has few of them, else a count and a grid of draws.
  static cudaError_t inject(Sim* s, int in, cudaStream_t st) {
    DevPtrs<T> d = s->ptrs<T>(in);
    const Geo& g = s->g;
    if (g.ninj <= kBlock) {
      const int threads = (std::max(g.ninj, g.ny) + 31) / 32 * 32;
      if (g.dim == 1) k_inject_run<T, 1><<<1, threads, 0, st>>>(d, g, s->ph);
      else k_inject_run<T, 2><<<1, threads, 0, st>>>(d, g, s->ph);
      return cudaGetLastError();
    }
    const int mult = (s->ph.inject_thermal ? 1 : 0) + (s->ph.cr_enable ? 1 : 0);
    k_inject_count<<<1, 1024, 0, st>>>(d.acc, d.inj, d.inj + g.ny, g.ny, s->ph.rate, mult);
    const int blocks = (g.ninj + 63) / 64;  // a draw is one long FP64 chain: spread them
    if (g.dim == 1) k_inject_draw<T, 1><<<blocks, 64, 0, st>>>(d, g, s->ph);
    else k_inject_draw<T, 2><<<blocks, 64, 0, st>>>(d, g, s->ph);
    return cudaGetLastError();
  }
  static void movers(Sim* s, int out, int what, cudaStream_t st) {
    const int tiles = (what & 1) ? (s->g.ntiles + 7) / 8 : 0;
    const int recs = (what & 2) ? (s->g.ninj + kBlock - 1) / kBlock : 0;
    const int grid = std::max(1, std::min(std::max(tiles, recs), 152 * 16));
    if (s->g.dim == 1) k_movers<T, 1><<<grid, kBlock, 0, st>>>(P(s), s->g, out, what);
    else k_movers<T, 2><<<grid, kBlock, 0, st>>>(P(s), s->g, out, what);
  }

  // Everything of a step after the push (movers, injection unless `drawn`,
  // moments, field advance, step counter); ev as in step().
  static cudaError_t step_rest(Sim* s, int in, cudaEvent_t* ev, bool drawn) {
    DevPtrs<T> d = s->ptrs<T>(in);
    const int out = 1 - in;
    cudaError_t e = cudaSuccess;
    auto mark = [&](int k) {
      if (ev) cudaEventRecord(ev[k], s->stream);
    };
    if (drawn) {
      // the movers (buckets) on the side stream, behind the draws and the push,
      // beside the moments and field advance, which read no bucket; the
      // moments need the draws' deposit
      if ((e = cudaEventRecord(s->ev_push, s->stream)) != cudaSuccess) return e;
      if ((e = cudaStreamWaitEvent(s->side, s->ev_push, 0)) != cudaSuccess) return e;
      movers(s, out, s->g.ninj ? 3 : 1, s->side);
      if ((e = cudaEventRecord(s->ev_join, s->side)) != cudaSuccess) return e;
      if ((e = cudaStreamWaitEvent(s->stream, s->ev_draw, 0)) != cudaSuccess) return e;
    } else {
      movers(s, out, 1, s->stream);
      mark(2);
      if (s->g.ninj) {
        if ((e = inject(s, in, s->stream)) != cudaSuccess) return e;
        movers(s, out, 2, s->stream);
      }
      mark(3);
    }
    const bool one = s->swaps_fields();  // (ends the step, too)
    if (!one && (e = moments(s)) != cudaSuccess) return e;
    mark(4);
    e = one ? fields_tiled1(s, in) : fields(s);
    if (e != cudaSuccess) return e;
    if (drawn && (e = cudaStreamWaitEvent(s->stream, s->ev_join, 0)) != cudaSuccess) return e;
    if (!one) k_step_end<<<1, 32, 0, s->stream>>>(d.ctr, d.inj, s->g);
    mark(5);
    return cudaGetLastError();
  }

  static cudaError_t step(Sim* s, int in, cudaEvent_t* ev) {
    // without phase events (and with the side stream of the captured step):
    // the draws beside the push
    const bool drawn = !ev && s->side && s->ev_fork && s->ev_draw && s->ev_push && s->ev_join;
    cudaError_t e = cudaSuccess;
    if (drawn) {
      if ((e = cudaEventRecord(s->ev_fork, s->stream)) != cudaSuccess) return e;
      if ((e = cudaStreamWaitEvent(s->side, s->ev_fork, 0)) != cudaSuccess) return e;
      if (s->g.ninj && (e = inject(s, in, s->side)) != cudaSuccess) return e;
      if ((e = cudaEventRecord(s->ev_draw, s->side)) != cudaSuccess) return e;
    }
    if (ev) cudaEventRecord(ev[0], s->stream);
    e = (s->g.dim == 1) ? push_dispatch<T, 1>(s, in) : push_dispatch<T, 2>(s, in);
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[1], s->stream);
    return step_rest(s, in, ev, drawn);
  }

  // ---- batched ensembles: one push launch over every run's CTA group
  static size_t batch_run_bytes() { return sizeof(BatchRun<T>); }
  static void fill_batch_run(const Sim* s, int in, int ncta, void* dst) {
    BatchRun<T> r;
    r.d = s->ptrs<T>(in);
    r.g = s->g;
    r.ph = s->ph;
    r.pc = push_const<T>(s->ph);
    r.in = in;
    r.out = 1 - in;
    r.ncta = ncta;
    r.n_sub = s->p.n_sub;
    memcpy(dst, &r, sizeof r);
  }
  // chunk: 0 or the large chunk (PushShape::kChunkLarge, its stages), or
  // the small chunk (kChunkSmall, its stages) for every run of the batch
  static bool batch_small(int chunk) {
    using S = PushShape<T>;
    return chunk == S::kChunkSmall && S::kChunkSmall != S::kChunkLarge;
  }
  static size_t batch_smem(int dim, int tx, int ty, int chunk) {
    using S = PushShape<T>;
    const int ch = batch_small(chunk) ? S::kChunkSmall : S::kChunkLarge;
    const int ns = batch_small(chunk) ? S::kStagesSmall : S::kStagesLarge;
    return dim == 1 ? PushLayout<T, 1>(tx, ty, ch, ns).bytes
                    : PushLayout<T, 2>(tx, ty, ch, ns).bytes;
  }
  template <int DIM, int CH, int NS, bool REL, int TXC = 0>
  static cudaError_t batch_kernel_setup(size_t smem, int* occ) {
    cudaError_t e = raise_smem<k_push_batch<T, DIM, CH, NS, REL, TXC>>(smem);
    if (e == cudaSuccess && occ)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          occ, k_push_batch<T, DIM, CH, NS, REL, TXC>, kBlock, smem);
    return e;
  }
  template <int CH, int NS>
  static cudaError_t batch_setup_shape(int dim, int rel, size_t smem, int* occ) {
    if (rel)
      return dim == 1 ? batch_kernel_setup<1, CH, NS, true>(smem, occ)
                      : batch_kernel_setup<2, CH, NS, true>(smem, occ);
    return dim == 1 ? batch_kernel_setup<1, CH, NS, false>(smem, occ)
                    : batch_kernel_setup<2, CH, NS, false>(smem, occ);
  }
  // sets the shared-memory attribute; occ (optional): CTAs per SM. rel: the
  // variant with the relativistic terms (some run has a finite c).
  // the 1D FP32 tile widths compiled into their own batched push
  static bool batch_width_compiled(int dim, int rel, int chunk, int txc) {
    return sizeof(T) == 4 && dim == 1 && !rel && !batch_small(chunk) &&
           (txc == 4 || txc == 8 || txc == 16);
  }
  static cudaError_t batch_setup(int dim, int rel, int chunk, int txc, size_t smem, int* occ) {
    using S = PushShape<T>;
    if (batch_width_compiled(dim, rel, chunk, txc)) {
      constexpr int CH = S::kChunkLarge, NS = S::kStagesLarge;
      if (txc == 4) return batch_kernel_setup<1, CH, NS, false, 4>(smem, occ);
      if (txc == 8) return batch_kernel_setup<1, CH, NS, false, 8>(smem, occ);
      return batch_kernel_setup<1, CH, NS, false, 16>(smem, occ);
    }
    if (batch_small(chunk))
      return batch_setup_shape<S::kChunkSmall, S::kStagesSmall>(dim, rel, smem, occ);
    return batch_setup_shape<S::kChunkLarge, S::kStagesLarge>(dim, rel, smem, occ);
  }
  template <int CH, int NS, bool REL>
  static void push_batch_launch(int dim, const BatchRun<T>* r, const int2* cta_map, int ncta,
                                size_t smem, cudaStream_t st) {
    if (dim == 1)
      k_push_batch<T, 1, CH, NS, REL><<<ncta, kBlock, smem, st>>>(r, cta_map);
    else
      k_push_batch<T, 2, CH, NS, REL><<<ncta, kBlock, smem, st>>>(r, cta_map);
  }
  static cudaError_t push_batch(int dim, int rel, int chunk, int txc, const void* runs,
                                const int2* cta_map, int ncta, size_t smem, cudaStream_t st) {
    using S = PushShape<T>;
    const BatchRun<T>* r = (const BatchRun<T>*)runs;
    if (batch_width_compiled(dim, rel, chunk, txc)) {
      constexpr int CH = S::kChunkLarge, NS = S::kStagesLarge;
      if (txc == 4) k_push_batch<T, 1, CH, NS, false, 4><<<ncta, kBlock, smem, st>>>(r, cta_map);
      else if (txc == 8) k_push_batch<T, 1, CH, NS, false, 8><<<ncta, kBlock, smem, st>>>(r, cta_map);
      else k_push_batch<T, 1, CH, NS, false, 16><<<ncta, kBlock, smem, st>>>(r, cta_map);
      return cudaGetLastError();
    }
    const bool sm = batch_small(chunk);
    if (rel) {
      if (sm) push_batch_launch<S::kChunkSmall, S::kStagesSmall, true>(dim, r, cta_map, ncta, smem, st);
      else push_batch_launch<S::kChunkLarge, S::kStagesLarge, true>(dim, r, cta_map, ncta, smem, st);
    } else {
      if (sm) push_batch_launch<S::kChunkSmall, S::kStagesSmall, false>(dim, r, cta_map, ncta, smem, st);
      else push_batch_launch<S::kChunkLarge, S::kStagesLarge, false>(dim, r, cta_map, ncta, smem, st);
    }
    return cudaGetLastError();
  }

  // a batched step over every run (all 1D with x walls): the draws, the rest
  static cudaError_t batch_draw(const void* runs, int nruns, cudaStream_t st) {
    k_inject_batch<T, 1><<<nruns, kBlock, 0, st>>>((const BatchRun<T>*)runs, nruns);
    return cudaGetLastError();
  }
  static cudaError_t batch_rest(const void* runs, const int* pre, int nruns, const int* nblk,
                                int n_sub_max, cudaStream_t st, cudaStream_t side,
                                cudaEvent_t fork, cudaEvent_t join) {
    const BatchRun<T>* r = (const BatchRun<T>*)runs;
    const size_t fsm = field1_smem<T>(n_sub_max, kF1);
    cudaError_t e = raise_smem<k_field1_batch<T>>(fsm);
    if (e != cudaSuccess) return e;
    const int n1 = nruns + 1;
    // the movers (buckets) beside the moments and field advance, which read
    // the deposit partials and far sums and no bucket
    if ((e = cudaEventRecord(fork, st)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(side, fork, 0)) != cudaSuccess) return e;
    k_movers_batch<T, 1><<<nblk[0], kBlock, 0, side>>>(r, pre, nruns);
    if ((e = cudaEventRecord(join, side)) != cudaSuccess) return e;
    k_field1_batch<T><<<nblk[1], field1_threads(kF1, n_sub_max), fsm, st>>>(r, pre + n1, nruns);
    if ((e = cudaStreamWaitEvent(st, join, 0)) != cudaSuccess) return e;
    return cudaGetLastError();
  }

  static cudaError_t insert_columns(Sim* s, int buf, const Columns& src, int n,
                                    const uint32_t* ids, unsigned long long first) {
    DevPtrs<T> d = P(s);
    if (s->g.dim == 1)
      k_insert_columns<T, 1><<<grid_for(n), kBlock, 0, s->stream>>>(d, src, s->g, buf, n, ids, first);
    else
      k_insert_columns<T, 2><<<grid_for(n), kBlock, 0, s->stream>>>(d, src, s->g, buf, n, ids, first);
    return cudaGetLastError();
  }

  static cudaError_t scan_counts(Sim* s, int buf) {
    DevPtrs<T> d = P(s);
    k_scan_counts<<<1, 1024, 0, s->stream>>>(d.cnt[buf], s->g.ntiles, s->g.tile_cap, d.mcnt,
                                             &d.ctr->live);
    return cudaGetLastError();
  }

  static cudaError_t pack_columns(Sim* s, int buf, int k0, int m, const Columns& dst) {
    DevPtrs<T> d = P(s);
    if (s->g.dim == 1)
      k_pack_columns<T, 1><<<tile_warps_grid(s), kBlock, 0, s->stream>>>(d, s->g, buf, d.mcnt, k0,
                                                                         m, dst);
    else
      k_pack_columns<T, 2><<<tile_warps_grid(s), kBlock, 0, s->stream>>>(d, s->g, buf, d.mcnt, k0,
                                                                         m, dst);
    return cudaGetLastError();
  }

  // CTAs of a kernel whose warps stride over the tiles
  static int tile_warps_grid(Sim* s) {
    return std::max(1, std::min((s->g.ntiles + kWarpsPerBlock - 1) / kWarpsPerBlock, 152 * 8));
  }

  static cudaError_t diag(Sim* s, int buf) {
    DevPtrs<T> d = P(s);
    cudaError_t e = cudaMemsetAsync(d.ctr->sums, 0, sizeof(d.ctr->sums), s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(&d.ctr->live, 0, sizeof(d.ctr->live), s->stream);
    if (e != cudaSuccess) return e;
    if (s->g.dim == 1)
      k_diag_particles<T, 1><<<tile_warps_grid(s), kBlock, 0, s->stream>>>(d, s->g, s->ph, buf);
    else
      k_diag_particles<T, 2><<<tile_warps_grid(s), kBlock, 0, s->stream>>>(d, s->g, s->ph, buf);
    // several nodes per thread, so that few of them take the FP64 expression
    const int grid = std::min(grid_for((long long)s->g.nx * s->g.ny), 152 * 4);
    k_diag_field<T><<<grid, kBlock, 0, s->stream>>>(d, s->g, s->ph);
    return cudaGetLastError();
  }

  static cudaError_t hist(Sim* s, int buf, int species) {
    DevPtrs<T> d = P(s);
    const Geo& g = s->g;
    cudaError_t e = cudaMemsetAsync(d.hist, 0,
                                    sizeof(unsigned long long) * s->ph.hist_nx * s->ph.hist_np,
                                    s->stream);
    if (e != cudaSuccess) return e;
    const int gx = g.dim == 1 ? kWarpsPerBlock : 1, gy = g.dim == 1 ? 1 : 4 * kWarpsPerBlock;
    const dim3 grid((g.ntx + gx - 1) / gx, (g.nty + gy - 1) / gy);
    // x bins a CTA's cells can reach: a span of gx TX cells anywhere in the box
    const long long span =
        (long long)ceil((double)gx * g.TX * s->ph.hist_nx / (double)g.nx) + 2;
    const int nbx = span * s->ph.hist_np <= kHistShared ? (int)span : 0;
    const size_t smem = sizeof(unsigned) * (size_t)nbx * s->ph.hist_np;
    if (g.dim == 1)
      k_hist<T, 1><<<grid, kBlock, smem, s->stream>>>(d, g, s->ph, buf, species, gx, gy, nbx);
    else
      k_hist<T, 2><<<grid, kBlock, smem, s->stream>>>(d, g, s->ph, buf, species, gx, gy, nbx);
    return cudaGetLastError();
  }

  static double* profile_region(Sim* s) { return (double*)(s->base + s->L.prof); }

  static int prof_grid(long long n) { return (int)((n + kProfThreads - 1) / kProfThreads); }

  static cudaError_t profile_B(Sim* s) {
    const int nx = s->g.nx;
    double* out = profile_region(s) + s->g.nxn + nx;
    k_profile_B<T><<<prof_grid(3LL * nx), kProfThreads, 0, s->stream>>>(P(s).B, nx, s->g.ny, out);
    return cudaGetLastError();
  }

  static cudaError_t spectrum_bperp(Sim* s) {
    const int nx = s->g.nx, ny = s->g.ny;
    double* out = profile_region(s) + s->g.nxn + 4 * (size_t)nx;
    cudaError_t e = cudaMemsetAsync(out, 0, 8 * ((size_t)nx / 2 + 1), s->stream);
    if (e != cudaSuccess) return e;
    FftPlan f;
    if (fft_plan(nx, ny, &f)) {
      double2* W = (double2*)(s->base + s->L.twiddle);
      const size_t smem = sizeof(double2) * (size_t)nx;
      e = cudaFuncSetAttribute(k_bperp_fft<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(sizeof(double2) * (size_t)kFftMax));
      if (e != cudaSuccess) return e;
      k_fft_twiddles<<<(nx + 127) / 128, 128, 0, s->stream>>>(W, nx);
      const int threads = nx >= 2048 ? kFftThreads : nx >= 512 ? 256 : 64;
      k_bperp_fft<T><<<ny, threads, smem, s->stream>>>(P(s).B, ny, f, W, out);
    } else {
      const long long work = (long long)(nx / 2 + 1) * ny;
      k_bperp_dft<T><<<grid_for(work), kBlock, 0, s->stream>>>(P(s).B, nx, ny, out);
    }
    return cudaGetLastError();
  }

  static cudaError_t spectrum_p(Sim* s, int buf, int species) {
    const int np = s->p.spec_np;
    const double* e = (const double*)(s->base + s->L.spec);
    unsigned long long* out = (unsigned long long*)(s->base + s->L.spec + 8 * ((size_t)np + 1));
    cudaError_t err = cudaMemsetAsync(out, 0, 8 * (size_t)np, s->stream);
    if (err != cudaSuccess) return err;
    const int copies = (long long)np * kWarpsPerBlock <= kSpecShared ? kWarpsPerBlock
                       : np <= kSpecShared                           ? 1
                                                                     : 0;
    // the FP32 bin: half the log2 of u.u is within about 1e-5 of the exact value
    // (|log2| <= 100: two units in the last place of the fast logarithm)
    const double per = (double)np / log2(s->p.spec_pmax / s->p.spec_pmin);
    const double eps = 2e-5 * per * (1.0 + 0.05 * fabs(log2(s->p.spec_pmin))) + 1e-6 * np;
    const size_t smem = sizeof(unsigned) * (size_t)np * copies;
    k_spectrum_p<T><<<tile_warps_grid(s), kBlock, smem, s->stream>>>(
        P(s), s->g, buf, species, np, copies, (float)log2(s->p.spec_pmin), (float)per,
        (float)std::min(eps, 1.0), e, out);
    return cudaGetLastError();
  }

  // which: FS_PROFILE_N or FS_PROFILE_DB2
  static cudaError_t profiles(Sim* s, int which) {
    const Geo& g = s->g;
    double* out = profile_region(s);
    if (which == FS_PROFILE_N)
      k_profile_n<T><<<prof_grid(g.nxn), kProfThreads, 0, s->stream>>>(P(s).n, g.nxn, g.ny, out);
    else
      k_profile_db2<T><<<(g.nx + 31) / 32, kBlock, 0, s->stream>>>(
          P(s).B, g.nx, g.ny, s->ph.b0x, s->ph.b0y, s->ph.b0z, out + g.nxn);
    return cudaGetLastError();
  }

  static cudaError_t export_grid(Sim* s, int what, int q0, int n, double* dst) {
    DevPtrs<T> d = P(s);
    const T* src = nullptr;
    int planes = 3, cols = s->g.nxn;
    switch (what) {
      case FS_B: src = d.B; cols = s->g.nx; break;
      case FS_E: src = d.E; break;
      case FS_BBAR: src = d.Bb; break;
      case FS_N: src = d.n; planes = 1; break;
      case FS_J: src = d.J; break;
      case FS_U: src = d.u; break;
      default: return cudaErrorInvalidValue;
    }
    k_export_grid<T><<<grid_for(n), kBlock, 0, s->stream>>>(src, planes, cols * s->g.ny, q0, n, dst,
                                                           d.ctr);
    return cudaGetLastError();
  }

  static cudaError_t import_B(Sim* s, const double* src, int q0, int n) {
    k_import_B<T><<<grid_for(n), kBlock, 0, s->stream>>>(P(s).B, src, s->g.nx * s->g.ny, q0, n);
    return cudaGetLastError();
  }

  static Ops make() {
    Ops o;
    o.init_particles = init_particles;
    o.deposit_all = deposit_all;
    o.moments = moments;
    o.ohm_final = ohm_final;
    o.step = step;
    o.insert_columns = insert_columns;
    o.scan_counts = scan_counts;
    o.pack_columns = pack_columns;
    o.diag = diag;
    o.hist = hist;
    o.profiles = profiles;
    o.export_grid = export_grid;
    o.import_B = import_B;
    o.step_rest = step_rest;
    o.batch_run_bytes = batch_run_bytes;
    o.fill_batch_run = fill_batch_run;
    o.batch_smem = batch_smem;
    o.batch_setup = batch_setup;
    o.push_batch = push_batch;
    o.batch_draw = batch_draw;
    o.batch_rest = batch_rest;
    o.profile_B = profile_B;
    o.spectrum_bperp = spectrum_bperp;
    o.spectrum_p = spectrum_p;
    return o;
  }
};

template <typename T>
size_t push_smem_bytes(int dim, int tx, int ty, int chunk) {
  using S = PushShape<T>;
  const int ns = (chunk == S::kChunkSmall) ? S::kStagesSmall : S::kStagesLarge;
  return dim == 1 ? PushLayout<T, 1>(tx, ty, chunk, ns).bytes
                  : PushLayout<T, 2>(tx, ty, chunk, ns).bytes;
}

}  // namespace fsx
