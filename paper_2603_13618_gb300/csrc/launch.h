// launch.h -- host-side launchers of the kernels in step_kernel.cuh, one explicit
// instantiation set per storage type (launch_f32.cu, launch_f64.cu, launch_f16.cu; the
// TMA, fixup, adjoint and plain-plane launchers exist for float and double only).
#pragma once

#include <cuda_runtime.h>

#include "adjoint_kernel.cuh"
#include "step_tma.cuh"

namespace kss {

// Grid of the fused step for an nx x ny lattice with tagging tile `tile` and
// `bands` tile bands per CTA (0: the default, step_bands(tile)).
template <class T>
inline dim3 step_grid(int nx, int ny, int tile, int bands = 0) {
  const int cols = 32 * Vec<T>::N;
  const int rows = tile * (bands > 0 ? bands : step_bands(tile));
  return dim3((unsigned)((nx + cols - 1) / cols), (unsigned)((ny + rows - 1) / rows), 1u);
}

// Grid g of the FP16 {Kn, KL, neq} step with eight cells per lane (CTA blocks of 256
// columns and at most 8 rows per warp of nw warps) for a lattice whose four-cell grid has
// `bands` tile bands per CTA, and its bands per CTA; false where its rows are not whole
// tiles or it would have more blocks than the four-cell grid (whose count sized the
// partial sums).
inline bool step_grid8(int nx, int ny, int tile, int bands, int nw, dim3& g, int& bands8) {
  const int rows = tile * bands, rows8 = rows < 8 * nw ? rows : 8 * nw;
  const dim3 g4 = step_grid<__half>(nx, ny, tile, bands);
  g = dim3(unsigned((nx + 255) / 256), unsigned((ny + rows8 - 1) / rows8), 1u);
  bands8 = rows8 / tile;
  return rows8 % tile == 0 && (long long)g.x * g.y <= (long long)g4.x * g4.y;
}

// mode: MODE_PLAIN / MODE_STD / MODE_FULL; pull: stream first; store: collide + write.
// Valid combinations: (any mode, pull, store) for steps; (STD/FULL, pull or not, no store)
// for evaluation passes.
template <class T>
cudaError_t launch_step(const StepParams<T>& p, int mode, bool pull, bool store,
                        cudaStream_t stream);

// CTAs (ranks) that share each block of an output step or evaluation pass of `nblocks`
// blocks of `rows` rows (step_kernel_split), or 0 where a block is one CTA's.  Blocks are
// shared where the ranks, at one row per warp of eight (FP32 arithmetic: or two), all fit on
// the GPU at once (two CTAs of 256 threads per SM); beyond that line the cluster's barriers
// cost more than the idle SMs.  FP64 rows, bound by the FP64 pipes that unsplit blocks leave
// idle, are shared out to 10/7 times as many blocks (in 32-row blocks, 108 on 152 SMs; single
// steps, unsplit / split): density step of 90 blocks 168 / 115 us, of smooth fields 125 / 102, of
// 108 blocks 167 / 131 and 120 / 118; of 112 blocks 168 / 144, but of smooth fields 120 / 127.
// {Kn, KL, neq} steps of the density step, unsplit / split, us: FP32 256^2 (16 blocks)
// 15.4 / 6.8, 512^2 (64) 17.5 / 8.4, 768^2 (144) 18.4 / 11.2 (20.5 at one row per warp), 1024^2
// (256) 21.7 / 32.8; FP64 64^2 (2) 322 / 21, 128^2 (8) 243 / 32, 512x256 (64) 227 / 100; FP16
// 512^2 (32 blocks of 256 columns) 21.0 / 9.0, 768^2 (72) 20.2 / 11.6, 1024^2 (128)
// 19.9 / 17.4.  All of Table 1, FP32, before the sums of a run's steps were left to the next
// one: 256^2 44.7 / 15.1, 512^2 44.1 / 19.1, 768^2 46.4 / 33.0.
template <class T>
int split_ranks(long long nblocks, int rows);
// The same for the step that launch_step (pull + store) or launch_step_aar takes with these
// parameters; *cells8: it takes eight cells per lane.
template <class T>
int step_split_ranks(const StepParams<T>& p, int mode, bool aar, bool* cells8);

// Two plain steps in one launch, from p.src to p.dst (step_plain_twice_kernel: FP32 storage,
// no two-relaxation model, no slab; faster at every size measured, 64^2 to 8192^2, so that
// only the grid's limit of rows bounds it); mid: where the state in between goes, or null.
constexpr int kTwiceRows = 8;  // rows per CTA
template <class T>
bool can_step_twice(int nx, int ny);
template <class T>
cudaError_t launch_plain_twice(const StepParams<T>& p, T* mid, cudaStream_t stream);

// One step with adaptive algorithm refinement: the two-relaxation collision in the
// region p.region (output steps rewrite it); mode as launch_step, always pull + store.
template <class T>
cudaError_t launch_step_aar(const StepParams<T>& p, int mode, cudaStream_t stream);

// One batched step (batch_step_kernel): `table` holds one StepParams per lattice
// (grid_x, nblocks and bands set), `items` the nitems CTA blocks; `ctas` CTAs (<= nitems)
// stride over the items.  mode MODE_PLAIN / MODE_STD / MODE_FULL; always pull + store.
template <class T>
cudaError_t launch_batch_step(const StepParams<T>* table, const BatchItem* items, int nitems,
                              int ctas, int mode, cudaStream_t stream, bool aar = false);

// One batched {Kn, KL, neq} step whose items' blocks (`rows` rows each) are shared out to
// `ranks` CTAs (batch_step_kernel_split, split_ranks); defer: the next step of the run forms
// this one's sums; prev: this one forms the previous one's.
template <class T>
cudaError_t launch_batch_split(const StepParams<T>* table, const BatchItem* items, int nitems,
                               int rows, int ranks, bool defer, bool prev, cudaStream_t stream);

// nsteps batched steps in one cooperative launch (batch_kernel_multi): ta / tb are the
// parameter tables of even / odd steps, mtab each lattice's MultiState, work the shared
// work counter (0 at launch); mode MODE_STD; ctas <= batch_multi_resident_ctas.
template <class T>
cudaError_t launch_batch_multi(const StepParams<T>* ta, const StepParams<T>* tb,
                               const MultiState* mtab, const BatchItem* items, int nitems,
                               int nsteps, uint32_t* work, int mode, int ctas,
                               cudaStream_t stream);
template <class T>
int batch_multi_resident_ctas(int mode);

// nsteps fused steps in one cooperative launch (step_kernel_multi): pa reads buffer A and
// writes B, pb the reverse; mode MODE_STD (the {Kn, KL, neq} set every step);
// ctas <= multi_resident_ctas.
template <class T>
cudaError_t launch_step_multi(const StepParams<T>& pa, const StepParams<T>& pb,
                              const MultiState& m, int mode, int ctas, cudaStream_t stream,
                              bool aar = false);
// CTAs of the multi-step kernel resident on the current device at once (0 on error).
template <class T>
int multi_resident_ctas(int mode, bool aar = false);

// The TMA-staged step (step_tma.cuh): mode MODE_PLAIN or MODE_STD, always pull + store;
// `ctas` persistent CTAs (one per SM).
template <class T>
cudaError_t launch_step_tma(const StepParams<T>& p, int mode, TmaPlan plan, int ctas,
                            cudaStream_t stream);

// fixup_kernel after a MODE_STD pass (step or evaluation; `pull` as that pass), with
// `ctas` CTAs of 256 threads striding over the tiles.
template <class T>
cudaError_t launch_fixup(const StepParams<T>& p, bool pull, int ctas, cudaStream_t stream);

// Rows per CTA (32, 16 or 8) for CTAs `cols` columns wide: the tallest that still gives
// at least two CTAs per SM, else 8.  Steps without outputs and the adjoint kernels use it
// (their results do not depend on the CTA shape, or are reduced in a fixed order).
inline int fill_rows(int nx, int ny, int cols, int nsm) {
  const long long gx = (nx + cols - 1) / cols;
  for (int r = 32; r >= 16; r /= 2)
    if (gx * ((ny + r - 1) / r) >= 2LL * nsm) return r;
  return 8;
}

// Adjoint kernels (adjoint_kernel.cuh) on the grid adj_grid(nx, ny, rows).
inline dim3 adj_grid(int nx, int ny, int rows = kAdjRows) {
  return dim3((unsigned)((nx + 32 * kAdjV - 1) / (32 * kAdjV)),
              (unsigned)((ny + rows - 1) / rows), 1u);
}
template <class T>
cudaError_t launch_adj_objective(const AdjParams<T>& p, cudaStream_t stream);
// One reverse step (p.rows rows per warp); chained: its predecessor in the stream is another
// reverse step of the segment, and nothing else writes the state p.f.
inline dim3 adj_reverse_grid(int nx, int ny, int rows) {
  return dim3((unsigned)((nx + 32 * kAdjV - 1) / (32 * kAdjV)),
              (unsigned)((ny - 1) / (kAdjWarps * rows) + 1), 1u);
}
// (the partials of one step: a double per warp)
inline long long adj_reverse_parts(int nx, int ny, int rows) {
  const dim3 g = adj_reverse_grid(nx, ny, rows);
  return (long long)g.x * g.y * kAdjWarps;
}
// Rows per warp of a reverse step: one, or up to four where that still leaves four waves of
// warps (28 per SM); more only where the grid's 65535 CTAs along y would not hold the rows
// (four: 1 048 560).
inline int adj_reverse_rows(int nx, int ny, int nsm) {
  int rows = 1;
  while (rows < 4 && adj_reverse_parts(nx, ny, 2 * rows) >= 4LL * 28 * nsm) rows *= 2;
  while (adj_reverse_grid(nx, ny, rows).y > 65535u) rows *= 2;
  return rows;
}
template <class T>
cudaError_t launch_adj_reverse(const AdjParams<T>& p, bool chained, cudaStream_t stream);
// *acc += the totals of nit reverse steps' n partials each, in step order (totals: [nit];
// count: a counter, 0 before and after).
template <class T>
cudaError_t launch_adj_totals(const double* part, int n, int nit, double* totals,
                              uint32_t* count, double* acc, cudaStream_t stream);
template <class T>
cudaError_t launch_adj_final(const AdjParams<T>& p, cudaStream_t stream);
// Population conversions for any storage S (float, double, __half deviations); the
// codec is that of the lattice (empty for float and double).
template <class S>
cudaError_t launch_init_equilibrium(const double* rho, const double* ux, const double* uy,
                                    S* f, long long plane, int pitch, int nx, int ny,
                                    const codec_t<S>& codec, cudaStream_t stream);
template <class S>
cudaError_t launch_init_equilibrium_f32(const float* rho, const float* ux, const float* uy,
                                        S* f, long long plane, int pitch, int nx, int ny,
                                        const codec_t<S>& codec, cudaStream_t stream);

template <class S>
cudaError_t launch_moments(const S* f, long long plane, int pitch, int nx, int ny, double* rho,
                           double* ux, double* uy, const codec_t<S>& codec, cudaStream_t stream);

template <class S>
cudaError_t launch_pops_to_dense(const S* src, long long plane, int pitch, int nx, int ny,
                                 double* dst, const codec_t<S>& codec, cudaStream_t stream);

template <class S>
cudaError_t launch_dense_to_pops(const double* src, long long plane, int pitch, int nx, int ny,
                                 S* dst, const codec_t<S>& codec, cudaStream_t stream);

// Plain pitched planes of an arithmetic type T (float, double): sensor fields, weights.
template <class T>
cudaError_t launch_pitched_to_dense(const T* src, long long plane, int pitch, int nx, int ny,
                                    int nplanes, double* dst, cudaStream_t stream);

template <class T>
cudaError_t launch_dense_to_pitched(const double* src, long long plane, int pitch, int nx,
                                    int ny, int nplanes, T* dst, cudaStream_t stream);

}  // namespace kss
