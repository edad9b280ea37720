// gp_sweeps_tile.cu -- banded FP32 sweeps over shared-memory tiles (paper, program summary:
// "Solution method"; the operator is the one of gp_sweeps.cu: each output is a (2W+1)-tap
// dot product on the odd extension of its line).
//
//   k_band_tile, k_batch_tile (the slots of a pool)
//                 y or z: a block copies 4 runs of consecutive line points, plus W on each
//                 side, of up to 32 vector positions into shared memory (cp.async, all in
//                 flight at once) and every thread computes one run from there.
//
// A run per thread that fetches its own neighbours (k_sweep_band_line) reads 21 points for
// 11 at W = 5: 90 MB through L2 per sweep of a 31 MB field, and two dependent fetches.  Here
// four runs share the halo (1.25 reads per point), all of a block's loads are in flight at
// once, and the taps are two-lane FP32 (6.5 FP32 instructions per point instead of 12).
// Measured per step (GB300; k_sweep_band_line -> here): 131 x 97 x 61 real 21.1 -> 16.9 us,
// complex 21.3 -> 19.2; 300 x 256 plane 10.6 -> 8.2, complex 9.2 -> 7.4; 64 x 48 x 32 13.7 ->
// 11.9; 240 x 200 x 160 31.9 -> 30.6, complex 66.6 -> 64.4.  What bounds it at 240 x 200 x 160:
// issue and latency together (2.3 instructions per clock, 22 warps per SM); a copy of the
// field takes 8.3 us where a sweep takes 14.
#include <algorithm>
#include <type_traits>

#include "gp_device.cuh"
#include "gp_split.cuh"

namespace gpk {

namespace {

constexpr int kTileCols = 32;      // y / z: vector positions per block, one per lane
constexpr int kTileRuns = 4;       // y / z: runs per block, one per warp
constexpr int kBatchTileThreads = 128;   // pools: runs times columns

// points per run: one turn of the (2W+1)-point ring (W = 3: two)
template <int W> __host__ __device__ constexpr int run_max() { return W == 3 ? 14 : 2 * W + 1; }

// One run of `len` outputs (at most run_max<W>()) down a column of float4 in shared memory:
// col[0] is W points before the first output, points are `stride` vectors apart.
// emit(u, value) receives output u.
template <int W, class TAPS, class EMIT>
__device__ __forceinline__ void band_run(const float4* col, int stride, int len, const TAPS& taps, EMIT emit) {
  constexpr int P = 2 * W + 1;
  float4 ring[P];
#pragma unroll
  for (int m = 0; m < 2 * W; ++m) ring[m] = col[m * stride];
#pragma unroll
  for (int u = 0; u < run_max<W>(); ++u) {
    if (u < len) {
      ring[(u + 2 * W) % P] = col[(u + 2 * W) * stride];
      const float2 lo = taps([&](int k) { const float4& r = ring[(u + W + k + P) % P]; return f2(r.x, r.y); });
      const float2 hi = taps([&](int k) { const float4& r = ring[(u + W + k + P) % P]; return f2(r.z, r.w); });
      emit(u, make_float4(lo.x, lo.y, hi.x, hi.y));
    }
  }
}

// Point of the line whose value (negated when it lies outside) stands at j of the odd
// extension about the ghosts -1 and n; -1 for the ghosts themselves and beyond reach.
__device__ __forceinline__ int image_of(int j, int n) {
  if (j >= 0 && j < n) return j;
  const int m = j < 0 ? -2 - j : 2 * n - j;
  return m >= 0 && m < n ? m : -1;
}

__device__ __forceinline__ float4 neg4(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }

// Norm partials of a block: kernel tail shared with k_sweep_band_line (see there).
template <int NW>
__device__ __forceinline__ void block_norm(FF acc, const SweepParams& p, FF* sh) {
  __syncthreads();
  if (p.norm_defer) {
    for (int o = 16; o > 0; o >>= 1) acc = ff_add(acc, ff_shfl_down(acc, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      FF s = sh[0];
      for (int w = 1; w < NW; ++w) s = ff_add(s, sh[w]);
      for (int c = 0; c < p.norm_copies; ++c)
        reinterpret_cast<FF*>(p.partials)[(size_t)c * gridDim.x + blockIdx.x] = s;
      if (blockIdx.x == 0) *p.scale_state = 1;
    }
  } else {
    norm_finish_ff(acc, reinterpret_cast<FF*>(p.partials), p.counter, gridDim.x, blockIdx.x, p.scale_out,
                   p.status, p.dV, p.counter + kNormGroupBase, kNormGroups, sh);
  }
}

}  // namespace

// ------------------------------------------------------------------- y, z

namespace {

// One block of a y or z sweep: `runs` runs of L points from point j0 of `cols` columns
// (runs * cols threads; thread: column c, run `run`), one float4 of x each.  `in` and `out`
// point to the first point of the thread's column (on: it exists), sv vectors between points,
// `valid` elements of its vectors inside the row, wt the weights (centre first at W).  at,
// nall: the column's index in the field and the field's size, for the bounds-checked build.
// Returns the sum of |u|^2 over the thread's run (NORM; POOL: value after value).
template <bool CPLX, bool NORM, int W, bool POOL>
__device__ __forceinline__ float tile_block(float4* tile, const float4* in, float4* out, size_t sv, int n, int j0, int L,
                                            int runs, int cols, int c, int run, bool on, int valid, const float* wt,
                                            long long at, long long nall, int* status) {
  const int rows = min(runs * L, n - j0) + 2 * W;
  const bool interior = j0 >= W && j0 - W + rows <= n;   // no image or ghost within reach
  if (interior) {
    const float4* src = in + (size_t)(j0 - W + run) * sv;
    float4* dst = tile + run * cols + c;
#pragma unroll 4
    for (int t = run; t < rows; t += runs) {
      if (on && GP_IN(at + (long long)(j0 - W + t) * (long long)sv, nall, status)) cp_async16(dst, src);
      src += runs * sv;
      dst += runs * cols;
    }
  } else {
    for (int t = run; t < rows; t += runs) {
      const int m = image_of(j0 - W + t, n);
      bool ok = on && m >= 0;
      if (ok && !GP_IN(at + (long long)m * (long long)sv, nall, status)) ok = false;
      cp_async16_zfill(tile + t * cols + c, in + (ok ? (size_t)m * sv : 0), ok);
    }
  }
  cp_async_commit();
  const std::conditional_t<POOL, BandChain<CPLX, W>, BandTaps<CPLX, W>> taps(wt);
  cp_async_wait<0>();
  if (!interior)   // images: negated by the thread that copied them
    for (int t = run; t < rows; t += runs) {
      const int j = j0 - W + t;
      if (j < 0 || j >= n) tile[t * cols + c] = neg4(tile[t * cols + c]);
    }
  __syncthreads();
  const int jr = j0 + run * L;
  if (!on || jr >= n) return 0.f;
  out += (size_t)jr * sv;
  float2 q = f2(0.f);
  band_run<W>(tile + run * L * cols + c, cols, min(L, n - jr), taps, [&](int u, float4 v) {
    if (!GP_IN(at + (long long)(jr + u) * (long long)sv, nall, status)) return;
    if (valid == (CPLX ? 2 : 4)) {
      *out = v;
      if (NORM && POOL) q.x = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, q.x))));
      else if (NORM) q = fma2(f2(v.z, v.w), f2(v.z, v.w), fma2(f2(v.x, v.y), f2(v.x, v.y), q));
    } else {
      const float e[4] = {v.x, v.y, v.z, v.w};
      float* os = reinterpret_cast<float*>(out);
      for (int i = 0; i < valid * (CPLX ? 2 : 1); ++i) {
        os[i] = e[i];
        if (NORM) q.x = fmaf(e[i], e[i], q.x);
      }
    }
    out += sv;   // (the runs emit in order)
  });
  return q.x + q.y;
}

}  // namespace

// Block: kTileRuns warps, lane = vector position (tile_cols of them), warp = run of tile_run
// points.  Blocks: position chunk fastest, then the other axis, then the line's parts.
template <bool CPLX, int AXIS, bool NORM, int W>
__global__ void __launch_bounds__(32 * kTileRuns) k_band_tile(const __grid_constant__ SweepParams p) {
  extern __shared__ __align__(16) float4 tile[];
  constexpr int EPT = CPLX ? 2 : 4;
  const int lane = threadIdx.x & 31, run = threadIdx.x >> 5;
  const int nx = p.nx, TC = p.tile_cols, L = p.tile_run;
  const int nvec = (nx + EPT - 1) / EPT, nchunk = (nvec + TC - 1) / TC;
  const int nother = AXIS == 1 ? p.nz : p.ny;
  const unsigned int b = blockIdx.x, rest = b / (unsigned int)nchunk;
  const int ch = (int)(b - rest * (unsigned int)nchunk);
  const int part = (int)(rest / (unsigned int)nother), o = (int)(rest - (unsigned int)part * nother);
  const int xv = ch * TC + lane;
  const bool on = lane < TC && xv < nvec;
  const size_t P = (size_t)p.pitch / EPT;   // row pitch in vectors
  const size_t sv = AXIS == 1 ? P : P * (size_t)p.ny;
  const size_t base = (AXIS == 1 ? (size_t)o * P * p.ny : (size_t)o * P) + (on ? xv : 0);
  pdl_begin();
  // the factor's dither (FP32, imaginary time): the step's x sweep has read the counter
  if (AXIS == 1 && p.step_ctr && blockIdx.x == 0 && threadIdx.x == 0) *p.step_ctr += 1;
  const float part_sum = tile_block<CPLX, NORM, W, false>(
      tile, static_cast<const float4*>(p.psi) + base, static_cast<float4*>(p.out) + base, sv, p.n, part * kTileRuns * L, L,
      kTileRuns, kTileCols, lane, run, on, min(EPT, nx - xv * EPT), p.band_wt, (long long)base, (long long)P * p.ny * p.nz,
      p.status);
  if (NORM) block_norm<kTileRuns>(FF{part_sum, 0.f}, p, reinterpret_cast<FF*>(tile));
}

// The same over the slots of a pool: block b of the launch is block blk of the nblk of one
// slot.  Its columns are 128 / runs consecutive (vector, other axis) pairs, so that narrow
// slots fill the lanes too, and short lines take fewer runs and more columns.  The z sweep's
// norm is reduced per slot (its own partials, counter and factor).  The fields are the bits of
// runs of three turns a thread (what the pool stepped with before, 24 mixed slots of 6.1e6
// points: six launches of 15 us at a tenth of the SMs' warps): the taps in Field::chain's
// order, the norm in FP32 within a turn.
template <bool CPLX, int AXIS, bool NORM, int W>
__global__ void __launch_bounds__(kBatchTileThreads) k_batch_tile(const __grid_constant__ BatchArgs b) {
  extern __shared__ __align__(16) float4 tile[];
  constexpr int EPT = CPLX ? 2 : 4;
  pdl_begin();
  const LineBlock lb = static_cast<const LineBlock*>(b.items)[blockIdx.x];
  const SlotDesc& d = b.slots[lb.slot];
  const int runs = d.tile_runs[AXIS], L = d.tile_run[AXIS], cols = kBatchTileThreads / runs;
  int run = (int)threadIdx.x / cols;
  const int c = (int)threadIdx.x - run * cols;
  if (run >= runs) run = 1 << 20;   // (128 threads are not a multiple of 3, 5 or 6 runs: no row, no output)
  const int nx = d.nx, n = AXIS == 1 ? d.ny : d.nz, nother = AXIS == 1 ? d.nz : d.ny;
  const int nvec = (nx + EPT - 1) / EPT, total = nvec * nother, nchunk = (total + cols - 1) / cols;
  const int part = lb.blk / nchunk, g = (lb.blk - part * nchunk) * cols + c;
  const bool on = g < total;
  const int o = on ? g / nvec : 0, xv = on ? g - o * nvec : 0;
  const size_t P = (size_t)d.pitch / EPT, sv = AXIS == 1 ? P : P * (size_t)d.ny;
  const size_t base = (AXIS == 1 ? (size_t)o * P * d.ny : (size_t)o * P) + xv;
  const float part_sum = tile_block<CPLX, NORM, W, true>(
      tile, static_cast<const float4*>(AXIS == 1 ? d.field : d.staging) + base,
      static_cast<float4*>(AXIS == 1 ? d.staging : d.field) + base, sv, n, part * runs * L, L, runs, cols, c, run, on,
      min(EPT, nx - xv * EPT), d.wt[AXIS] + (kBandHalfMax - W) * (CPLX ? 2 : 1), (long long)base,
      (long long)P * d.ny * d.nz, b.status);
  if (NORM) {
    __syncthreads();   // the tile is idle now: the norm's per-warp sums go there
    norm_finish_ff(FF{part_sum, 0.f}, reinterpret_cast<FF*>(d.partials), d.counter, (unsigned int)lb.nblk,
                   (unsigned int)lb.blk, d.scale, b.status, d.dV, nullptr, 1, reinterpret_cast<FF*>(tile));
  }
}

// ------------------------------------------------------------------ launchers

namespace {

using Kernel = void (*)(SweepParams);

template <int W> Kernel tile_kernel_w(int axis, bool cplx, bool norm) {
  if (axis == 1) return cplx ? k_band_tile<true, 1, false, W> : norm ? k_band_tile<false, 1, true, W> : k_band_tile<false, 1, false, W>;
  return cplx ? k_band_tile<true, 2, false, W> : k_band_tile<false, 2, true, W>;
}
Kernel tile_kernel(int axis, int w, bool cplx, bool norm) {
  switch (w) {
    case 3: return tile_kernel_w<3>(axis, cplx, norm);
    case 5: return tile_kernel_w<5>(axis, cplx, norm);
    case 8: return tile_kernel_w<8>(axis, cplx, norm);
    default: return nullptr;
  }
}
int run_max_of(int w) { return w == 3 ? run_max<3>() : w == 5 ? run_max<5>() : run_max<8>(); }

size_t tile_smem(const SweepParams& p) {
  return (size_t)(kTileRuns * p.tile_run + 2 * p.band_w) * kTileCols * sizeof(float4);
}

template <class ARGS> cudaError_t launch_tile(void (*k)(ARGS), const ARGS& p, int grid, int threads, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = st;
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  return cudaLaunchKernelEx(&cfg, k, p);
}

}  // namespace

// Runs of nearly equal length, no longer than run_max; the last block of a line may hold
// fewer.  Returns the blocks of the launch.
long long band_tile_setup(int axis, SweepParams* p, bool complex_field) {
  const int nvec = complex_field ? (p->nx + 1) / 2 : (p->nx + 3) / 4;
  const int chunks = (nvec + kTileCols - 1) / kTileCols;
  const int most = kTileRuns * run_max_of(p->band_w);
  const int parts = (p->n + most - 1) / most, per = (p->n + parts - 1) / parts;
  p->tile_cols = (nvec + chunks - 1) / chunks;
  p->tile_run = (per + kTileRuns - 1) / kTileRuns;
  const int blocks_line = (p->n + kTileRuns * p->tile_run - 1) / (kTileRuns * p->tile_run);
  Kernel k = tile_kernel(axis, p->band_w, complex_field, p->plane_norm != 0);
  if (!k || cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (kTileRuns * run_max_of(p->band_w) + 2 * p->band_w) * kTileCols * 16) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (long long)chunks * (axis == 1 ? p->nz : p->ny) * blocks_line;
}

cudaError_t launch_band_tile(int axis, const SweepParams& p, bool complex_field, int grid, cudaStream_t st) {
  return launch_tile(tile_kernel(axis, p.band_w, complex_field, p.plane_norm != 0), p, grid, 32 * kTileRuns,
                     tile_smem(p), st);
}

// ---- pools

// Runs per block (at most six; turns 1, 2: so many) and points per run of a line of n points
// at half-width w.  Where the norm is summed a run is one turn of the ring: a slot's factor, and
// with it its field, then depends on no launch shape but through the turns' order in the sum.
void batch_tile_shape(int n, int w, int turns, bool norm, int* runs, int* run) {
  const int most = norm ? 2 * w + 1 : run_max_of(w), need = (n + most - 1) / most, r = turns >= 3 ? 6 : turns;
  const int parts = (need + r - 1) / r;
  *runs = (need + parts - 1) / parts;
  *run = norm ? most : (n + parts * *runs - 1) / (parts * *runs);
}

long long batch_tile_blocks(int nx, int nother, int n, int runs, int run, bool complex_field) {
  const long long total = (long long)((nx + (complex_field ? 1 : 3)) / (complex_field ? 2 : 4)) * nother;
  const int cols = kBatchTileThreads / runs;
  return (total + cols - 1) / cols * ((n + runs * run - 1) / (runs * run));
}

size_t batch_tile_smem(int runs, int run, int w) {
  return (size_t)(runs * run + 2 * w) * (kBatchTileThreads / runs) * sizeof(float4);
}

using BatchKernel = void (*)(BatchArgs);
template <int W> static BatchKernel batch_tile_kernel_w(int axis, bool cplx) {
  if (axis == 1) return cplx ? k_batch_tile<true, 1, false, W> : k_batch_tile<false, 1, false, W>;
  return cplx ? k_batch_tile<true, 2, false, W> : k_batch_tile<false, 2, true, W>;
}
static BatchKernel batch_tile_kernel(int axis, int w, bool cplx) {
  return w == 3 ? batch_tile_kernel_w<3>(axis, cplx) : w == 5 ? batch_tile_kernel_w<5>(axis, cplx) : batch_tile_kernel_w<8>(axis, cplx);
}

cudaError_t launch_batch_tile(int axis, int w, const BatchArgs& b, bool complex_field, size_t smem, cudaStream_t st) {
  const BatchKernel k = batch_tile_kernel(axis, w, complex_field);
  // (up to 66 KB: one run of 17 points and its halo at half-width 8)
  const cudaError_t e = smem <= 48 * 1024 ? cudaSuccess
                                          : cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                                 (int)batch_tile_smem(1, run_max_of(w), w));
  return e != cudaSuccess ? e : launch_tile(k, b, b.nitems, kBatchTileThreads, smem, st);
}

}  // namespace gpk
