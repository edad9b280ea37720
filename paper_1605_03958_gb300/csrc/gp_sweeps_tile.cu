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
// Measured per step (GB300; k_sweep_band_line -> here, x and y apart): 131 x 97 x 61 real 18.1 ->
// 15.4 us, complex 17.9 -> 15.9; 300 x 256 plane 10.4 -> 8.2, complex 9.1 -> 7.6; 64 x 48 x 32 12.6 ->
// 9.9, complex 11.0 -> 9.4; 128 x 128 x 96 16.5 -> 14.3; 240 x 200 x 160 31.4 -> 31.3.  What bounds it
// at 240 x 200 x 160: latency and issue together (1.4-1.5 instructions per clock with cold caches, 25
// warps per SM); a copy of the field takes 8.3 us where a sweep takes 14.
#include <algorithm>
#include <type_traits>

#include "gp_device.cuh"
#include "gp_split.cuh"

namespace gpk {

namespace {

constexpr int kTileCols = 32;      // y / z: vector positions per block, one per lane
constexpr int kTileRuns = 4;       // y / z: runs per block, one per warp
constexpr int kBatchTileThreads = 128;   // pools: runs times columns
constexpr int kXyThreads = 256;    // x and y together
constexpr int kXyRows = 12;        // rows per block at most (64^3 9.3 us a step, 96 x 80 x 64 complex 11.1,
                                   // 256 x 32 x 32 9.6; with 32 rows 9.2, 12.2, 11.1)
// Grids that take it (separate -> joined, us per step, real / complex): 64^3 11.1 -> 9.3 /
// 10.4 -> 8.9, 96 x 80 x 64 11.7 -> 10.7 / 12.1 -> 11.1, 256 x 32 x 32 10.2 -> 9.6 / 10.3 -> 9.6;
// and not: 131 x 97 x 61 15.4 -> 18.3 / 15.9 -> 20.0, 24 x 100 x 80 (720 blocks) 12.8 -> 13.3 /
// 12.1 -> 11.5
constexpr long long kXyPoints = 1 << 19, kXyBlocks = 600;
constexpr int kXyWidth = 256;      // a warp's lanes

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
  if (p.step_count && blockIdx.x == 0 && threadIdx.x == 0) *p.step_ctr += 1;
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

// ------------------------------------------------------------------- x and y

// Banded x and y sweeps in one launch, for small 3D grids: a block takes xy_rows consecutive
// rows of one plane, plus W on each side, into shared memory, applies the pending factor, the
// pointwise substep and the x operator to them there (a warp on its own rows, in place), and
// then the y operator down the columns, written out of place.
//
// A small grid's step is a chain of latencies (launch, first loads, the norm's partials), not
// of work, and a launch less takes a third of it away: 64 x 48 x 32 9.8 -> 8.3 us per step
// (complex 9.3 -> 7.5), 33 x 60 x 50 12.1 -> 8.7 (10.8 -> 8.7).  The price is the x work of 2W halo rows a
// block and about 78 instructions per point in all, against 35 of the separate sweeps: from
// about 2^19 points on that is what bounds it (240 x 200 x 160: 40 us against 31; blocks of a
// cluster that exchange their edge rows instead, 44).
//
// x: a lane owns eight consecutive elements of a row, 32 / lanes-per-row rows at a time; the W
// neighbours come from the lanes beside it by shuffles, the odd images at the row's ends from
// the lane's own and left-hand elements.  Real taps run two-lane on the pairs (e, e + 4).  Rows
// stand in shared memory with vector v at v ^ (v >> 3 & VPL - 1), so that neither eight lanes
// VPL vectors apart (x) nor eight neighbouring vectors (y) meet in a bank.
// y: as in k_band_tile, one run of xy_run points per thread; the odd images of the plane's
// first and last rows are stored along with the rows.
template <bool CPLX, int W> struct XRow {
  static constexpr int EPT = CPLX ? 2 : 4, VPL = 8 / EPT;
  using F = Field<float, CPLX>;
  using E = typename F::E;
  E v[8], lo[W + 1], hi[W + 1];   // lo[m]: m points left of the first, hi[m]: right of the last
  // position j of the row relative to the lane's first element
  __device__ __forceinline__ E at(int j) const { return j < 0 ? lo[-j] : j >= 8 ? hi[j - 7] : v[j]; }
  // images of a row that ends after the first c elements of this lane: 0 at the ghost c,
  // -at(2c - j) at j > c
  template <int C> __device__ __forceinline__ void end_own() {
#pragma unroll
    for (int j = C; j < 8; ++j) v[j] = j == C || 2 * C - j < -W ? F::zero() : F::scaled(at(2 * C - j), -1.f);
  }
  template <int C> __device__ __forceinline__ void end_hi() {
#pragma unroll
    for (int m = 1; m <= W; ++m) {
      const int i = 2 * C - 7 - m;
      hi[m] = i == C || i < -W ? F::zero() : F::scaled(at(i), -1.f);
    }
  }
  __device__ __forceinline__ void end_own(int c) {
    switch (c) {
      case 1: end_own<1>(); break;
      case 2: end_own<2>(); break;
      case 3: end_own<3>(); break;
      case 4: end_own<4>(); break;
      case 5: end_own<5>(); break;
      case 6: end_own<6>(); break;
      case 7: end_own<7>(); break;
    }
  }
  __device__ __forceinline__ void end_hi(int c) {
    switch (c) {
      case 1: end_hi<1>(); break;
      case 2: end_hi<2>(); break;
      case 3: end_hi<3>(); break;
      case 4: end_hi<4>(); break;
      case 5: end_hi<5>(); break;
      case 6: end_hi<6>(); break;
      case 7: end_hi<7>(); break;
      default: end_hi<8>(); break;
    }
  }
  // the pointwise substep by the short polynomial: the operations of
  // Field::nonlinear_small, two real points at a time
  __device__ __forceinline__ void small(const E (&fx)[8], E fr, float dtg) {
    if constexpr (CPLX) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = F::nonlinear_small(v[e], F::mul(fx[e], fr), dtg * F::abs2(v[e]));
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 c = f2(v[e], v[e + 4]), z = mul2(f2(-dtg), mul2(c, c));
        float2 q = fma2(z, f2(1.f / 24.f), f2(1.f / 6.f));
        q = fma2(z, q, f2(0.5f));
        q = fma2(z, q, f2(1.f));
        q = fma2(z, q, f2(1.f));
        const float2 r = mul2(mul2(c, mul2(f2(fx[e], fx[e + 4]), f2(fr))), q);
        v[e] = r.x;
        v[e + 4] = r.y;
      }
    }
  }
  __device__ __forceinline__ void start() {
#pragma unroll
    for (int m = 1; m <= W; ++m) lo[m] = m == 1 ? F::zero() : F::scaled(v[m - 2], -1.f);
  }
  __device__ __forceinline__ void result(const BandChain<CPLX, W>& taps, float4 (&o)[VPL]) const {
    if constexpr (CPLX) {
#pragma unroll
      for (int q = 0; q < VPL; ++q) {
        const float2 a = taps([&](int k) { return at(2 * q + k); });
        const float2 b = taps([&](int k) { return at(2 * q + 1 + k); });
        o[q] = make_float4(a.x, a.y, b.x, b.y);
      }
    } else {
      float2 pr[4 + 2 * W];   // pr[W + j] = (at(j), at(j + 4))
#pragma unroll
      for (int j = -W; j < 4 + W; ++j) pr[W + j] = f2(at(j), at(j + 4));
      float2 r[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) r[e] = taps([&](int k) { return pr[W + e + k]; });
      o[0] = make_float4(r[0].x, r[1].x, r[2].x, r[3].x);
      o[1] = make_float4(r[0].y, r[1].y, r[2].y, r[3].y);
    }
  }
};

template <int VPL> __device__ __forceinline__ int xy_swizzle(int v) { return v ^ ((v >> 3) & (VPL - 1)); }

__device__ __forceinline__ float shfl_el(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ float2 shfl_el(float2 v, int src) {
  return f2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

template <bool CPLX, int W>
__global__ void __launch_bounds__(kXyThreads) k_band_xy(const __grid_constant__ SweepParams p) {
  extern __shared__ __align__(16) float4 tile[];
  using F = Field<float, CPLX>;
  using E = typename F::E;
  using X = XRow<CPLX, W>;
  constexpr int EPT = X::EPT, VPL = X::VPL, NW = kXyThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nx = p.nx, ny = p.ny;
  const int nl = (nx + 7) / 8, RV = nl * VPL;       // lanes of eight elements and vectors per row
  const int RP = 32 / nl;                           // rows per warp pass
  const int rp = lane / nl, li = lane - rp * nl;
  const unsigned int parts = (unsigned int)p.xy_parts;
  const int k = (int)(blockIdx.x / parts), part = (int)(blockIdx.x - (unsigned int)k * parts);
  const int j0 = part * p.xy_rows, out_rows = min(p.xy_rows, ny - j0);
  const int jlo = max(0, j0 - W), nreal = min(ny, j0 + out_rows + W) - jlo;
  const int P = p.pitch / EPT;
  const size_t plane = (size_t)k * ny * P;
  const long long nall = (long long)P * ny * p.nz;
  (void)nall;
  const int npass = (nreal + RP - 1) / RP;
  pdl_begin();
  const float4* in = static_cast<const float4*>(p.psi) + plane;
  for (int idx = threadIdx.x; idx < nreal * RV; idx += kXyThreads) {
    const int row = idx / RV, v = idx - row * RV;
    const bool ok = v < P && GP_IN((long long)plane + (long long)(jlo + row) * P + v, nall, p.status);
    cp_async16_zfill(tile + (size_t)(jlo - j0 + W + row) * RV + xy_swizzle<VPL>(v),
                     in + (ok ? (size_t)(jlo + row) * P + v : 0), ok);   // (past the pitch: zeros)
  }
  cp_async_commit();
  // the ghost rows
  for (int v = threadIdx.x; v < RV; v += kXyThreads) {
    if (j0 < W) tile[(size_t)(W - 1 - j0) * RV + v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j0 + out_rows + W > ny) tile[(size_t)(ny - j0 + W) * RV + v] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // the pending factor (see k_sweep_x_reg), while the rows are on their way
  __shared__ float s_block;
  {
    const double f = p.norm_defer
                         ? deferred_scale(p.partials + (size_t)(blockIdx.x % p.norm_copies) * p.norm_blocks,
                                          p.norm_blocks, p.dV, p.status, blockIdx.x == 0, p.scale_state, p.scale)
                         : 0.0;
    // (rounded as the separate x sweep of such rows does)
    const double g = p.norm_defer ? f : *p.scale;
    if (threadIdx.x == 0)
      s_block = p.band_reg ? (float)(g * step_dither(p.step_ctr)) : (float)g * step_dither_f(p.step_ctr);
  }
  const BandChain<CPLX, W> taps(p.band_wt);
  const float dtg = p.band_dtg;
  const bool pw = p.pw != 0;
  const int ends = nx - 8 * (nl - 1);               // elements of a row's last lane
  const bool first = li == 0, last = li == nl - 1;
  const unsigned int row_lanes = nl >= 32 ? 0xffffffffu : ((1u << nl) - 1u) << (rp < RP ? rp * nl : 0);
  E fx[8];
#pragma unroll
  for (int q = 0; q < VPL; ++q) {
    const int v = li * VPL + q;
    const float4 f = v < P ? __ldg(static_cast<const float4*>(p.band_fx) + v) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int e = 0; e < EPT; ++e) fx[q * EPT + e] = reinterpret_cast<const E*>(&f)[e];
  }
  const E* fyz = static_cast<const E*>(p.band_fyz) + (size_t)k * ny + jlo;
  cp_async_wait<0>();
  __syncthreads();
  const float s = s_block;
  for (int q = warp; q < npass; q += NW) {
    const int row = q * RP + rp;
    const bool on = rp < RP && row < nreal;
    const int j = jlo + row;                        // line position
    float4* trow = tile + (size_t)(j - j0 + W) * RV;
    const E fr = on ? fyz[row] : F::zero();
    X x;
    float ymax = 0.f;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const float4 c = on ? trow[xy_swizzle<VPL>(li * VPL + u)] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e < EPT; ++e) x.v[u * EPT + e] = F::scaled(reinterpret_cast<const E*>(&c)[e], s);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) ymax = fmaxf(ymax, F::abs2(x.v[e]));
    ymax *= fabsf(dtg);   // (monotonic: the largest rounded argument)
    // a row takes the short polynomial when every argument in it allows that
    const unsigned int big = __ballot_sync(0xffffffffu, !(ymax <= 0.0625f));
    if (!pw) {
    } else if ((big & row_lanes) == 0u) {
      x.small(fx, fr, dtg);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) x.v[e] = F::nonlinear_full(x.v[e], F::mul(fx[e], fr), dtg * F::abs2(x.v[e]));
    }
    // neighbours: left, the images in a ragged last lane, right
#pragma unroll
    for (int m = 1; m <= W; ++m) x.lo[m] = shfl_el(x.v[8 - m], (lane + 31) & 31);
    if (first) x.start();
    if (ends != 8 && last) x.end_own(ends);
#pragma unroll
    for (int m = 1; m <= W; ++m) x.hi[m] = shfl_el(x.v[m - 1], (lane + 1) & 31);
    if (last) x.end_hi(ends);
    float4 o[VPL];
    x.result(taps, o);
    if (!on) continue;
    // the row, and its odd image about a ghost row within the block's reach
    const int jl = -2 - j, jr = 2 * ny - j;
    const bool il = jl >= j0 - W, ir = jr < j0 + out_rows + W;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int c = xy_swizzle<VPL>(li * VPL + u);
      trow[c] = o[u];
      if (il) tile[(size_t)(jl - j0 + W) * RV + c] = neg4(o[u]);
      if (ir) tile[(size_t)(jr - j0 + W) * RV + c] = neg4(o[u]);
    }
  }
  __syncthreads();
  const BandTaps<CPLX, W> ytaps(p.band_wt_y);
  const int nvec = (nx + EPT - 1) / EPT, L = p.xy_run;
  const int items = (out_rows + L - 1) / L * nvec;
  for (int i = threadIdx.x; i < items; i += kXyThreads) {
    const int run = i / nvec, c = i - run * nvec, jr = run * L;
    const size_t at = plane + (size_t)(j0 + jr) * P + c;
    float4* out = static_cast<float4*>(p.out) + at;
    const int valid = min(EPT, nx - c * EPT);
    band_run<W>(tile + (size_t)jr * RV + xy_swizzle<VPL>(c), RV, min(L, out_rows - jr), ytaps, [&](int u, float4 v) {
      if (!GP_IN((long long)at + (long long)u * P, nall, p.status)) return;
      if (valid == EPT) {
        *out = v;
      } else {
        const float e[4] = {v.x, v.y, v.z, v.w};
        float* os = reinterpret_cast<float*>(out);
        for (int m = 0; m < valid * (CPLX ? 2 : 1); ++m) os[m] = e[m];
      }
      out += P;   // (the runs emit in order)
    });
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

// ---- x and y

static Kernel xy_kernel(int w, bool cplx) {
  if (w == 3) return cplx ? k_band_xy<true, 3> : k_band_xy<false, 3>;
  return cplx ? k_band_xy<true, 5> : k_band_xy<false, 5>;
}

bool band_xy_setup(SweepParams* p, bool complex_field) {
  const int w = p->band_w;
  const int nvec = complex_field ? (p->nx + 1) / 2 : (p->nx + 3) / 4, parts = (p->ny + kXyRows - 1) / kXyRows;
  if ((w != 3 && w != 5) || p->nx < 8 || p->nx > kXyWidth || p->nz < 2 || (long long)p->nz * parts > kXyBlocks ||
      (long long)p->nx * p->ny * p->nz > kXyPoints)
    return false;
  p->xy_rows = (p->ny + parts - 1) / parts;
  p->xy_parts = (p->ny + p->xy_rows - 1) / p->xy_rows;
  // at least as many runs as the threads make, of three points or more; no longer than a ring's turn
  const int runs = std::max((p->xy_rows + run_max_of(w) - 1) / run_max_of(w), kXyThreads / nvec);
  p->xy_run = std::max((p->xy_rows + runs - 1) / runs, std::min(p->xy_rows, 3));
  // (at most 22 rows of 2 KB)
  p->xy_smem = (p->xy_rows + 2 * w) * ((p->nx + 7) / 8) * (complex_field ? 4 : 2) * (int)sizeof(float4);
  return true;
}

cudaError_t launch_band_xy(const SweepParams& p, bool complex_field, cudaStream_t st) {
  return launch_tile(xy_kernel(p.band_w, complex_field), p, p.nz * p.xy_parts, kXyThreads, (size_t)p.xy_smem, st);
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
