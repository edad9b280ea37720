// gp_sweeps64.cu -- the Crank-Nicolson sweeps of one split-step Crank-Nicolson step for
// fields stored in FP64 (the paper's precision): the real field of imaginary time and
// the complex field of real time (paper, program summary: "Solution method"; imag3d /
// real3d summaries).  Same method and recurrence as the tile kernels of gp_sweeps.cu:
//   forward   d_j = B_j d_{j-1} + [A_j v_j + B_j (v_{j-1} + v_{j+1})],
//   back      u_j = d_j + B_j u_{j+1},
// A_j = m_j (1 - 2a), B_j = a m_j, m_j the Thomas pivots (computed in FP64 on the host).
//
// FP64 arithmetic is narrow on this part: the whole GPU retires about 0.5 T FP64 lane
// operations per second (FP32: 35 T), a warp's FP64 instruction costs the same with
// any number of active lanes, and one warp per scheduler keeps a scheduler's FP64 unit
// busy (a dependent FP64 chain hides its latency at that rate).  So these kernels
//   * keep all 32 lanes of every warp on useful work,
//   * spread their warps evenly over the SMs' schedulers (no full-line shared-memory
//     tile: occupancy is set by registers, not by the line length),
//   * spend as few FP64 instructions per point as the method allows: 13 for x with the
//     pointwise substep (real field; the exp polynomial's degree chosen per group of
//     points from a bound on its argument), 5 for y and z, 1 more in z for the norm.
// Memory traffic is secondary: a sweep reads and writes the field twice (forward values
// stored in place, then the back substitution), mostly through L2, in a fraction of
// its arithmetic time.
//
// Lines of at least 16 points with |a| <= 1/32 (every configuration at dt <= h^2 / 8) take
// the increment form instead (second half of this file), which moves all but one or two
// FP64 operations per point to the FP32 pipe.  The kernels of this first half serve the
// others: shorter lines, larger time steps.
//
//   x    a warp owns 32 consecutive rows, one row per lane.  Rows are contiguous, so a
//        warp moves them through shared memory in chunks of C columns (32 real / 16
//        complex, padded rows against bank conflicts): a chunk is loaded and stored
//        coalesced (lane = column) and the recurrence walks it lane = row.  The pending
//        renormalisation factor and the pointwise substep are applied on the load.
//   y/z  a thread owns one line; lanes are consecutive x, so every access is coalesced.
//        The line streams forward (forward values in place) and back, loads issued kU
//        elements ahead.  z sums |u|^2 of its output for the renormalisation factor.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "gp_device.cuh"
#include "gp_split.cuh"

namespace gpk {

namespace {

constexpr int kU64 = 8;          // y / z: elements loaded ahead of the recurrence
constexpr int kX64Warps = 4;     // x: warps per block (each on its own 32 rows)
constexpr int kLineThreads = 128;

// (-1)^k / k!, k = 0..9: the Taylor coefficients of exp(-y)
__device__ constexpr double kSignedInvFact[10] = {
    1.0, -1.0, 1.0 / 2.0, -1.0 / 6.0, 1.0 / 24.0, -1.0 / 120.0, 1.0 / 720.0, -1.0 / 5040.0,
    1.0 / 40320.0, -1.0 / 362880.0};

template <class E>
__device__ __forceinline__ E coef64(const E* T, int j, int head, E bulk) {
  return j < head ? __ldg(T + j) : bulk;
}

// |y| as an ordered integer (IEEE-754 bits without the sign); NaN sorts above every
// finite bound, so a NaN takes the library branch and propagates.
__device__ __forceinline__ unsigned long long abs_bits(double y) {
  return (unsigned long long)__double_as_longlong(y) & 0x7fffffffffffffffull;
}
// Bounds on the argument of exp(-y) / cis(-y) for the Taylor polynomials below: their
// remainders stay under 2^-56 (a quarter of an FP64 ulp of 1).
constexpr unsigned long long kBits2m10 = 0x3F50000000000000ull;  // 2^-10: exp, degree 4
constexpr unsigned long long kBits2m8 = 0x3F70000000000000ull;   // 2^-8:  cos 4 / sin 5
constexpr unsigned long long kBits2m7 = 0x3F80000000000000ull;   // 2^-7:  exp, degree 6
constexpr unsigned long long kBits2m4 = 0x3FB0000000000000ull;   // 2^-4:  exp 9, cos 8 / sin 9

// Pointwise substep of one chunk group on load (lane = column).  x[u] are raw field
// values of NG rows of one column; rf[u] their rows' trap factors exp(-dt (V_y + V_z))
// (or cis(-dt (V_y + V_z))); the column's factor exp(-dt V_x) and the pending scale s
// are folded into the polynomial's coefficients c[k] = s fx (-1)^k / k!.
//   real:    v <- (x rf) * sum_k c_k y^k,   y = (dt g s^2) x^2
//            -- 8 FP64 instructions per point at degree 4 (x^2, y, x rf, 4 Horner, 1)
template <int NG>
__device__ __forceinline__ void pointwise_real(double (&x)[NG], const double (&rf)[NG],
                                               const double (&c)[10], double cy) {
  double y[NG];
  unsigned long long mb = 0;
#pragma unroll
  for (int u = 0; u < NG; ++u) {
    y[u] = cy * (x[u] * x[u]);
    mb = max(mb, abs_bits(y[u]));
    x[u] = x[u] * rf[u];
  }
  if (__all_sync(0xffffffffu, mb <= kBits2m10)) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      double q = fma(y[u], c[4], c[3]);
      q = fma(y[u], q, c[2]);
      q = fma(y[u], q, c[1]);
      x[u] *= fma(y[u], q, c[0]);
    }
  } else if (__all_sync(0xffffffffu, mb <= kBits2m7)) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      double q = fma(y[u], c[6], c[5]);
#pragma unroll
      for (int k = 4; k >= 1; --k) q = fma(y[u], q, c[k]);
      x[u] *= fma(y[u], q, c[0]);
    }
  } else if (__all_sync(0xffffffffu, mb <= kBits2m4)) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      double q = fma(y[u], c[9], c[8]);
#pragma unroll
      for (int k = 7; k >= 1; --k) q = fma(y[u], q, c[k]);
      x[u] *= fma(y[u], q, c[0]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < NG; ++u) x[u] *= c[0] * exp(-y[u]);
  }
}

//   complex: v <- (x rf) * (G (cos th - i sin th)),  th = (dt g s^2) |x|^2, G = s fx
//            -- 21 FP64 instructions per point with the degree-4 / 5 polynomials
template <int NG>
__device__ __forceinline__ void pointwise_cplx(double2 (&x)[NG], const double2 (&rf)[NG],
                                               double2 G, double cy) {
  double th[NG];
  unsigned long long mb = 0;
#pragma unroll
  for (int u = 0; u < NG; ++u) {
    th[u] = cy * fma(x[u].x, x[u].x, x[u].y * x[u].y);
    mb = max(mb, abs_bits(th[u]));
    x[u] = cmul(x[u], rf[u]);
  }
  double cs[NG], sn[NG];
  if (__all_sync(0xffffffffu, mb <= kBits2m8)) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      const double t2 = th[u] * th[u];
      cs[u] = fma(t2, fma(t2, 1.0 / 24.0, -0.5), 1.0);
      sn[u] = th[u] * fma(t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), 1.0);
    }
  } else if (__all_sync(0xffffffffu, mb <= kBits2m4)) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      const double t2 = th[u] * th[u];
      double c = fma(t2, 1.0 / 40320.0, -1.0 / 720.0);
      c = fma(t2, c, 1.0 / 24.0);
      c = fma(t2, c, -0.5);
      cs[u] = fma(t2, c, 1.0);
      double s = fma(t2, 1.0 / 362880.0, -1.0 / 5040.0);
      s = fma(t2, s, 1.0 / 120.0);
      s = fma(t2, s, -1.0 / 6.0);
      sn[u] = th[u] * fma(t2, s, 1.0);
    }
  } else {
#pragma unroll
    for (int u = 0; u < NG; ++u) sincos(th[u], &sn[u], &cs[u]);
  }
#pragma unroll
  for (int u = 0; u < NG; ++u) {
    // H = G (cs - i sn)
    const double2 H = make_double2(fma(G.x, cs[u], G.y * sn[u]), fma(G.y, cs[u], -G.x * sn[u]));
    x[u] = cmul(x[u], H);
  }
}

}  // namespace

// ------------------------------------------------------------------ sweep x

template <bool CPLX> struct X64Geom {
  using E = typename Field<double, CPLX>::E;
  static constexpr int C = CPLX ? 16 : 32;   // columns per chunk
  static constexpr int LD = C + 1;           // padded chunk row, elements
  static constexpr int RPI = 32 / C;         // rows per 32-lane load
  static constexpr int NG = 8;               // loads in flight per lane
  static constexpr size_t warp_elems = 2 * 32 * LD + 32;   // two chunk buffers + row factors
  static constexpr size_t smem = kX64Warps * warp_elems * sizeof(E);
};

// x: the parity of the step whose maximum it adds to (one thread of the launch also leaves
// the step count for y); y: that maximum, and the end of the step (one thread of the launch).
__device__ __forceinline__ int amax_parity(int* amax, bool one) {
  const int n = amax[kAmaxStep];
  if (one) amax[kAmaxCopy] = n;
  return n & 1;
}
__device__ __forceinline__ int amax_of_step(const int* amax) {
  return amax[kAmaxMax + (amax[kAmaxCopy] & 1)];
}
__device__ __forceinline__ void amax_end_step(int* amax) {
  const int n = amax[kAmaxCopy];
  amax[kAmaxNow] = amax[kAmaxMax + (n & 1)];
  amax[kAmaxMax + (~n & 1)] = 0;
  amax[kAmaxStep] = (int)((unsigned int)n + 1u);
}

template <bool CPLX>
__global__ void __launch_bounds__(kX64Warps * 32) k_sweep_x64(const __grid_constant__ SweepParams p) {
  using F = Field<double, CPLX>;
  using E = typename F::E;
  using G = X64Geom<CPLX>;
  constexpr int C = G::C, LD = G::LD, RPI = G::RPI, NG = G::NG;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  E* wbase = reinterpret_cast<E*>(smem) + (size_t)wib * G::warp_elems;
  auto buf = [&](int c) { return wbase + (c & 1) * (32 * LD); };   // chunk c's buffer
  E* rowf = wbase + 2 * 32 * LD;
  const long long nrows = (long long)p.ny * p.nz;
  const long long r0 = ((long long)blockIdx.x * kX64Warps + wib) * 32;
  pdl_begin();
  const int par = amax_parity(p.inc_amax, blockIdx.x == 0 && threadIdx.x == 0);
  if (r0 >= nrows) return;
  int vmax = 0;
  const int rows = (int)min(32LL, nrows - r0);
  const int nx = p.nx, P = p.pitch, head = p.head;
  E* field = static_cast<E*>(p.psi) + (size_t)r0 * P;
  const double s = *p.scale;
  const bool pw = p.pw != 0;
  const double cy = p.dt * p.g * s * s;
  const E* fx = static_cast<const E*>(p.band_fx);
  const E* A = static_cast<const E*>(p.A);
  const E* B = static_cast<const E*>(p.B);
  const E Ab = __ldg(A + nx - 1), Bb = __ldg(B + nx - 1);
  rowf[lane] = lane < rows ? __ldg(static_cast<const E*>(p.band_fyz) + r0 + lane) : F::zero();
  __syncwarp();

  const int lc = lane % C, lr = lane / C;   // load geometry: column and row offset
  const int nch = (nx + C - 1) / C;

  // chunk c of the warp's rows into b, lane = column: pending factor and pointwise
  // substep applied (columns past nx and rows past `rows` read as zero)
  auto load_chunk = [&](int c, E* b) {
    const int col = c * C + lc;
    const bool cin = col < nx;
    const E f = cin ? __ldg(fx + col) : F::zero();
    double cr[10];
    double2 Gc = make_double2(0.0, 0.0);
    if constexpr (!CPLX) {
      const double sf = s * f;
#pragma unroll
      for (int k = 0; k < 10; ++k) cr[k] = sf * kSignedInvFact[k];   // s fx (-1)^k / k!
    } else {
      Gc = make_double2(s * f.x, s * f.y);
    }
#pragma unroll
    for (int g0 = 0; g0 < 32; g0 += NG * RPI) {
      E xv[NG], rf[NG];
#pragma unroll
      for (int u = 0; u < NG; ++u) {
        const int rho = g0 + u * RPI + lr;
        xv[u] = (cin && rho < rows && GP_IN((r0 + rho) * P + col, nrows * P, p.status))
                    ? field[(size_t)rho * P + col] : F::zero();
        rf[u] = rowf[rho];
      }
      if (!pw) {
#pragma unroll
        for (int u = 0; u < NG; ++u) xv[u] = F::scaled(xv[u], s);
      } else if constexpr (!CPLX) {
        pointwise_real<NG>(xv, rf, cr, cy);
      } else {
        pointwise_cplx<NG>(xv, rf, Gc, cy);
      }
#pragma unroll
      for (int u = 0; u < NG; ++u) {
        vmax = imax(vmax, high_word(xv[u]));
        b[(g0 + u * RPI + lr) * LD + lc] = xv[u];
      }
    }
  };
  // chunk c of b to the field, lane = column
  auto store_chunk = [&](int c, const E* b) {
    const int col = c * C + lc;
    if (col >= nx) return;
#pragma unroll 8
    for (int rr = 0; rr < 32; rr += RPI) {
      const int rho = rr + lr;
      if (rho < rows && GP_IN((r0 + rho) * P + col, nrows * P, p.status))
        field[(size_t)rho * P + col] = b[rho * LD + lc];
    }
  };
  // forward values of chunk c's v (lane = row), in place; the element after the
  // chunk comes from the next chunk's buffer
  E prev = F::zero(), dprev = F::zero();
  auto forward = [&](int c, E* b, const E* bn) {
    E* rowp = b + lane * LD;
    const int j0 = c * C;
#pragma unroll
    for (int jj = 0; jj < C; ++jj) {
      const int j = j0 + jj;
      if (j < nx) {
        const E cur = rowp[jj];
        const E nxt = jj + 1 < C ? rowp[jj + 1] : (j + 1 < nx ? bn[lane * LD] : F::zero());
        const E bj = coef64(B, j, head, Bb);
        const E d = F::chain(bj, dprev, F::rhs(coef64(A, j, head, Ab), bj, prev, nxt, cur));
        rowp[jj] = d;
        prev = cur;
        dprev = d;
      }
    }
  };
  E unext = F::zero();
  auto back = [&](int c, E* b) {
    E* rowp = b + lane * LD;
    const int j0 = c * C;
#pragma unroll
    for (int jj = C - 1; jj >= 0; --jj) {
      const int j = j0 + jj;
      if (j < nx) {
        const E u = F::chain(coef64(B, j, head, Bb), unext, rowp[jj]);
        rowp[jj] = u;
        unext = u;
      }
    }
  };

  load_chunk(0, buf(0));
  for (int c = 0; c < nch; ++c) {
    if (c + 1 < nch) load_chunk(c + 1, buf(c + 1));
    __syncwarp();
    forward(c, buf(c), buf(c + 1));
    __syncwarp();
    // the last chunk's forward values stay in shared memory for the back substitution
    if (c + 1 < nch) store_chunk(c, buf(c));
  }
  vmax = __reduce_max_sync(0xffffffffu, vmax);
  if (lane == 0) atomicMax(p.inc_amax + kAmaxMax + par, vmax);
  for (int c = nch - 1; c >= 0; --c) {
    E* b = buf(c);
    if (c + 1 < nch) {
      const int col = c * C + lc;   // plain copy of the forward values back in
#pragma unroll 8
      for (int rr = 0; rr < 32; rr += RPI) {
        const int rho = rr + lr;
        b[rho * LD + lc] = (col < nx && rho < rows && GP_IN((r0 + rho) * P + col, nrows * P, p.status))
                               ? field[(size_t)rho * P + col] : F::zero();
      }
      __syncwarp();
    }
    back(c, b);
    __syncwarp();
    store_chunk(c, b);
  }
}

// -------------------------------------------------------------- sweeps y, z

// AXIS 1 (y) or 2 (z): thread g owns line (i = g mod nx, c = g / nx), c the z index
// (y sweep) or the y index (z sweep).  With NORM the block sums |u|^2 and the last
// block turns the partials into the renormalisation factor.
template <bool CPLX, int AXIS, bool NORM>
__global__ void __launch_bounds__(kLineThreads) k_sweep_line64(const __grid_constant__ SweepParams p) {
  using F = Field<double, CPLX>;
  using E = typename F::E;
  pdl_begin();
  if (AXIS == 1 && blockIdx.x == 0 && threadIdx.x == 0) amax_end_step(p.inc_amax);
  const int nx = p.nx, n = p.n, head = p.head;
  const long long nlines = (long long)nx * (AXIS == 1 ? p.nz : p.ny);
  const long long g = (long long)blockIdx.x * kLineThreads + threadIdx.x;
  double acc = 0.0;
  const int i = (int)(g % nx);
  const long long c = g / nx;
  const size_t P = (size_t)p.pitch;
  const size_t stride = AXIS == 1 ? P : P * (size_t)p.ny;
  const size_t first = (AXIS == 1 ? (size_t)c * P * p.ny : (size_t)c * P) + i;
  // the line's last element inside the field (bounds checks; the block still reaches
  // the norm's barriers)
  if (g < nlines && GP_IN(first + (size_t)(n - 1) * stride, (long long)p.nz * p.ny * (long long)P, p.status)) {
    E* line = static_cast<E*>(p.psi) + first;
    const E* A = static_cast<const E*>(p.A);
    const E* B = static_cast<const E*>(p.B);
    const E Ab = __ldg(A + n - 1), Bb = __ldg(B + n - 1);
    auto rd = [&](int j) -> E { return (j >= 0 && j < n) ? line[(size_t)j * stride] : F::zero(); };

    E prev = F::zero(), dprev = F::zero(), cur = rd(0);
    E nxt[kU64];
#pragma unroll
    for (int u = 0; u < kU64; ++u) nxt[u] = rd(u + 1);
    for (int j0 = 0; j0 < n; j0 += kU64) {
      E pre[kU64];
#pragma unroll
      for (int u = 0; u < kU64; ++u) pre[u] = rd(j0 + kU64 + u + 1);
#pragma unroll
      for (int u = 0; u < kU64; ++u) {
        const int j = j0 + u;
        if (j < n) {
          const E b = coef64(B, j, head, Bb);
          const E d = F::chain(b, dprev, F::rhs(coef64(A, j, head, Ab), b, prev, nxt[u], cur));
          line[(size_t)j * stride] = d;
          prev = cur;
          cur = nxt[u];
          dprev = d;
        }
      }
#pragma unroll
      for (int u = 0; u < kU64; ++u) nxt[u] = pre[u];
    }

    E unext = F::zero();
    E dv[kU64];
#pragma unroll
    for (int u = 0; u < kU64; ++u) dv[u] = rd(n - 1 - u);
    for (int j0 = n - 1; j0 >= 0; j0 -= kU64) {
      E pre[kU64];
#pragma unroll
      for (int u = 0; u < kU64; ++u) pre[u] = rd(j0 - kU64 - u);
#pragma unroll
      for (int u = 0; u < kU64; ++u) {
        const int j = j0 - u;
        if (j >= 0) {
          const E v = F::chain(coef64(B, j, head, Bb), unext, dv[u]);
          line[(size_t)j * stride] = v;
          unext = v;
          if constexpr (NORM) acc = fma(v, v, acc);
        }
      }
#pragma unroll
      for (int u = 0; u < kU64; ++u) dv[u] = pre[u];
    }
  }
  if constexpr (NORM) norm_finish(acc, p.partials, p.counter, gridDim.x, blockIdx.x, p.scale_out,
                                  p.status, p.dV);
}

// ------------------------------------------- sweeps y, z in increment form

// The CN solve of a line as v plus an increment: with K the second difference (zero
// ghosts), u = (I + aK)^{-1} (I - aK) v = v + 2a (I + aK)^{-1} s, s_j = v_{j-1} - 2 v_j +
// v_{j+1}, and I + aK = (a / rho) (1 - rho S) (1 - rho S^{-1}) (S the shift), so
//   y_j = s_j + rho y_{j-1},   z_j = y_j + rho z_{j+1},   u_j = v_j + 2 rho z_j.
// z vanishes at the ghosts (it is odd about them): z_n = 0 starts the backward pass and
// y_{-1} = -rho sum_k rho^k s_k the forward one.  |rho| <= 1/32 here (a <= 1/32), so the
// recursions forget: a segment's carry-in is the 12-term tail (head) of its neighbour
// (rho^12 < 2^-60), its far six terms in FP32 (rho^6 < 2^-29).
//
// What bounds it: FP64 arithmetic runs at 1/64 of FP32's rate here, so the increment is
// formed in two-part FP32 (gp_split.cuh) and one DADD per point is left (14.7 us of FP64
// pipe for 240 x 200 x 160 real points), against five FP64 operations per real point and
// 18 per complex one in k_sweep_line64.  Measured at 240 x 200 x 160 (GB300, event-timed
// launches): y 80 -> 43 us, z with its norm 106 -> 55 us; complex y 245 -> 92 us, z 290 ->
// 84 us.  Now bound by issue (2.1-2.3 of 4 instructions per clock, z with its norm 1.6; 113-116 per
// real point, 252-268 per complex one) and the FP64 pipe (33-38 %, z with its norm 61 %).
//
// Accuracy: s is exact and the increment's 48 bits are far below the final rounding as long as
// the increment is small against v.  Relative L2 error of a sweep against quadruple precision
// is about the root of (4e-17)^2, the rounding of u, plus (1e-14 |a| rms(s) / rms(v))^2: waves
// of 64 points at a = 0.025, k h = 0.3: 5.9e-17 (the FP64 recurrence 1.0e-16), 0.6: 9.7e-17,
// 0.9: 1.5e-16, white noise 4.5e-16 (1.2e-16); complex ones the same (recurrence 1.3e-16).  So
// a block whose points have |a| rms(s) > rms(v) / 128 evaluates its lines in FP64 (noise
// 5.7e-17), and so does one with values too large for FP32's range or not finite.
//
// A thread owns one 16-byte vector position (two real x or one complex x) and a segment of
// 16 points of the line; the block holds whole lines (all segments of inc_x positions),
// so the sweep works in place: every load precedes the first barrier, every store follows
// it.  The segment's values arrive by cp.async (all in flight, no registers held) in
// the thread's 16 shared-memory slots and the recursions work there in place; v is read
// again, four points ahead, for the final addition.  (The segment in registers: 128 of
// them, one block of 13 warps per SM, 68 us against 54 us for y.)  Blocks of about 128
// threads: 96 and 192 measured slower over the three axes.
constexpr int kIncL = 16;        // points per segment
constexpr int kIncG = 4;         // values of v read ahead in the backward pass
constexpr int kIncH = 12;        // terms of a carry
constexpr int kIncNear = 6;      // of those, the near ones in two-part arithmetic
constexpr int kIncThreads = 256; // most threads per block
constexpr double kIncRough = 128.0;  // a block is rough from rms(v) / rms(s) = kIncRough |a|

// Fields of that size and less are not for FP32's exponent range (gp_split.cuh): increments
// lose bits from 2^-150, which leaves 2^60 for the field's smaller values and for what a step
// changes.  They are computed in FP64 throughout.
constexpr int kIncTiny = (1023 - 90) << 20;

// A power of two that takes values times 2^kSplitShift to units of the field's largest (amax:
// its high word): that becomes 1 to 2.
__device__ __forceinline__ float inc_unit(int amax) {
  const int t = min(addmax0(amax, -kSplitOff), 253 << 20);
  return bits_f((uint32_t)(254 - (t >> 20)) << 23);
}

template <bool CPLX> struct IncRho;
template <> struct IncRho<false> {
  Coef r;
  double d;
  __device__ explicit IncRho(const SweepParams& p)
      : r(coef_pair(f2(p.rho_f[0]), f2(p.rho_f[1]))), d(p.rho[0]) {}
  __device__ __forceinline__ Prod mul(const Two& x) const { return two_mul(r, x); }
  __device__ __forceinline__ float2 mul_add(float2 x, float2 s) const { return fma2(r.h, x, s); }
  __device__ __forceinline__ double2 mul_add(double2 x, double2 s) const {
    return make_double2(fma(d, x.x, s.x), fma(d, x.y, s.y));
  }
};
template <> struct IncRho<true> {
  Coef r, i;   // i holds (-im, im): it multiplies (im, re)
  double2 d;
  __device__ explicit IncRho(const SweepParams& p)
      : r(coef_pair(f2(p.rho_f[0]), f2(p.rho_f[1]))),
        i(coef_pair(f2(-p.rho_f[2], p.rho_f[2]), f2(-p.rho_f[3], p.rho_f[3]))),
        d(make_double2(p.rho[0], p.rho[1])) {}
  __device__ __forceinline__ Prod mul(const Two& x) const {
    Two sw;
    sw.h = f2(x.h.y, x.h.x);
    sw.l = f2(x.l.y, x.l.x);
    return prod_add(two_mul(i, sw), two_mul(r, x));
  }
  __device__ __forceinline__ float2 mul_add(float2 x, float2 s) const {
    return fma2(i.h, f2(x.y, x.x), fma2(r.h, x, s));
  }
  __device__ __forceinline__ double2 mul_add(double2 x, double2 s) const { return cfma(d, x, s); }
};

// The 12-term carry sum_k rho^k at(k).
template <class RHO, class AT> __device__ __forceinline__ Two inc_carry(const RHO& rho, AT at) {
  float2 t = at(kIncH - 1).h;
#pragma unroll
  for (int k = kIncH - 2; k >= kIncNear; --k) t = rho.mul_add(t, at(k).h);
  Two w;
  w.h = t;
  w.l = f2(0.f);
#pragma unroll
  for (int k = kIncNear - 1; k >= 0; --k) w = two_add(at(k), rho.mul(w));
  return w;
}
template <class RHO, class AT> __device__ __forceinline__ double2 inc_carry64(const RHO& rho, AT at) {
  double2 t = at(kIncH - 1);
  for (int k = kIncH - 2; k >= 0; --k) t = rho.mul_add(t, at(k));
  return t;
}

__device__ __forceinline__ void put_two(float4* q, const Two& w) {
  *q = make_float4(w.h.x, w.h.y, w.l.x, w.l.y);
}
__device__ __forceinline__ Two get_two(const float4* q) {
  const float4 f = *q;
  return two_scalar(f2(f.x, f.y), f2(f.z, f.w));
}
__device__ __forceinline__ void put_d2(float4* q, double2 w) { *reinterpret_cast<double2*>(q) = w; }
__device__ __forceinline__ double2 get_d2(const float4* q) { return *reinterpret_cast<const double2*>(q); }

// One thread's segment [j0, j0 + kIncL) of a line of n points: slot[u TS] holds its v
// (zero from n on) and is overwritten; carry (and carry + T) are its exchange places, the
// neighbouring segments' lie X threads away; before / after: the values at j0 - 1 and
// j0 + kIncL (zero outside the line).  io.load(u): v again for the final addition;
// io.store(u, v, c): the increment c of point j0 + u (j0 + u < n); io.rd(j): v of any point
// of the line (FP64 path).  Every thread of the block must call it; `on`: the thread owns a
// segment; unit: inc_unit; limit: inc_rough; tiny: the FP64 path (these the same in every thread).
template <bool CPLX, class IO>
__device__ __forceinline__ void inc_segment(const IncRho<CPLX>& rho, float4* slot, int TS, float4* carry,
                                            int T, int X, int sg, int nseg, int j0, int n, bool on,
                                            double2 before, double2 after, float unit, float limit, bool tiny, IO& io) {
  int tmax = 0;
  // sums of |s|^2 and |v|^2 over half of the block's points (pairs of neighbours: no wave is
  // missed at its zeros), in units of the field's largest value; each value counts as 2^-10 at
  // least (noise below that, in the far tails, adds nothing to the field's error)
  float2 rough = f2(0.f), mass = f2(kIncL / 2 * 0x1p-20f);
  {
    const double2 v0 = get_d2(slot);
    Three a = split3(before.x, before.y, &tmax), b = split3(v0.x, v0.y, &tmax);
#pragma unroll 8
    for (int u = 0; u < kIncL; ++u) {
      const double2 vn = u + 1 < kIncL ? get_d2(slot + (u + 1) * TS) : after;
      const Three c = split3(vn.x, vn.y, &tmax);
      const Two s = second_difference(a, b, c);
      put_two(slot + u * TS, s);
      if (u % 4 >= 2) {
        const float2 sh = mul2(s.h, f2(unit)), vh = mul2(b.h, f2(unit));
        if (j0 + u < n) rough = fma2(sh, sh, rough);
        mass = fma2(vh, vh, mass);
      }
      a = b;
      b = c;
    }
  }
  // a tiny field, values out of range or a rough block (see kIncRough): in FP64
  __shared__ float2 part[kIncThreads / 32];
  {
    float2 sum = on ? f2(rough.x + rough.y, mass.x + mass.y) : f2(0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      sum = add2(sum, f2(__shfl_xor_sync(0xffffffffu, sum.x, o), __shfl_xor_sync(0xffffffffu, sum.y, o)));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
  }
  const bool big = __syncthreads_or(tiny || (on && tmax >= kSplitTooBig));
  float2 sum = part[0];
  for (unsigned int w = 1; w < blockDim.x / 32; ++w) sum = add2(sum, part[w]);
  if (!big && sum.x * limit < sum.y) {
    // carry out to the next segment: the tail of s; the first segment also starts itself
    put_two(carry, inc_carry(rho, [&](int k) { return get_two(slot + (kIncL - 1 - k) * TS); }));
    Prod pr = prod_zero();
    if (sg == 0)
      pr = rho.mul(two_neg(prod_two(rho.mul(inc_carry(rho, [&](int k) { return get_two(slot + k * TS); })))));
    __syncthreads();
    if (sg > 0) pr = rho.mul(get_two(carry - X));
#pragma unroll 4
    for (int u = 0; u < kIncL; ++u) {
      const Two y = j0 + u < n ? two_add(get_two(slot + u * TS), pr) : two_zero();
      put_two(slot + u * TS, y);
      pr = rho.mul(y);
    }
    put_two(carry + T, inc_carry(rho, [&](int k) { return get_two(slot + k * TS); }));
    double2 v[kIncG];   // v again, the last group
#pragma unroll
    for (int q = 0; q < kIncG; ++q) v[q] = io.load(kIncL - kIncG + q);
    __syncthreads();
    pr = prod_zero();
    if (on && sg + 1 < nseg) pr = rho.mul(get_two(carry + T + X));
    for (int g = kIncL - kIncG; g >= 0; g -= kIncG) {
      double2 nxt[kIncG];   // the group below, in flight while this one is computed
#pragma unroll
      for (int q = 0; q < kIncG; ++q) nxt[q] = g > 0 ? io.load(g - kIncG + q) : v[q];
#pragma unroll
      for (int q = kIncG - 1; q >= 0; --q) {
        const int u = g + q;
        pr = rho.mul(two_add(get_two(slot + u * TS), pr));
        const Two c = two_norm(pr);
        const double2 cd = make_double2(to_double(c.h.x, c.l.x, 1), to_double(c.h.y, c.l.y, 1));
        if (on && j0 + u < n) io.store(u, v[q], cd);
      }
#pragma unroll
      for (int q = 0; q < kIncG; ++q) v[q] = nxt[q];
    }
  } else {
    // the same recursions in FP64
    {
      double2 a = before, b = io.rd(j0);
      for (int u = 0; u < kIncL; ++u) {
        const double2 c = io.rd(j0 + u + 1);
        put_d2(slot + u * TS, make_double2((c.x - b.x) - (b.x - a.x), (c.y - b.y) - (b.y - a.y)));
        a = b;
        b = c;
      }
    }
    const double2 zero = make_double2(0.0, 0.0);
    put_d2(carry, inc_carry64(rho, [&](int k) { return get_d2(slot + (kIncL - 1 - k) * TS); }));
    double2 prev = zero;
    if (sg == 0) {
      const double2 t = rho.mul_add(inc_carry64(rho, [&](int k) { return get_d2(slot + k * TS); }), zero);
      prev = make_double2(-t.x, -t.y);
    }
    __syncthreads();
    if (sg > 0) prev = get_d2(carry - X);
    for (int u = 0; u < kIncL; ++u) {
      prev = j0 + u < n ? rho.mul_add(prev, get_d2(slot + u * TS)) : zero;
      put_d2(slot + u * TS, prev);
    }
    put_d2(carry + T, inc_carry64(rho, [&](int k) { return get_d2(slot + k * TS); }));
    __syncthreads();
    double2 z = zero;
    if (on && sg + 1 < nseg) z = get_d2(carry + T + X);
    for (int u = kIncL - 1; u >= 0; --u) {
      z = rho.mul_add(z, get_d2(slot + u * TS));
      const double2 v = io.load(u), c = rho.mul_add(z, zero);
      if (on && j0 + u < n) io.store(u, v, make_double2(2.0 * c.x, 2.0 * c.y));
    }
  }
}

// (80 registers: six blocks of 128 threads per SM, as many as their shared memory leaves room for;
// the z sweep with its norm took 116 by itself, and 61.9 us instead of 55.3)
template <bool CPLX, int AXIS, bool NORM>
__global__ void __maxnreg__(80) k_sweep_inc64(const __grid_constant__ SweepParams p) {
  extern __shared__ __align__(16) float4 inc_smem[];
  const int X = p.inc_x, nseg = p.inc_seg, n = p.n;
  const int tid = threadIdx.x, T = blockDim.x;
  float4* slot = inc_smem + tid;               // [kIncL][T]: v, then s, then y (two-part or FP64)
  float4* carry = inc_smem + kIncL * T + tid;  // [2][T]: tails of s, heads of y
  pdl_begin();
  const int sg = tid / X, xl = tid - sg * X;
  const int nvec = CPLX ? p.nx : (p.nx + 1) / 2;
  const int ntile = (nvec + X - 1) / X;
  const int o = blockIdx.x / ntile, xv = (blockIdx.x - o * ntile) * X + xl;
  const size_t P = (size_t)(CPLX ? p.pitch : p.pitch / 2);   // row pitch in vectors
  const int j0 = sg * kIncL;
  struct IO {
    double2* line;
    size_t stride;
    int j0, n;
    bool on;
    double acc;
    long long first, nall;   // bounds checks
    int* status;
    __device__ bool inside(int j) const {
      return on && j >= 0 && j < n && GP_IN(first + (long long)j * (long long)stride, nall, status);
    }
    __device__ double2 rd(int j) const { return inside(j) ? line[(size_t)j * stride] : make_double2(0.0, 0.0); }
    __device__ double2 load(int u) const { return rd(j0 + u); }
    __device__ void store(int u, double2 v, double2 c) {
      const double2 w = make_double2(v.x + c.x, v.y + c.y);
      if (!GP_IN(first + (long long)(j0 + u) * (long long)stride, nall, status)) return;
      line[(size_t)(j0 + u) * stride] = w;
      if constexpr (NORM) acc = fma(w.x, w.x, fma(w.y, w.y, acc));
    }
  } io;
  io.on = sg < nseg && xv < nvec;
  io.stride = AXIS == 1 ? P : P * (size_t)p.ny;
  io.first = (long long)((AXIS == 1 ? (size_t)o * P * p.ny : (size_t)o * P) + (io.on ? xv : 0));
  io.nall = (long long)P * p.ny * p.nz;   // vectors of the field
  io.line = reinterpret_cast<double2*>(p.psi) + io.first;
  io.j0 = j0;
  io.n = n;
  io.acc = 0.0;
  io.status = p.status;
#pragma unroll
  for (int u = 0; u < kIncL; ++u) {
    const bool ok = io.inside(j0 + u);
    cp_async16_zfill(slot + u * T, io.line + (ok ? (size_t)(j0 + u) * io.stride : 0), ok);
  }
  cp_async_commit();
  const double2 before = io.rd(j0 - 1), after = io.rd(j0 + kIncL);
  const IncRho<CPLX> rho(p);
  const int amax = AXIS == 1 ? amax_of_step(p.inc_amax) : p.inc_amax[kAmaxNow];
  if (AXIS == 1 && blockIdx.x == 0 && tid == 0) amax_end_step(p.inc_amax);
  cp_async_wait<0>();
  inc_segment<CPLX>(rho, slot, T, carry, T, X, sg, nseg, j0, n, io.on, before, after, inc_unit(amax),
                    p.inc_rough, amax < kIncTiny, io);
  if constexpr (NORM) norm_finish(io.acc, p.partials, p.counter, gridDim.x, blockIdx.x, p.scale_out,
                                  p.status, p.dV);
}

// ---------------------------------------------- sweep x in increment form

// The pending factor and the pointwise substep as an increment too: with f the trap
// factor, e = s f exp(-y) - 1 (real; complex: s f cis(-y) - 1), y = dt g s^2 |v|^2,
//   e = E + (1 + E) q,   E = ex + er + ex er,   q = exp(-y) - 1 (cis(-y) - 1),
// ex the column's factor less 1 (two-part table, from expm1 / sin^2 in FP64), er the
// row's times the pending factor, less 1; v' = v + v e: real, e as FP64 and one DFMA; complex,
// v e in two-part FP32 and one DADD per part.  q is skipped where every lane of the warp has
// |y| < 2^-56, and taken from short or long Taylor sums by the size of y.
//
// 48 bits of e are 53 of v' as long as e is small.  Relative error against quadruple precision,
// two-part / FP64 products (1e-16), at |E| = 1e-3, 1/64, 0.1, 0.28: real 0.6 / 0.9, 0.8 / 0.9, 2.7 /
// 1.0, 6.6 / 1.0, complex 0.6 / 1.1, 1.0 / 1.1, 5.0 / 1.1, 17 / 1.1; at y = 1/128, 0.02, 0.1: 0.7 /
// 1.0, 1.2 / 1.1, 8.6 / 1.1 and (1/256) 0.7 / 1.0, 1.3 / 1.0, 5.4 / 1.2.  So
//   |y| from kIncY to kIncLead: q's leading term (-y, -i y) in FP64, four operations per real
//     value and seven per complex one, the rest of e as before;
//   |E| from kIncE to kIncBigE: E in FP64 too, nine and eighteen operations, unless the value is so
//     small against the field's largest that two parts' error stays below 3e-17 of that;
//   |y| > kIncLead, |E| > kIncBigE, values out of range, a tiny field: products in FP64 (they round the
//     factors' product alike at every step: an error that grows with the steps),
// each for a warp as a whole.
// Measured at 240 x 200 x 160 with the solve: 284 us (k_sweep_x64 at its shortest
// polynomial; 620 us where the density calls for the longer one) -> 87 us, complex 686
// -> 197 us; 189 and 502 instructions per point, FP64 pipe 55 and 47 %.
//
// A block owns inc_x row vectors (real: pairs of rows; complex: rows) and works in three
// passes: lanes along the rows (coalesced) for the substep, v' to the field and to the
// segments' slots in shared memory; one segment of 16 columns per thread for the solve
// (as the y / z kernel; the increments replace the slots); lanes along the rows again
// for u = v' + c.
constexpr float kIncBigE = 0.25f;
constexpr float kIncE = 1.f / 64;
template <bool CPLX> constexpr float kIncY = CPLX ? 1.f / 256 : 1.f / 128;
constexpr float kIncLead = 1.f / 16;

// v' in FP64 (f: the folded factor times the trap factors; real, complex)
__device__ __forceinline__ double pointwise64(double v, double f, double cy) {
  const double y = cy * (v * v);
  const unsigned long long mb = abs_bits(y);
  double q;
  if (mb <= kBits2m10) {
    q = fma(y, fma(y, fma(y, fma(y, kSignedInvFact[4], kSignedInvFact[3]), 0.5), -1.0), 1.0);
  } else if (mb <= kBits2m4) {
    q = fma(y, kSignedInvFact[9], kSignedInvFact[8]);
#pragma unroll
    for (int k = 7; k >= 0; --k) q = fma(y, q, kSignedInvFact[k]);
  } else {
    q = exp(-y);
  }
  return v * f * q;
}

__device__ __forceinline__ double2 pointwise64(double2 v, double2 f, double cy) {
  const double th = cy * fma(v.x, v.x, v.y * v.y);
  const unsigned long long mb = abs_bits(th);
  double cs, sn;
  if (mb <= kBits2m8) {
    const double t2 = th * th;
    cs = fma(t2, fma(t2, 1.0 / 24.0, -0.5), 1.0);
    sn = th * fma(t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), 1.0);
  } else {
    sincos(th, &sn, &cs);
  }
  return cmul(cmul(v, f), make_double2(cs, -sn));
}

// The real pair's or complex value's v' with the leading terms in FP64: y's (|y| <= kIncLead), and if
// `wide` E's, from the column's factor(s) less 1 (ca, cb; complex: ca) and the row's (er), which loses
// nothing to the factors' product; dense: y is not nothing; e: E, cyc: cy, V: v in two parts.
template <bool CPLX>
__device__ __forceinline__ double2 pointwise_lead(double2 v, Two e, const Two& V, const Coef& cyc, double cy, bool dense,
                                                  bool wide, double2 ca, double2 er) {
  Two rest = two_zero();
  if (dense) {
    const Two h = two_scalar(mul2(V.h, f2(0x1p-56f)), mul2(V.l, f2(0x1p-56f)));
    Two d = two_mul(h, h);
    if (CPLX) d = two_add(d, two_swap(d));
    const Two y = prod_two(two_mul(cyc, d));
    rest = CPLX ? two_cis_neg_rest(y) : two_expm1_neg_rest(y);
    const Two q = two_add(rest, CPLX ? two_scalar(f2(0.f, -y.h.y), f2(0.f, -y.l.y)) : two_neg(y));
    rest = two_add(rest, CPLX ? two_cmul(e, q) : two_mul(e, q));
  }
  if (!wide) rest = two_add(e, rest);
  const Two c = two_norm(CPLX ? two_cmul(V, rest) : rest);
  const int k = CPLX ? 0 : kSplitShift;
  const double2 w = make_double2(to_double(c.h.x, c.l.x, k), to_double(c.h.y, c.l.y, k));
  double2 E = make_double2(0.0, 0.0);
  if constexpr (CPLX) {
    const double th = cy * fma(v.x, v.x, v.y * v.y);
    if (!wide) return make_double2(v.x + fma(th, v.y, w.x), v.y + fma(-th, v.x, w.y));
    E = cfma(ca, er, make_double2(ca.x + er.x, ca.y + er.y));
    const double2 dv = cfma(v, make_double2(E.x, E.y - th), w);
    return make_double2(v.x + dv.x, v.y + dv.y);
  } else {
    if (wide) E = make_double2(fma(ca.x, er.x, ca.x + er.x), fma(ca.y, er.x, ca.y + er.x));
    return make_double2(fma(v.x, E.x + fma(-cy * v.x, v.x, w.x), v.x), fma(v.y, E.y + fma(-cy * v.y, v.y, w.y), v.y));
  }
}

// (Registers, 240 x 200 x 160: real 96, 87 us, against 97 with the FP64 paths laid out freely; complex
// 128, 197 us and 27.3 at 101 x 77 x 53; 80, 178 and 29.3)
template <bool CPLX>
__global__ void __maxnreg__(CPLX ? 128 : 96) k_sweep_xinc64(const __grid_constant__ SweepParams p) {
  extern __shared__ __align__(16) float4 inc_smem[];
  const int X = p.inc_x, nseg = p.inc_seg, nx = p.nx;
  const int tid = threadIdx.x, T = blockDim.x, TS = T + 1;   // one slot of padding: see `place`
  constexpr int RPV = CPLX ? 1 : 2;                          // rows per row vector
  const int rows_t = X * RPV;
  float4* slots = inc_smem;                                  // [kIncL][TS]
  float4* carry = inc_smem + kIncL * TS + tid;               // [2][T]
  float4* rowc = inc_smem + kIncL * TS + 2 * T;              // per tile row: the row's factor
  const long long nrows = (long long)p.ny * p.nz;
  const long long r0 = (long long)blockIdx.x * rows_t;
  const int rows = (int)min((long long)rows_t, nrows - r0);
  const int P = CPLX ? p.pitch : p.pitch / 2, nvec = CPLX ? nx : (nx + 1) / 2;   // vectors per row
  double2* field = reinterpret_cast<double2*>(p.psi) + (size_t)r0 * P;
  const long long nall = nrows * P, at0 = r0 * P;            // bounds checks
  (void)nall;
  (void)at0;
  __shared__ double head_d[3];   // the factor applied ahead, the one folded in, dt g s^2
  __shared__ int head_max, head_now;   // the block's largest value, the field's before the substep
  const IncRho<CPLX> rho(p);
  pdl_begin();
  // FP64 is slow even a few operations per thread: one thread forms the block's scalars
  if (tid == 0) {
    const double s = *p.scale;
    // folded into the rows' increments unless it is far from 1 (or not a number)
    const bool fold = fabs(s - 1.0) <= 0.0625;
    head_d[0] = fold ? 1.0 : s;
    head_d[1] = fold ? s : 1.0;
    head_d[2] = p.dt * p.g * head_d[1] * head_d[1];
    head_max = 0;
    // (kAmaxNow is that of the field without its pending factor)
    const int now = p.inc_amax[kAmaxNow];
    head_now = fold ? now : high_word(__hiloint2double(now, 0) * s);
  }
  const int par = amax_parity(p.inc_amax, blockIdx.x == 0 && tid == 0);
  __syncthreads();
  const bool tiny = head_now < kIncTiny;
  const float unit = inc_unit(head_now);
  const double spre = head_d[0], s = head_d[1], cy = head_d[2];
  const bool pre = __double2hiint(spre) != 0x3ff00000 || __double2loint(spre) != 0;
  const bool pw = p.pw != 0;
  const bool work = pw || __double2hiint(s) != 0x3ff00000 || __double2loint(s) != 0;
  // rows' factors f = s (trap factor) and er = f - 1: real (f, f', er, er'); complex
  // f, f with its parts exchanged, er, each (re, im, re', im')
  for (int r = tid; r < rows; r += T) {
    if constexpr (!CPLX) {
      const double f0 = pw ? static_cast<const double*>(p.band_fyz)[r0 + r] : 1.0;
      const double f = f0 * s, e = fma(f0, s, -1.0);
      const float fh = (float)f, eh = (float)e;
      rowc[r] = make_float4(fh, (float)(f - (double)fh), eh, (float)(e - (double)eh));
    } else {
      const double2 f0 = pw ? static_cast<const double2*>(p.band_fyz)[r0 + r] : make_double2(1.0, 0.0);
      const double fr = f0.x * s, fi = f0.y * s, er = fma(f0.x, s, -1.0);
      const float rh = (float)fr, ih = (float)fi, eh = (float)er;
      const float rl = (float)(fr - (double)rh), il = (float)(fi - (double)ih);
      rowc[3 * r] = make_float4(rh, ih, rl, il);
      rowc[3 * r + 1] = make_float4(ih, rh, il, rl);
      rowc[3 * r + 2] = make_float4(eh, ih, (float)(er - (double)eh), il);
    }
  }
  __syncthreads();
  const double cyp = pw ? cy : 0.0;
  const Coef cyc = coef_pair(f2((float)cyp), f2((float)(cyp - (double)(float)cyp)));
  int vmax = 0;
  // In the two passes along the rows a thread keeps to one vector position (column) per
  // chunk of `per` positions and walks down the tile, `grp` rows at a time.  Column c of
  // row r lies in the slot of segment c / 16, point c mod 16, row vector r / RPV; points
  // are TS slots apart, so that lanes on consecutive columns spread over the banks.
  const int nchunk = (nvec + T - 1) / T, per = (nvec + nchunk - 1) / nchunk, grp = T / per;
  const int ro = tid / per, co = tid - ro * per;
  const int rounds = (rows_t + grp - 1) / grp;
  auto place = [&](int cv) {   // of row 0; row r is 16 / RPV bytes times r further
    const int c = CPLX ? cv : 2 * cv;
    return reinterpret_cast<double*>(slots + (c % kIncL) * TS + (c / kIncL) * X);
  };
  for (int ch = 0; ch < nchunk; ++ch) {
    const int cv = ch * per + co;
    const bool con = ro < grp && cv < nvec;
    float4 ext = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pw && con) ext = __ldg(static_cast<const float4*>(p.inc_ex) + cv);
    // the column's factor as the constant of the products with the rows' factors
    const Coef ex = CPLX ? coef_pair(f2(ext.x), f2(ext.z)) : coef_pair(f2(ext.x, ext.y), f2(ext.z, ext.w));
    const Coef exi = coef_pair(f2(-ext.y, ext.y), f2(-ext.w, ext.w));
    double* dst = place(con ? cv : 0);
    const double2 zero = make_double2(0.0, 0.0);
    auto fetch = [&](int r) {
      return con && r < rows && GP_IN(at0 + (long long)r * P + cv, nall, p.status)
                 ? field[(size_t)r * P + cv] : zero;
    };
    auto factor = [&](const float4* rc) {   // E of the column and a row
      if constexpr (!CPLX) {
        const float4 f = rc[0];
        return two_add(two_scalar(f2(f.z), f2(f.w)), two_mul(ex, two_scalar(f2(f.x), f2(f.y))));
      } else {
        return two_add(get_two(rc + 2), prod_add(two_mul(exi, get_two(rc + 1)), two_mul(ex, get_two(rc))));
      }
    };
    double2 nxt = fetch(ro);
    for (int q = 0; q < rounds; ++q) {   // (full rounds: every lane takes part in the votes)
      const int r = ro + q * grp;
      const bool live = con && r < rows;
      double2 v = nxt;
      if (q + 1 < rounds) nxt = fetch(r + grp);
      if (pre) {
        v.x *= spre;
        v.y *= spre;
      }
      const int vm = high_word(v);
      vmax = imax(vmax, vm);
      if (work) {
        const float4* rc = rowc + (CPLX ? 3 : 1) * (live ? r : 0);
        Two e = factor(rc);
        const float em = fmaxf(fabsf(e.h.x), fabsf(e.h.y));
        const float size = bits_f((uint32_t)min(addmax0(vm, -kSplitOff), 253 << 20) << 3) * unit;
        bool ok = !tiny && (em <= kIncE || (em <= kIncBigE && em * size <= 0x1p-8f));
        int tmax = 0;
        float ym = 0.f;
        Two V;
        if (CPLX) {
          V = split2(v.x, v.y, &tmax);
          ok = ok && tmax < kSplitTooBig;
        }
        if (pw && !__all_sync(0xffffffffu, vm < p.inc_quiet)) {
          if (!CPLX) V = split2(v.x, v.y, &tmax);
          // y = cy |v|^2 in natural scale
          const Two h = two_scalar(mul2(V.h, f2(0x1p-56f)), mul2(V.l, f2(0x1p-56f)));
          Two d = two_mul(h, h);
          if (CPLX) d = two_add(d, two_swap(d));   // re^2 + im^2 in both lanes
          const Two y = prod_two(two_mul(cyc, d));
          ym = fmaxf(fabsf(y.h.x), fabsf(y.h.y));
          ok = ok && tmax < kSplitTooBig;
          Two qv;
          if (__all_sync(0xffffffffu, ym <= 0x1p-10f || !ok))
            qv = CPLX ? two_cis_neg_m1_small(y) : two_expm1_neg_small(y);
          else
            qv = CPLX ? two_cis_neg_m1(y) : two_expm1_neg(y);
          e = two_add(two_add(e, qv), CPLX ? two_cmul(e, qv) : two_mul(e, qv));
        }
        if (__all_sync(0xffffffffu, (ok && ym <= kIncY<CPLX>) || !live)) {
          if constexpr (CPLX) {
            const Two c = two_norm(two_cmul(V, e));
            v.x += to_double(c.h.x, c.l.x, 0);
            v.y += to_double(c.h.y, c.l.y, 0);
          } else {
            const Two c = two_norm(e);
            v.x = fma(v.x, to_double(c.h.x, c.l.x, kSplitShift), v.x);
            v.y = fma(v.y, to_double(c.h.y, c.l.y, kSplitShift), v.y);
          }
        } else {
          int big = 0;
          const Two W = split2(v.x, v.y, &big);
          const bool wide = !__all_sync(0xffffffffu, ok || !live);
          const bool fit = !tiny && em <= kIncBigE && ym <= kIncLead && big < kSplitTooBig;
          if (__all_sync(0xffffffffu, fit || !live)) {
            double2 ca = make_double2(0.0, 0.0), er = ca;
            if (wide && live) {
              // the column's factor less 1: small, from its two parts; else the FP64 factor's is closer
              auto sum = [](float a, float b) { return to_double(a, 0.f, kSplitShift) + to_double(b, 0.f, kSplitShift); };
              const bool parts = em <= 0.0625f;
              if (pw) {
                if (parts) {
                  ca = make_double2(sum(ext.x, ext.z), sum(ext.y, ext.w));
                } else if constexpr (CPLX) {
                  ca = static_cast<const double2*>(p.band_fx)[cv];
                  ca.x -= 1.0;
                } else {
                  const double* fx = static_cast<const double*>(p.band_fx) + 2 * cv;
                  ca = make_double2(fx[0] - 1.0, fx[1] - 1.0);
                }
              }
              if constexpr (CPLX) {
                const double2 rf = pw ? static_cast<const double2*>(p.band_fyz)[r0 + r] : make_double2(1.0, 0.0);
                er = make_double2(fma(rf.x, s, -1.0), rf.y * s);
              } else {
                er.x = fma(pw ? static_cast<const double*>(p.band_fyz)[r0 + r] : 1.0, s, -1.0);
              }
            }
            const bool dense = pw && !__all_sync(0xffffffffu, vm < p.inc_quiet);
            v = pointwise_lead<CPLX>(v, factor(rc), W, cyc, dense ? cyp : 0.0, dense, wide, ca, er);
          } else if (live) {
            // |y| < 2^-56: the factor alone (the far field, where |E| is large and v small: two
            // to ten FP64 operations instead of ten to thirty; 240 x 200 x 160 at h = 0.2, where
            // that is most of the grid: x 237 -> 119 us, complex 453 -> 264)
            const bool quiet = !pw || vm < p.inc_quiet;
            if constexpr (!CPLX) {
              const double fr = pw ? s * static_cast<const double*>(p.band_fyz)[r0 + r] : s;
              const double* fx = static_cast<const double*>(p.band_fx);
              const double f0 = pw ? fr * fx[2 * cv] : fr, f1 = pw ? fr * fx[2 * cv + 1] : fr;
              v.x = quiet ? v.x * f0 : pointwise64(v.x, f0, cyp);
              v.y = quiet ? v.y * f1 : pointwise64(v.y, f1, cyp);
            } else {
              const double2 rf = pw ? static_cast<const double2*>(p.band_fyz)[r0 + r] : make_double2(1.0, 0.0);
              const double2 f = pw ? static_cast<const double2*>(p.band_fx)[cv] : make_double2(1.0, 0.0);
              const double2 f0 = cmul(make_double2(s * f.x, s * f.y), rf);
              v = quiet ? cmul(v, f0) : pointwise64(v, f0, cyp);
            }
          }
        }
      }
      if (live && (work || pre) && GP_IN(at0 + (long long)r * P + cv, nall, p.status))
        field[(size_t)r * P + cv] = v;
      if (con && r < rows_t) {
        if constexpr (CPLX) {
          *reinterpret_cast<double2*>(dst + 2 * r) = v;
        } else {
          dst[r] = v.x;
          dst[r + 2 * TS] = v.y;
        }
      }
    }
  }
  vmax = __reduce_max_sync(0xffffffffu, vmax);
  if ((tid & 31) == 0) atomicMax(&head_max, vmax);
  __syncthreads();
  if (tid == 0) atomicMax(p.inc_amax + kAmaxMax + par, head_max);
  {
    const int sg = tid / X, xl = tid - sg * X;
    const int j0 = sg * kIncL;
    struct IO {
      float4* slot;
      const double* row[2];   // v' of the thread's row(s) in the field
      int TS, j0, nx, pitch;
      bool on;
      long long first, nall;   // bounds checks: first vector of row[0], the field's vectors
      int* status;
      __device__ double2 rd(int j) const {
        if (!on || j < 0 || j >= nx) return make_double2(0.0, 0.0);
        if (!GP_IN(first + (!CPLX && row[1] ? pitch : 0) + (CPLX ? j : j / 2), nall, status)) return make_double2(0.0, 0.0);
        if constexpr (CPLX) return reinterpret_cast<const double2*>(row[0])[j];
        return make_double2(row[0][j], row[1] ? row[1][j] : 0.0);
      }
      __device__ double2 load(int) const { return make_double2(0.0, 0.0); }
      __device__ void store(int u, double2, double2 c) { put_d2(slot + u * TS, c); }
    } io;
    io.on = sg < nseg && xl * RPV < rows;
    io.slot = slots + tid;
    io.TS = TS;
    io.j0 = j0;
    io.nx = nx;
    io.pitch = P;
    io.first = at0 + (long long)(xl * RPV) * P;
    io.nall = nall;
    io.status = p.status;
    io.row[0] = reinterpret_cast<const double*>(field + (size_t)(xl * RPV) * P);
    io.row[1] = !CPLX && xl * RPV + 1 < rows ? reinterpret_cast<const double*>(field + (size_t)(xl * RPV + 1) * P)
                                             : nullptr;
    // columns past the row read as zero
    for (int u = max(0, (CPLX ? nx : 2 * nvec) - j0); u < kIncL; ++u)
      if (tid < X * nseg) put_d2(slots + tid + u * TS, make_double2(0.0, 0.0));
    double2 before = make_double2(0.0, 0.0), after = before;
    if (io.on && sg > 0) before = get_d2(slots + tid - X + (kIncL - 1) * TS);
    if (io.on && sg + 1 < nseg) after = get_d2(slots + tid + X);
    __syncthreads();
    inc_segment<CPLX>(rho, slots + tid, TS, carry, T, X, sg, nseg, j0, nx, io.on, before, after,
                      unit, p.inc_rough, tiny, io);
  }
  __syncthreads();
  for (int ch = 0; ch < nchunk; ++ch) {
    const int cv = ch * per + co;
    if (ro >= grp || cv >= nvec) continue;
    const double* src = place(cv);
    const bool pad = !CPLX && 2 * cv + 1 >= nx;
#pragma unroll 4
    for (int r = ro; r < rows; r += grp) {
      if (!GP_IN(at0 + (long long)r * P + cv, nall, p.status)) continue;
      const double2 v = field[(size_t)r * P + cv];
      const double2 c = CPLX ? *reinterpret_cast<const double2*>(src + 2 * r)
                             : make_double2(src[r], pad ? 0.0 : src[r + 2 * TS]);
      field[(size_t)r * P + cv] = make_double2(v.x + c.x, v.y + c.y);
    }
  }
}

// ------------------------------------------------------------------ launchers

size_t x64_smem(bool complex_field) {
  return complex_field ? X64Geom<true>::smem : X64Geom<false>::smem;
}

static cudaError_t inc64_prepare();
cudaError_t sweep64_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_sweep_x64<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)X64Geom<false>::smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_sweep_x64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)X64Geom<true>::smem);
  if (e == cudaSuccess) e = inc64_prepare();
  return e;
}

long long sweep64_blocks(int axis, int nx, int ny, int nz) {
  if (axis == 0) {
    const long long warps = ((long long)ny * nz + 31) / 32;
    return (warps + kX64Warps - 1) / kX64Warps;
  }
  const long long lines = (long long)nx * (axis == 1 ? nz : ny);
  return (lines + kLineThreads - 1) / kLineThreads;
}

cudaError_t launch_sweep64(int axis, const SweepParams& p, bool complex_field, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = st;
  cfg.gridDim = dim3((unsigned)sweep64_blocks(axis, p.nx, p.ny, p.nz));
  if (axis == 0) {
    cfg.blockDim = dim3(kX64Warps * 32);
    cfg.dynamicSmemBytes = x64_smem(complex_field);
    return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_x64<true>, p)
                         : cudaLaunchKernelEx(&cfg, k_sweep_x64<false>, p);
  }
  cfg.blockDim = dim3(kLineThreads);
  if (axis == 1)
    return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_line64<true, 1, false>, p)
                         : cudaLaunchKernelEx(&cfg, k_sweep_line64<false, 1, false>, p);
  // the norm is summed in imaginary time only (real field)
  return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_line64<true, 2, false>, p)
                       : cudaLaunchKernelEx(&cfg, k_sweep_line64<false, 2, true>, p);
}

// Lines of at least 16 points (a carry's 12 terms lie within a segment and its line) and
// a <= 1/32 (rho^12 < 2^-60).  Positions per block: enough for about 256 threads on short
// lines, fewer on long ones so that a block keeps to kIncThreads; whole tiles of nearly
// equal width.
bool inc64_setup(int axis, SweepParams* p, std::complex<double> a, bool complex_field, int nsm) {
  p->inc_x = 0;
  if (p->n < 16 || std::abs(a) > 1.0 / 32) return false;
  // block rows: 16-byte vectors along x (y, z sweeps) or pairs of rows / rows (x sweep)
  const long long nrows = (long long)p->ny * p->nz;
  const int nvec = axis == 0 ? (int)(complex_field ? nrows : (nrows + 1) / 2)
                             : complex_field ? p->nx : (p->nx + 1) / 2;
  const int nseg = (p->n + kIncL - 1) / kIncL;
  const int most = std::max(1, std::min(kIncThreads / nseg, std::max(axis == 0 ? 4 : 8, 128 / nseg)));
  int tiles = (nvec + most - 1) / most;
  // x: an equal number of blocks for every SM (its passes along the rows take the longer the
  // more rows a block has, and a block more than its neighbours an SM's whole share: 128 x 96 x 64
  // 192 blocks 41 us, 280 33; 64 x 48 x 32 24 blocks 18.5 us, 128 14.6, complex 48 blocks 20.5,
  // 140 16.6; 300 x 256 plane 22 blocks 21 us, 128 14.8)
  if (axis == 0) tiles = (tiles + nsm - 1) / nsm * nsm;
  p->inc_seg = nseg;
  p->inc_x = (nvec + tiles - 1) / tiles;
  p->inc_threads = (p->inc_x * nseg + 31) / 32 * 32;
  // x, grids of at most two blocks per SM: more threads than segments share the passes along the
  // rows (64 x 48 x 32, then 24 blocks: x 22.5 -> 19.3 us, 101 x 77 x 53 complex step 75 -> 58 us;
  // larger grids would lose resident blocks)
  if (axis == 0 && (nvec + p->inc_x - 1) / p->inc_x <= 2 * nsm) p->inc_threads = kIncThreads;
  p->inc_rough = (float)(kIncRough * kIncRough * std::norm(a));
  const std::complex<double> r = 2.0 * a / (1.0 + 2.0 * a + std::sqrt(1.0 + 4.0 * a));
  const double part[2] = {r.real(), r.imag()};
  for (int q = 0; q < 2; ++q) {
    p->rho[q] = part[q];
    p->rho_f[2 * q] = (float)part[q];
    p->rho_f[2 * q + 1] = (float)(part[q] - (double)p->rho_f[2 * q]);
  }
  return true;
}

// x: slots with one of padding per point, carries, the rows' factors (real: two rows of one
// float4 per row vector; complex: one row of three)
static size_t inc64_x_smem(unsigned threads, int X) {
  return ((size_t)kIncL * (threads + 1) + 2 * threads + 3 * X) * sizeof(float4);
}

// shared-memory limit of the increment kernels (blocks of kIncThreads)
static cudaError_t inc64_prepare() {
  void (*const k[5])(SweepParams) = {k_sweep_inc64<false, 1, false>, k_sweep_inc64<false, 1, true>,
                                     k_sweep_inc64<false, 2, true>, k_sweep_inc64<true, 1, false>,
                                     k_sweep_inc64<true, 2, false>};
  for (auto f : k) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)((kIncL + 2) * kIncThreads * sizeof(float4)));
    if (e != cudaSuccess) return e;
  }
  void (*const kx[2])(SweepParams) = {k_sweep_xinc64<false>, k_sweep_xinc64<true>};
  for (auto f : kx) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)inc64_x_smem(kIncThreads, kIncThreads));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

long long inc64_blocks(int axis, const SweepParams& p, bool complex_field) {
  if (axis == 0) {
    const long long rows = (long long)p.inc_x * (complex_field ? 1 : 2);
    return ((long long)p.ny * p.nz + rows - 1) / rows;
  }
  const int nvec = complex_field ? p.nx : (p.nx + 1) / 2;
  return (long long)((nvec + p.inc_x - 1) / p.inc_x) * (axis == 1 ? p.nz : p.ny);
}

cudaError_t launch_inc64(int axis, const SweepParams& p, bool complex_field, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = st;
  cfg.gridDim = dim3((unsigned)inc64_blocks(axis, p, complex_field));
  cfg.blockDim = dim3((unsigned)p.inc_threads);
  cfg.dynamicSmemBytes = (size_t)(kIncL + 2) * cfg.blockDim.x * sizeof(float4);
  if (axis == 0) {
    cfg.dynamicSmemBytes = inc64_x_smem(cfg.blockDim.x, p.inc_x);
    // high word of the |v| below which |y| < 2^-56 (complex: each part), the folded factor
    // being at most 1.0625
    SweepParams q = p;
    const double most = 0x1p-56 / (1.13 * p.dt * std::fabs(p.g));
    double lim = std::sqrt(complex_field ? 0.5 * most : most);
    if (!(lim < 1e200)) lim = 1e200;   // g = 0
    uint64_t w;
    std::memcpy(&w, &lim, 8);
    q.inc_quiet = (int)(w >> 32);
    return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_xinc64<true>, q)
                         : cudaLaunchKernelEx(&cfg, k_sweep_xinc64<false>, q);
  }
  if (axis == 1 && p.plane_norm) return cudaLaunchKernelEx(&cfg, k_sweep_inc64<false, 1, true>, p);
  if (axis == 1)
    return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_inc64<true, 1, false>, p)
                         : cudaLaunchKernelEx(&cfg, k_sweep_inc64<false, 1, false>, p);
  return complex_field ? cudaLaunchKernelEx(&cfg, k_sweep_inc64<true, 2, false>, p)
                       : cudaLaunchKernelEx(&cfg, k_sweep_inc64<false, 2, true>, p);
}

}  // namespace gpk
