// gp_reduce.cu -- one-pass FP64 reductions and field conversions around the SSCN
// step: observables (energy, chemical potential, rms sizes), the norm of a fresh
// state, the initial Gaussian, host-layout import / export, and the integrated
// densities of Eq. 1 and its 3D analogues (paper, "Summary of revisions").
//
// Every reduction runs on a fixed launch shape (kReduceBlocks x kReduceThreads),
// sums in a fixed order (per thread, then a shuffle tree, then the blocks' partials
// in index order by the last block to finish), and is therefore deterministic.
#include <algorithm>

#include "gp_device.cuh"
#include "gp_split.cuh"

namespace gpk {

template <class R, bool CPLX> struct Load;
template <class R> struct Load<R, false> {
  static __device__ __forceinline__ double2 at(const void* psi, size_t idx, double s) {
    return make_double2((double)static_cast<const R*>(psi)[idx] * s, 0.0);
  }
};
template <class R> struct Load<R, true> {
  static __device__ __forceinline__ double2 at(const void* psi, size_t idx, double s) {
    const typename Cplx<R>::T v = static_cast<const typename Cplx<R>::T*>(psi)[idx];
    return make_double2((double)v.x * s, (double)v.y * s);
  }
};

__device__ __forceinline__ double dabs2(double2 v) { return fma(v.x, v.x, v.y * v.y); }
__device__ __forceinline__ double dabs2_diff(double2 a, double2 b) {
  const double x = a.x - b.x, y = a.y - b.y;
  return fma(x, x, y * y);
}

// Fixed-order block sum of NACC accumulators into partials[blockIdx.x * NACC + c];
// returns true in the last block to finish, after its fixed-order total over all
// blocks has been written to tot[0..NACC-1] (shared memory).  Every thread of every
// block must call it.
template <int NACC>
__device__ bool block_reduce_last(double (&acc)[NACC], double* partials, unsigned int* counter,
                                  double* tot) {
  __shared__ double warp_part[kReduceThreads / 32][NACC];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < NACC; ++c) {
    double v = acc[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) warp_part[warp][c] = v;
  }
  __syncthreads();
  if (threadIdx.x < NACC) {
    double v = 0.0;
    for (int w = 0; w < kReduceThreads / 32; ++w) v += warp_part[w][threadIdx.x];
    partials[(size_t)blockIdx.x * NACC + threadIdx.x] = v;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return false;
  __threadfence();
  // the blocks' partials of each accumulator: thread t takes blocks t, t + T, ...
  // (Neumaier), then a shuffle tree and the warps in order -- a fixed order, and
  // short FP64 dependency chains (one thread walking all blocks would take a chain
  // of four FP64 operations per block)
  const unsigned int nb = gridDim.x;
#pragma unroll
  for (int c = 0; c < NACC; ++c) {
    double s = 0.0, comp = 0.0;
    for (unsigned int b = threadIdx.x; b < nb; b += blockDim.x) {
      const double x = __ldcg(partials + (size_t)b * NACC + c);
      const double u = s + x;
      comp += (fabs(s) >= fabs(x)) ? (s - u) + x : (x - u) + s;
      s = u;
    }
    double v = s + comp;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) warp_part[warp][c] = v;
  }
  __syncthreads();
  if (threadIdx.x < NACC) {
    double v = 0.0;
    for (int w = 0; w < kReduceThreads / 32; ++w) v += warp_part[w][threadIdx.x];
    tot[threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

// ---------------------------------------------------------------- observables

template <class R, bool CPLX>
__global__ void __launch_bounds__(kReduceThreads) k_observables(const FieldParams p) {
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t P = (size_t)p.pitch, plane = P * ny;
  const double s = *p.scale;
  const double* Vx = p.tab;
  const double* Vy = Vx + nx;
  const double* Vz = Vy + ny;
  const double* X2 = Vz + nz;
  const double* Y2 = X2 + nx;
  const double* Z2 = Y2 + ny;
  double acc[kObsAcc];
#pragma unroll
  for (int c = 0; c < kObsAcc; ++c) acc[c] = 0.0;
  const long long nrows = (long long)ny * nz;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x) {
    const int j = (int)(r % ny), k = (int)(r / ny);
    const size_t base = (size_t)r * P;
    const double vyz = Vy[j] + Vz[k];
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
      const size_t idx = base + i;
      const double2 v = Load<R, CPLX>::at(p.psi, idx, s);
      const double d = dabs2(v);
      acc[0] += d;
      acc[1] += (Vx[i] + vyz) * d;
      acc[2] += d * d;
      const double2 z0 = make_double2(0.0, 0.0);
      const double2 wx = (i + 1 < nx) ? Load<R, CPLX>::at(p.psi, idx + 1, s) : z0;
      const double2 wy = (j + 1 < ny) ? Load<R, CPLX>::at(p.psi, idx + P, s) : z0;
      const double2 wz = (k + 1 < nz) ? Load<R, CPLX>::at(p.psi, idx + plane, s) : z0;
      acc[3] += dabs2_diff(wx, v) + (i == 0 ? d : 0.0);  // edge (i, i+1), ghost edge at i = 0
      acc[4] += dabs2_diff(wy, v) + (j == 0 ? d : 0.0);
      acc[5] += dabs2_diff(wz, v) + (k == 0 ? d : 0.0);
      acc[6] += X2[i] * d;
      acc[7] += Y2[j] * d;
      acc[8] += Z2[k] * d;
    }
  }
  __shared__ double tot[kObsAcc];
  if (!block_reduce_last<kObsAcc>(acc, p.partials, p.counter, tot)) return;
  if (threadIdx.x == 0) {
    const double dV = p.hx * p.hy * p.hz;
    const double norm = tot[0] * dV;
    const double epot = tot[1] * dV;
    const double eint = 0.5 * p.g * tot[2] * dV;
    const double ekin =
        0.5 * dV * (tot[3] / (p.hx * p.hx) + tot[4] / (p.hy * p.hy) +
                    (p.nz == 1 ? 0.0 : tot[5] / (p.hz * p.hz)));   // 2D: no z kinetic term
    const double x2 = tot[6] * dV / norm, y2 = tot[7] * dV / norm, z2 = tot[8] * dV / norm;
    double* o = p.out;
    o[0] = norm;
    o[1] = ekin + epot + 2.0 * eint;
    o[2] = ekin + epot + eint;
    o[3] = ekin;
    o[4] = epot;
    o[5] = eint;
    o[6] = sqrt(x2);
    o[7] = sqrt(y2);
    o[8] = sqrt(z2);
    o[9] = sqrt(x2 + y2 + z2);
  }
}

// ------------------------------------- observables by sums on the FP32 pipe

// The same sums with the arithmetic on the FP32 pipe (gp_split.cuh: FP64 operations and
// conversions run at 1/64 of FP32's rate here, and k_observables spends 32-45 of them per
// point: 590 us for 240 x 200 x 160 complex64 points, where reading the field takes 9 us).
// FP32 values are taken as they are, FP64 ones as three FP32 parts, all 53 bits: their
// differences are exact that way (from 48 bits the kinetic sum of a finely sampled field is off by
// 2^-48 over the relative difference of neighbours).  Squares are two-part; a sum of them has
// three parts, adds without error but for its third part's rounding, and moves to FP64 (in shared
// memory) every two dozen terms.  With two-part sums the low part was rounded at every
// addition, and because a sum of two squares is never 3 mod 4 in its last bits, ties went down
// more often than up: sums 2e-16..5e-16 too small, fourth powers 1e-15.  The weights
// are exact in x: (2i - nx + 1)^2 h^2 / 4 with the integer part in FP32; y and z weigh a row's
// sum in FP64; the potential energy follows from the three.  The pending factor is applied
// to the sums.  Fields whose largest value (times the factor) lies outside
// [2^-16, 2^24], where sums of weighted fourth powers could leave FP32's range, and small grids (fewer than
// 2^15 points, where k_observables takes no longer and there is less to average over) go
// to k_observables; out[10] receives the largest |component| and out[11] the factor for the
// host's check.
// Measured (240 x 200 x 160, the whole call): complex64 736 -> 187 us, FP32 real 124, FP64 real
// 451 -> 159, complex128 611 -> 250; bound by its FP32 instructions.  Error against extended
// precision as k_observables': at most 4 x 2^-53 relative, no lean to one side (two-part sums: 137
// us and up to 17 x 2^-53).
// A warp takes a row at a time, consecutive warps consecutive rows (y neighbours from L1),
// the next 32 columns' loads in flight.
constexpr int kObsTwoBlocks = 304;   // two resident blocks per SM

// A value pair: columns (2c, 2c + 1), or (re, im) of column c.
template <class R> struct PairValue;
template <> struct PairValue<float> {
  float2 v;
  __device__ __forceinline__ Two two() const { return two_scalar(v, f2(0.f)); }
  __device__ __forceinline__ PairValue next(const PairValue& n) const { return {f2(v.y, n.v.x)}; }   // one column on
  __device__ __forceinline__ Two minus(const PairValue& b) const {
    Two d;
    two_sum(v, mul2(b.v, f2(-1.f)), &d.h, &d.l);
    return d;
  }
};
template <> struct PairValue<double> {
  Three v;
  __device__ __forceinline__ Two two() const {
    const float2 h = add2(v.h, v.m);
    return two_scalar(h, add2(sub2(v.m, sub2(h, v.h)), v.l));
  }
  __device__ __forceinline__ PairValue next(const PairValue& n) const {
    PairValue r;
    r.v.h = f2(v.h.y, n.v.h.x);
    r.v.m = f2(v.m.y, n.v.m.x);
    r.v.l = f2(v.l.y, n.v.l.x);
    return r;
  }
  __device__ __forceinline__ Two minus(const PairValue& b) const {
    float2 s, e, f;
    two_sum(v.h, mul2(b.v.h, f2(-1.f)), &s, &e);
    Two d;
    two_sum(s, sub2(v.m, b.v.m), &d.h, &f);
    d.l = add2(f, add2(sub2(v.l, b.v.l), e));
    return d;
  }
};
template <class R, bool CPLX> struct PairLoad;
template <bool CPLX> struct PairLoad<float, CPLX> {
  using V = float2;
  static __device__ __forceinline__ V load(const void* row, int c, int nc) {   // zero from nc on
    return c < nc ? static_cast<const float2*>(row)[c] : f2(0.f);
  }
  static __device__ __forceinline__ PairValue<float> value(V v, int c, int nx, int*) {
    if (!CPLX && 2 * c + 1 >= nx) v.y = 0.f;
    return {v};
  }
};
template <bool CPLX> struct PairLoad<double, CPLX> {
  using V = double2;
  static __device__ __forceinline__ V load(const void* row, int c, int nc) {
    return c < nc ? static_cast<const double2*>(row)[c] : make_double2(0.0, 0.0);
  }
  static __device__ __forceinline__ PairValue<double> value(V v, int c, int nx, int* tmax) {
    if (!CPLX && 2 * c + 1 >= nx) v.y = 0.0;
    PairValue<double> r;
    r.v = split3(v.x, v.y, tmax, kSplitOff1);
    return r;
  }
};

// A sum of two-part numbers in three parts, two lanes.
struct SquareSum {
  float2 h = make_float2(0.f, 0.f), l = h, m = h;
  __device__ __forceinline__ void add(const Two& q) {
    float2 f, g, k, t;
    two_sum(h, q.h, &t, &f);
    h = t;
    two_sum(l, q.l, &t, &g);
    two_sum(t, f, &l, &k);
    m = add2(m, add2(g, k));
  }
  // lane x, or both lanes (NaN: infinities or NaN among the values)
  __device__ __forceinline__ double total(bool both) const {
    auto d = [](float x) { return to_double(x, 0.f, kSplitShift); };
    double s = (d(h.x) + d(l.x)) + d(m.x);
    if (both) s += (d(h.y) + d(l.y)) + d(m.y);
    return fabsf(h.x) + fabsf(h.y) <= 1e30f ? s : (double)__int_as_float(0x7fc00000);
  }
};

template <class R, bool CPLX>
__global__ void __launch_bounds__(kReduceThreads, 2) k_observables_two(const FieldParams p) {
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const int nc = CPLX ? nx : (nx + 1) / 2;   // column pairs
  const size_t rowb = (size_t)p.pitch * sizeof(R) * (CPLX ? 2 : 1);
  const unsigned char* field = static_cast<const unsigned char*>(p.psi);
  const int lane = threadIdx.x & 31;
  const int nrows = ny * nz;
  using L = PairLoad<R, CPLX>;
  constexpr bool LOW = sizeof(R) == 8;   // values have low parts
  // v^2 = q.h + q.l + what `low` receives, which all sums take in FP64 at the end (rounded away,
  // the square of the low part, never negative, would bias them).  full: nothing rounds but low
  // itself; else q.l does, which is exact for a v without a low part.
  auto square = [](const Two& v, float2* low, bool full) {
    Two q;
    const float2 v2 = add2(v.h, v.h);
    q.h = mul2(v.h, v.h);
    const float2 res = fma2(v.h, v.h, mul2(q.h, f2(-1.f)));
    *low = fma2(v.l, v.l, *low);
    if (full) {
      const float2 p = mul2(v2, v.l), pe = fma2(v2, v.l, mul2(p, f2(-1.f)));
      float2 e;
      two_sum(res, p, &q.l, &e);
      *low = add2(*low, add2(e, pe));
    } else {
      q.l = fma2(v2, v.l, res);
    }
    return q;
  };
  auto edge = [&](const PairValue<R>& a, const PairValue<R>& b, float2* low) { return square(a.minus(b), low, LOW); };
  float2 lSX = f2(0.f), lS4 = f2(0.f), lX = f2(0.f), lY = f2(0.f), lZ = f2(0.f);
  float lS = 0.f, lSY = 0.f, lSZ = 0.f;
  SquareSum SX, S4, KX, KY, KZ;
  float vmax = 0.f;
  int tmax = 0;
  __shared__ double sums[8][kReduceThreads];   // S, SX, SY, SZ, S4, KX, KY, KZ
  auto drain = [&](int i, SquareSum& t, bool both) {
    sums[i][threadIdx.x] += t.total(both);
    t = SquareSum();
  };
#pragma unroll
  for (int i = 0; i < 8; ++i) sums[i][threadIdx.x] = 0.0;
  const double* Y2 = p.tab + 2 * nx + ny + nz;   // y^2, then z^2
  const int often = max(1, 24 / ((nc + 31) / 32));   // rows between two drains
  int due = often;
  const int step = gridDim.x * (kReduceThreads / 32);
  for (int r = blockIdx.x * (kReduceThreads / 32) + (threadIdx.x >> 5); r < nrows; r += step) {
    const int k = r / ny, j = r - k * ny;
    const unsigned char* row = field + (size_t)r * rowb;
    SquareSum SR;
    float2 lSR = f2(0.f);
    auto fetch = [&](int c, typename L::V (&b)[4]) {   // a point and its three neighbours
      b[0] = L::load(row, c, nc);
      b[1] = L::load(row, c + 1, nc);
      b[2] = L::load(row + rowb, c, j + 1 < ny ? nc : 0);
      b[3] = L::load(row + rowb * ny, c, k + 1 < nz ? nc : 0);
    };
    typename L::V cur[4], ahead[4];
    fetch(lane, cur);
    for (int c = lane; c < nc; c += 32) {
      fetch(c + 32, ahead);
      const PairValue<R> at = L::value(cur[0], c, nx, &tmax), nxt = L::value(cur[1], c + 1, nx, &tmax),
                         wy = L::value(cur[2], c, nx, &tmax), wz = L::value(cur[3], c, nx, &tmax);
      const Two v = at.two();
#pragma unroll
      for (int q = 0; q < 4; ++q) cur[q] = ahead[q];
      const PairValue<R> wx = CPLX ? nxt : at.next(nxt);
      vmax = fmaxf(vmax, fmaxf(fabsf(v.h.x), fabsf(v.h.y)));
      float2 ll = f2(0.f);
      const Two q = square(v, &ll, LOW);
      SR.add(q);
      lSR = add2(lSR, ll);
      // (2i - nx + 1)^2 below 2^22: exact in FP32
      const float w0 = (float)(2 * (CPLX ? c : 2 * c) - nx + 1), w1 = CPLX ? w0 : w0 + 2.f;
      const float2 wc = f2(w0 * w0, w1 * w1);
      Two qx;
      qx.h = mul2(wc, q.h);
      qx.l = fma2(wc, q.l, fma2(wc, q.h, mul2(qx.h, f2(-1.f))));
      SX.add(qx);
      Two d = q;
      float2 rest = f2(0.f);   // of d
      if (CPLX) {
        const Two o = two_swap(q);
        float2 e, f, l, g;
        two_sum(q.h, o.h, &d.h, &e);
        two_sum(q.l, o.l, &l, &f);
        two_sum(l, e, &d.l, &g);
        rest = add2(f, g);
      }
      S4.add(square(d, &lS4, true));
      if (CPLX) lS4 = fma2(add2(d.h, d.h), rest, lS4);
      if (LOW) {   // the squares of the values' low parts in the weighted and fourth-power sums
        lSX = fma2(wc, ll, lSX);
        lS4 = fma2(add2(d.h, d.h), CPLX ? add2(ll, f2(ll.y, ll.x)) : ll, lS4);
      }
      KX.add(edge(wx, at, &lX));
      KY.add(edge(wy, at, &lY));
      KZ.add(edge(wz, at, &lZ));
      if (c == 0) {   // the ghost edge at i = 0
        const float2 m = f2(1.f, CPLX ? 1.f : 0.f);
        KX.add(two_scalar(mul2(q.h, m), mul2(q.l, m)));
        if (LOW) lX = fma2(m, ll, lX);
      }
      if (j == 0) {
        KY.add(q);
        if (LOW) lY = add2(lY, ll);
      }
      if (k == 0) {
        KZ.add(q);
        if (LOW) lZ = add2(lZ, ll);
      }
    }
    {
      const double sr = SR.total(true), y2 = Y2[j], z2 = Y2[ny + k];
      sums[0][threadIdx.x] += sr;
      sums[2][threadIdx.x] = fma(y2, sr, sums[2][threadIdx.x]);
      sums[3][threadIdx.x] = fma(z2, sr, sums[3][threadIdx.x]);
      if (LOW) {
        const float lr = lSR.x + lSR.y;
        lS += lr;
        lSY = fmaf((float)y2, lr, lSY);
        lSZ = fmaf((float)z2, lr, lSZ);
      }
    }
    if (--due > 0 && r + step < nrows) continue;
    due = often;
    drain(1, SX, true);
    drain(4, S4, !CPLX);
    drain(5, KX, true);
    drain(6, KY, true);
    drain(7, KZ, true);
  }
  if (LOW && tmax >= kSplitTooBig) vmax = __int_as_float(0x7f800000);   // out of FP32's range, for the host's check
  double acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = sums[i][threadIdx.x];
  auto both = [](float2 l) { return (double)l.x + (double)l.y; };
  acc[4] += CPLX ? (double)lS4.x : both(lS4);
  acc[5] += both(lX);
  acc[6] += both(lY);
  acc[7] += both(lZ);
  if (LOW) {
    acc[0] += (double)lS;
    acc[1] += both(lSX);
    acc[2] += (double)lSY;
    acc[3] += (double)lSZ;
  }
  const unsigned int wmax = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
  __shared__ unsigned int bmax;
  if (threadIdx.x == 0) bmax = 0u;
  __syncthreads();
  if (lane == 0) atomicMax(&bmax, wmax);
  __syncthreads();
  double* maxima = p.partials + (size_t)gridDim.x * 8;
  if (threadIdx.x == 0) maxima[blockIdx.x] = (double)__uint_as_float(bmax);
  __shared__ double tot[8];
  if (!block_reduce_last<8>(acc, p.partials, p.counter, tot)) return;
  unsigned int m = 0u;
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x)
    m = max(m, __float_as_uint((float)__ldcg(maxima + b)));
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) atomicMax(&bmax, m);
  __syncthreads();
  if (threadIdx.x == 0) {
    // (products of constants in an order, and with a remainder, that leave no rounding error that
    // would be the same for every field)
    const double s = *p.scale, s2 = s * s;
    const double area = p.hx * p.hy, dV = area * p.hz;
    const double dVl = fma(area, p.hz, -dV) + fma(p.hx, p.hy, -area) * p.hz;
    auto integral = [&](double x) { return fma(x, dVl, x * dV); };
    const double sum = tot[0] * s2, norm = integral(sum);
    const double sx = tot[1] * s2 * 0.25 * p.hx * p.hx, sy = tot[2] * s2;
    const double sz = nz == 1 ? 0.0 : tot[3] * s2;
    const double epot = integral(sx * p.v2[0] + sy * p.v2[1] + sz * p.v2[2]);
    const double eint = integral(tot[4] * s2 * s2 * (0.5 * p.g));
    const double ekin = integral(0.5 * s2 * (tot[5] / p.hx / p.hx + tot[6] / p.hy / p.hy +
                                             (nz == 1 ? 0.0 : tot[7] / p.hz / p.hz)));
    const double x2 = sx / sum, y2 = sy / sum, z2 = sz / sum;
    double* o = p.out;
    o[0] = norm;
    o[1] = ekin + epot + 2.0 * eint;
    o[2] = ekin + epot + eint;
    o[3] = ekin;
    o[4] = epot;
    o[5] = eint;
    o[6] = sqrt(x2);
    o[7] = sqrt(y2);
    o[8] = sqrt(z2);
    o[9] = sqrt(x2 + y2 + z2);
    o[10] = (double)__uint_as_float(bmax);
    o[11] = s;
  }
}

// ------------------------------------------------------ norm of a fresh field

// Real field only (used after the Gaussian initialisation): *out = 1/sqrt(norm).
template <class R>
__global__ void __launch_bounds__(kReduceThreads) k_norm_to_scale(const FieldParams p) {
  const int nx = p.nx;
  const size_t P = (size_t)p.pitch;
  double acc[1] = {0.0};
  const long long nrows = (long long)p.ny * p.nz;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x)
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
      const double v = (double)static_cast<const R*>(p.psi)[(size_t)r * P + i];
      acc[0] += v * v;
    }
  __shared__ double tot[1];
  if (!block_reduce_last<1>(acc, p.partials, p.counter, tot)) return;
  if (threadIdx.x == 0) {
    const double norm = tot[0] * p.hx * p.hy * p.hz;
    if (!(norm > 0.0) || !isfinite(norm)) atomicOr(p.status, kStatusNonFinite);
    *p.out = 1.0 / sqrt(norm);
  }
}

// ------------------------------------------- standalone pointwise substep

// psi <- P(psi) with the half step's separable trap factors and dtg = (dt / 2) g, the
// same arithmetic as the sweeps' fused substep (Field policies); with NORM the norm
// of the result becomes the pending factor.
template <class R, bool CPLX, bool NORM>
__global__ void __launch_bounds__(kReduceThreads) k_half_pointwise(const FieldParams p, const void* fx,
                                                                   const void* fyz, double dtg_d,
                                                                   int apply_scale) {
  using F = Field<R, CPLX>;
  using E = typename F::E;
  const int nx = p.nx;
  const size_t P = (size_t)p.pitch;
  const R s = apply_scale ? (R)(*p.scale) : R(1);
  const R dtg = (R)dtg_d;
  const E* fxt = static_cast<const E*>(fx);
  const E* fyt = static_cast<const E*>(fyz);
  E* psi = static_cast<E*>(p.psi);
  double acc[1] = {0.0};
  // chunks of CH rows, the chunk's CH * nx points spread over the block, U per thread
  // in flight: all U loads are issued before any store
  constexpr int U = 4, CH = 8;
  const long long nrows = (long long)p.ny * p.nz;
  const int per = CH * nx;   // points per chunk
  for (long long r0 = (long long)blockIdx.x * CH; r0 < nrows; r0 += (long long)gridDim.x * CH) {
    const int rows = (int)min((long long)CH, nrows - r0);
    const int cnt = rows * nx;
    for (int base = threadIdx.x; base < cnt; base += blockDim.x * U) {
      E v[U], f[U];
      size_t at[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = base + u * blockDim.x;
        const int q = e < cnt ? e : 0;
        const int rl = q / nx, i = q - rl * nx;
        at[u] = (size_t)(r0 + rl) * P + i;
        v[u] = psi[at[u]];
        f[u] = F::mul(fxt[i], fyt[r0 + rl]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (base + u * (int)blockDim.x >= cnt) continue;
        const E w = F::scaled(v[u], s);
        const R y = dtg * F::abs2(w);
        const E out = fabs(y) <= R(0.0625) ? F::nonlinear_small(w, f[u], y) : F::nonlinear_full(w, f[u], y);
        psi[at[u]] = out;
        if (NORM) acc[0] += (double)F::abs2(out);
      }
    }
    (void)per;
  }
  if (NORM) {
    __shared__ double tot[1];
    if (!block_reduce_last<1>(acc, p.partials, p.counter, tot)) return;
    if (threadIdx.x == 0) {
      const double norm = tot[0] * p.hx * p.hy * p.hz;
      if (!(norm > 0.0) || !isfinite(norm)) atomicOr(p.status, kStatusNonFinite);
      *p.out = 1.0 / sqrt(norm);
    }
  }
}

// FP32 field (words = 1 real, 2 complex floats per element) times the pending factor,
// packed into rows of nx elements in dst (not the field): 16-byte vectors when the
// rows are contiguous and a multiple of four floats, else one float per thread.
__global__ void k_export_f32(const FieldParams p, int words, float* __restrict__ dst) {
  const float s = (float)(*p.scale);
  const float* src = static_cast<const float*>(p.psi);
  const size_t rw = (size_t)p.nx * words, pw = (size_t)p.pitch * words;
  const size_t nrows = (size_t)p.ny * p.nz;
  if (rw == pw && rw % 4 == 0) {
    const size_t n4 = nrows * rw / 4;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(dst);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
      float4 v = s4[i];
      v.x *= s;
      v.y *= s;
      v.z *= s;
      v.w *= s;
      d4[i] = v;
    }
    return;
  }
  for (size_t r = blockIdx.x; r < nrows; r += gridDim.x)
    for (size_t i = threadIdx.x; i < rw; i += blockDim.x) dst[r * rw + i] = src[r * pw + i] * s;
}

// The reverse: packed rows of nx elements in src into the FP32 field (pad columns
// zero), as they are (no factor).
__global__ void k_import_f32(const FieldParams p, int words, const float* __restrict__ src) {
  float* dst = static_cast<float*>(p.psi);
  const size_t rw = (size_t)p.nx * words, pw = (size_t)p.pitch * words;
  const size_t nrows = (size_t)p.ny * p.nz;
  if (rw == pw && rw % 4 == 0) {
    const size_t n4 = nrows * rw / 4;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(dst);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x)
      d4[i] = s4[i];
    return;
  }
  for (size_t r = blockIdx.x; r < nrows; r += gridDim.x)
    for (size_t i = threadIdx.x; i < pw; i += blockDim.x) dst[r * pw + i] = i < rw ? src[r * rw + i] : 0.f;
}

// ------------------------------------------------------------ initial Gaussian

// The largest of the values a block's threads wrote (vmax: their high words) into the field's
// word; every thread of the block calls it.
__device__ __forceinline__ void field_max(int vmax, int* amax) {
  if (!amax) return;
  vmax = __reduce_max_sync(0xffffffffu, vmax);
  if ((threadIdx.x & 31) == 0) atomicMax(amax + kAmaxNow, vmax);
}

template <class R>
__global__ void k_init_gaussian(const FieldParams p, double wx, double wy, double wz) {
  const int nx = p.nx, ny = p.ny, P = p.pitch;
  const long long nrows = (long long)ny * p.nz;
  int vmax = 0;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x) {
    const int j = (int)(r % ny), k = (int)(r / ny);
    const double y = (j - 0.5 * (ny - 1)) * p.hy;
    const double z = (k - 0.5 * (p.nz - 1)) * p.hz;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      double v = 0.0;
      if (i < nx) {
        const double x = (i - 0.5 * (nx - 1)) * p.hx;
        v = exp(-0.5 * (wx * x * x + wy * y * y + wz * z * z));
      }
      static_cast<R*>(p.psi)[(size_t)r * P + i] = (R)v;
      vmax = max(vmax, high_word(v));
    }
  }
  field_max(vmax, p.amax);
}

// ------------------------------------------------- host layout <-> device field

template <class R, bool CPLX>
__global__ void k_import(const FieldParams p, const double* __restrict__ src) {
  using C = typename Cplx<R>::T;
  const int nx = p.nx, P = p.pitch;
  const long long nrows = (long long)p.ny * p.nz;
  int vmax = 0;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x)
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      const size_t d = (size_t)r * P + i, q = (size_t)r * nx + i;
      const double re = i >= nx ? 0.0 : CPLX ? src[2 * q] : src[q];
      const double im = CPLX && i < nx ? src[2 * q + 1] : 0.0;
      vmax = max(vmax, max(high_word(re), high_word(im)));
      if (CPLX) {
        static_cast<C*>(p.psi)[d] = C{(R)re, (R)im};
      } else {
        static_cast<R*>(p.psi)[d] = (R)re;
      }
    }
  field_max(vmax, p.amax);
}

template <class R, bool CPLX>
__global__ void k_export(const FieldParams p, double* __restrict__ dst, int as_complex) {
  const int nx = p.nx;
  const size_t P = (size_t)p.pitch;
  const double s = *p.scale;
  const long long nrows = (long long)p.ny * p.nz;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x)
    for (int i = threadIdx.x; i < nx; i += blockDim.x) {
      const double2 v = Load<R, CPLX>::at(p.psi, (size_t)r * P + i, s);
      const size_t q = (size_t)r * nx + i;
      if (as_complex) {
        dst[2 * q] = v.x;
        dst[2 * q + 1] = v.y;
      } else {
        dst[q] = v.x;
      }
    }
}

// ------------------------------------------------------- integrated densities

// Sums of squares of FP32 values below 4 in modulus, on the FP32 pipe and two at a time: the
// square's two exact parts are cut at fixed binary places (adding and subtracting a constant
// rounds to its grid: the error-free vector transformation of Rump, Ogita and Oishi's AccSum, SIAM
// J. Sci. Comput. 31, 2008), so that sums of sixteen of the upper two cuts are exact, of 2^-16 and
// 2^-36, and only the third, below 2^-32, rounds: 2^-56 of the largest square.
struct Squares {
  float2 h, m, l;
};
__device__ __forceinline__ float2 on_grid(float2 x, float c) { return add2(add2(x, f2(c)), f2(-c)); }
__device__ __forceinline__ void add_square(Squares& t, float2 a) {
  constexpr float kGrid1 = 192.f, kGrid2 = 0x1.8p-13f;
  const float2 qh = mul2(a, a), ql = fma2(a, a, mul2(qh, f2(-1.f)));
  const float2 h = on_grid(qh, kGrid1), rest = sub2(qh, h);
  const float2 m = on_grid(rest, kGrid2), n = on_grid(ql, kGrid2);
  t.h = add2(t.h, h);
  t.m = add2(t.m, add2(m, n));
  t.l = add2(t.l, add2(sub2(rest, m), sub2(ql, n)));
}
__device__ __forceinline__ void add_lanes(Squares& t) {   // both lanes: their sum
  t.h = add2(t.h, f2(t.h.y, t.h.x));
  t.m = add2(t.m, f2(t.m.y, t.m.x));
  t.l = add2(t.l, f2(t.l.y, t.l.x));
}
// the exponent field of the power of two that values up to m are divided by: the largest is 1 to
// 4 then (all subnormal: less, but their squares are multiples of 2^-44, and every sum is exact)
__device__ __forceinline__ int square_exponent(float m) { return min((int)(__float_as_uint(m) >> 23), 253); }
__device__ __forceinline__ float square_scale(int ex) { return __uint_as_float((unsigned int)(254 - ex) << 23); }
__device__ __forceinline__ bool finite_sums(float2 h) { return fabsf(h.x) + fabsf(h.y) <= 1e30f; }
// acc plus the sum of lane x (y) of values that were divided by 2^(ex - 127)
__device__ __forceinline__ double add_sum(double acc, float h, float m, float l, int ex) {
  const int k = kSplitShift + 2 * (ex - 127);
  const Two n = two_norm(two_scalar(f2(h), f2(m)));
  return (acc + to_double(n.h.x, n.l.x, k)) + to_double(l, 0.f, k);
}

// |psi|^2 summed along one direction, kDensSum terms per thread: chunk ch of the nsum
// rows `step` elements apart, for every column and each of the rows_out starting rows
// `out_step` apart; part[(ch rows_out + o) nx + i].  One 16-byte vector per thread and
// row.  FP64 work is what the sums must not wait for (see k_observables_two): FP32 values are
// squared and added eight at a time as Squares, then in FP64; FP64 values cost one or two
// FP64 operations each.  The factor is applied by the final sum.  Error against extended
// precision as of FP64 sums throughout, 2e-16 rms (in two parts, eight terms at a time, 0.6e-15..
// 1.7e-15).  Measured (240 x 200 x 160 complex64, the whole call): 52-54 us per density (two parts
// 45-55, FP64 sums 202-239).
constexpr int kDensSum = 32;
template <class R, bool CPLX>
__global__ void __launch_bounds__(128) k_density_partial(const FieldParams p, int rows_out, size_t out_step,
                                                         int nsum, size_t step, double* __restrict__ part) {
  constexpr int W = 16 / (int)sizeof(R) / (CPLX ? 2 : 1);   // columns per vector
  const int nx = p.nx, nvec = (nx + W - 1) / W;
  const unsigned int t = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned int xv = t % (unsigned int)nvec, rest = t / (unsigned int)nvec;
  const int o = (int)(rest % (unsigned int)rows_out), ch = (int)(rest / (unsigned int)rows_out);
  const int r0 = ch * kDensSum, r1 = min(nsum, r0 + kDensSum);
  if (r0 >= nsum) return;
  constexpr int EB = (int)sizeof(R) * (CPLX ? 2 : 1);
  const float4* src = reinterpret_cast<const float4*>(static_cast<const unsigned char*>(p.psi) +
                                                      ((size_t)o * out_step + (size_t)xv * W) * EB);
  const size_t sv = step * EB / 16;
  double acc[W];
#pragma unroll
  for (int e = 0; e < W; ++e) acc[e] = 0.0;
  for (int r = r0; r < r1; r += 8) {
    float4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = r + q < r1 ? src[(size_t)(r + q) * sv] : make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (sizeof(R) == 8) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double2 d = *reinterpret_cast<const double2*>(&v[q]);
        if (CPLX) {
          acc[0] = fma(d.x, d.x, fma(d.y, d.y, acc[0]));
        } else {
          acc[0] = fma(d.x, d.x, acc[0]);
          acc[W - 1] = fma(d.y, d.y, acc[W - 1]);
        }
      }
    } else {
      // values are scaled by a power of two that takes the column's largest of the eight to 1..2,
      // which keeps the squares in FP32's range (columns apart: one can lie far below another)
      float m[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        m[0] = fmaxf(m[0], fabsf(v[q].x));
        m[1] = fmaxf(m[1], fabsf(v[q].y));
        m[2] = fmaxf(m[2], fabsf(v[q].z));
        m[3] = fmaxf(m[3], fabsf(v[q].w));
      }
      if (CPLX) {
        m[0] = m[1] = fmaxf(m[0], m[1]);
        m[2] = m[3] = fmaxf(m[2], m[3]);
      }
      int ex[4];
      float sc[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ex[i] = square_exponent(m[i]);
        sc[i] = square_scale(ex[i]);
      }
      Squares s0{f2(0.f), f2(0.f), f2(0.f)}, s1 = s0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        add_square(s0, mul2(f2(v[q].x, v[q].y), f2(sc[0], sc[1])));
        add_square(s1, mul2(f2(v[q].z, v[q].w), f2(sc[2], sc[3])));
      }
      if (CPLX) {
        add_lanes(s0);
        add_lanes(s1);
      }
      if (finite_sums(s0.h) && finite_sums(s1.h)) {
        acc[0] = add_sum(acc[0], s0.h.x, s0.m.x, s0.l.x, ex[0]);
        if (CPLX) {
          acc[1 % W] = add_sum(acc[1 % W], s1.h.x, s1.m.x, s1.l.x, ex[2]);
        } else {
          acc[1 % W] = add_sum(acc[1 % W], s0.h.y, s0.m.y, s0.l.y, ex[1]);
          acc[2 % W] = add_sum(acc[2 % W], s1.h.x, s1.m.x, s1.l.x, ex[2]);
          acc[3 % W] = add_sum(acc[3 % W], s1.h.y, s1.m.y, s1.l.y, ex[3]);
        }
      } else {   // infinities or NaN among the values
        for (int q = 0; q < 8; ++q) {
          const float e[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
          for (int i = 0; i < 4; ++i) acc[CPLX ? i / 2 % W : i % W] += (double)e[i] * (double)e[i];
        }
      }
    }
  }
  double* dst = part + ((size_t)ch * rows_out + o) * nx + (size_t)xv * W;
#pragma unroll
  for (int e = 0; e < W; ++e)
    if ((int)xv * W + e < nx) dst[e] = acc[e];
}

// out[q] = w scale^2 sum over ch of part[ch total + q], q < total: blockDim.x outputs per
// block, each of its rows of threads (a power of two) on every blockDim.y-th chunk, then added
// in a tree (in order, 64 of them made the error of 1D densities 3e-16 instead of 1e-16).
// (Few outputs of many chunks: 8 x 64 threads, so that the FP64 additions spread over
// more SMs; 240 sums of 1000 chunks took 22 us on 8 blocks of 32 outputs.)
__global__ void __launch_bounds__(512) k_density_combine(const double* __restrict__ part, int nch,
                                                         long long total, double w, const double* scale,
                                                         double* __restrict__ out) {
  __shared__ double sm[64 * 9];
  const int bx = blockDim.x, by = blockDim.y;
  const long long q = (long long)blockIdx.x * bx + threadIdx.x;
  double acc = 0.0;
  if (q < total)
#pragma unroll 4
    for (int c = threadIdx.y; c < nch; c += by) acc += part[(size_t)c * total + q];
  double* mine = sm + threadIdx.y * (bx + 1) + threadIdx.x;
  *mine = acc;
  for (int half = by / 2; half > 0; half /= 2) {
    __syncthreads();
    if ((int)threadIdx.y < half) *mine += mine[half * (bx + 1)];
  }
  if (threadIdx.y == 0 && q < total) {
    const double s = scale ? *scale : 1.0;
    out[q] = *mine * (w * s * s);
  }
}

// out[r] = w sum_i |psi|^2 of row r = k ny + j, eight rows per warp: the lanes' sums of the
// eight are added by a butterfly that halves the rows a lane carries at every exchange
// (nine FP64 additions for eight rows; forty with a tree per row made FP64 the bound).
template <class R, bool CPLX>
__global__ void __launch_bounds__(256) k_density_sum_rows(const FieldParams p, double w, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nrows = p.ny * p.nz;
  const int r0 = 8 * warp;
  if (r0 >= nrows) return;
  const double s = *p.scale;
  const int nc = CPLX ? p.nx : (p.nx + 1) / 2;   // column pairs
  double sum[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    double acc = 0.0;
    const R* base = static_cast<const R*>(p.psi) + (size_t)(r0 + t) * p.pitch * (CPLX ? 2 : 1);
    const int n = r0 + t < nrows ? nc : 0;
    if constexpr (sizeof(R) == 8) {
      const double2* row = reinterpret_cast<const double2*>(base);
      for (int c = lane; c < n; c += 32) {
        double2 v = row[c];
        if (!CPLX && 2 * c + 1 >= p.nx) v.y = 0.0;
        acc = fma(v.x, v.x, fma(v.y, v.y, acc));
      }
    } else {
      const float2* row = reinterpret_cast<const float2*>(base);
      for (int c0 = lane; c0 < n; c0 += 32 * 8) {   // eight pairs, as in k_density_partial
        float2 v[8];
        float m = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int c = c0 + 32 * q;
          v[q] = c < n ? row[c] : f2(0.f);
          if (!CPLX && 2 * c + 1 >= p.nx) v[q].y = 0.f;
          m = fmaxf(m, fmaxf(fabsf(v[q].x), fabsf(v[q].y)));
        }
        const int ex = square_exponent(m);
        const float2 sc = f2(square_scale(ex));
        Squares s0{f2(0.f), f2(0.f), f2(0.f)};
#pragma unroll
        for (int q = 0; q < 8; ++q) add_square(s0, mul2(v[q], sc));
        add_lanes(s0);
        if (finite_sums(s0.h)) {
          acc = add_sum(acc, s0.h.x, s0.m.x, s0.l.x, ex);
        } else {   // infinities or NaN among the values
          for (int q = 0; q < 8; ++q)
            acc = fma((double)v[q].x, (double)v[q].x, fma((double)v[q].y, (double)v[q].y, acc));
        }
      }
    }
    sum[t] = acc;
  }
  // lane bits 4, 3, 2 choose the row that a lane ends up with, bits 1 and 0 the quarter
#pragma unroll
  for (int half = 4, bit = 16; half >= 1; half >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (t >= half) break;
      const double keep = up ? sum[t + half] : sum[t], give = up ? sum[t] : sum[t + half];
      sum[t] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
    }
  }
  double v = sum[0];
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  const int r = r0 + (lane >> 2);
  if ((lane & 3) == 0 && r < nrows) out[r] = v * (w * s * s);
}

// out[r] = w * sum_c in[r*cols + c], one warp per row
__global__ void k_rows_sum(const double* __restrict__ in, int rows, int cols, double w,
                           double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= rows) return;
  double acc = 0.0;
  for (int c = lane; c < cols; c += 32) acc += in[(size_t)warp * cols + c];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) out[warp] = acc * w;
}

// ---------------------------------------------------------------- launchers

static unsigned int grid_for_rows(const FieldParams& p) {
  const long long nrows = (long long)p.ny * p.nz;
  return (unsigned int)(nrows < 4096 ? nrows : 4096);
}

bool observables_two(const FieldParams& p) {
  return (long long)p.nx * p.ny * p.nz >= (1LL << 15);
}

template <class R>
cudaError_t launch_observables(const FieldParams& p, bool complex_field, bool two, cudaStream_t st) {
  if (two) {
    if (complex_field)
      k_observables_two<R, true><<<kObsTwoBlocks, kReduceThreads, 0, st>>>(p);
    else
      k_observables_two<R, false><<<kObsTwoBlocks, kReduceThreads, 0, st>>>(p);
    return cudaGetLastError();
  }
  if (complex_field)
    k_observables<R, true><<<kReduceBlocks, kReduceThreads, 0, st>>>(p);
  else
    k_observables<R, false><<<kReduceBlocks, kReduceThreads, 0, st>>>(p);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_resolve_scale(double* scale, int* state, const double* partials,
                                                      int nb, double dV, int* status) {
  if (*state == 0) return;   // uniform: every thread reads the same word
  const double f = deferred_scale(partials, nb, dV, status, true);
  if (threadIdx.x == 0) {
    *scale = f;
    *state = 0;
  }
}

cudaError_t launch_resolve_scale(double* scale, int* state, const double* partials, int nb,
                                 double dV, int* status, cudaStream_t st) {
  k_resolve_scale<<<1, 256, 0, st>>>(scale, state, partials, nb, dV, status);
  return cudaGetLastError();
}

template <class R> cudaError_t launch_norm_to_scale(const FieldParams& p, cudaStream_t st) {
  k_norm_to_scale<R><<<kReduceBlocks, kReduceThreads, 0, st>>>(p);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_half_pointwise(const FieldParams& p, bool complex_field, const void* fx,
                                  const void* fyz, double dtg, bool apply_scale, bool norm,
                                  cudaStream_t st) {
  const int as = apply_scale ? 1 : 0;
  if (complex_field) {
    if (norm) k_half_pointwise<R, true, true><<<kReduceBlocks, kReduceThreads, 0, st>>>(p, fx, fyz, dtg, as);
    else k_half_pointwise<R, true, false><<<kReduceBlocks, kReduceThreads, 0, st>>>(p, fx, fyz, dtg, as);
  } else {
    if (norm) k_half_pointwise<R, false, true><<<kReduceBlocks, kReduceThreads, 0, st>>>(p, fx, fyz, dtg, as);
    else k_half_pointwise<R, false, false><<<kReduceBlocks, kReduceThreads, 0, st>>>(p, fx, fyz, dtg, as);
  }
  return cudaGetLastError();
}


cudaError_t launch_export_f32(const FieldParams& p, bool complex_field, float* dst, cudaStream_t st) {
  k_export_f32<<<grid_for_rows(p), 256, 0, st>>>(p, complex_field ? 2 : 1, dst);
  return cudaGetLastError();
}

cudaError_t launch_import_f32(const FieldParams& p, bool complex_field, const float* src, cudaStream_t st) {
  k_import_f32<<<grid_for_rows(p), 256, 0, st>>>(p, complex_field ? 2 : 1, src);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_init_gaussian(const FieldParams& p, double wx, double wy, double wz,
                                 cudaStream_t st) {
  k_init_gaussian<R><<<grid_for_rows(p), 256, 0, st>>>(p, wx, wy, wz);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_import(const FieldParams& p, const double* src, bool complex_field,
                          cudaStream_t st) {
  if (complex_field)
    k_import<R, true><<<grid_for_rows(p), 256, 0, st>>>(p, src);
  else
    k_import<R, false><<<grid_for_rows(p), 256, 0, st>>>(p, src);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_export(const FieldParams& p, double* dst, bool complex_field, bool as_complex,
                          cudaStream_t st) {
  if (complex_field)
    k_export<R, true><<<grid_for_rows(p), 256, 0, st>>>(p, dst, 1);
  else
    k_export<R, false><<<grid_for_rows(p), 256, 0, st>>>(p, dst, as_complex ? 1 : 0);
  return cudaGetLastError();
}

static void launch_combine(const double* part, int nch, long long total, double w, const double* scale,
                           double* out, cudaStream_t st) {
  const dim3 block = nch <= 16 ? dim3(32, 8) : dim3(8, 64);
  k_density_combine<<<(unsigned int)((total + block.x - 1) / block.x), block, 0, st>>>(part, nch, total, w, scale, out);
}

// |psi|^2 over the lines of a direction into out (see launch_density): the partial sums go
// behind it
template <class R>
static cudaError_t density_lines(const FieldParams& p, bool complex_field, int rows_out, size_t out_step,
                                 int nsum, size_t step, double w, double* out, cudaStream_t st) {
  const int W = 16 / (int)sizeof(R) / (complex_field ? 2 : 1);
  const int nvec = (p.nx + W - 1) / W, nch = (nsum + kDensSum - 1) / kDensSum;
  const long long total = (long long)rows_out * p.nx;
  double* part = out + total;
  const unsigned int blocks = (unsigned int)(((long long)nvec * rows_out * nch + 127) / 128);
  if (complex_field)
    k_density_partial<R, true><<<blocks, 128, 0, st>>>(p, rows_out, out_step, nsum, step, part);
  else
    k_density_partial<R, false><<<blocks, 128, 0, st>>>(p, rows_out, out_step, nsum, step, part);
  launch_combine(part, nch, total, w, p.scale, out, st);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_density(const FieldParams& p, bool complex_field, int which, double* out, cudaStream_t st) {
  const size_t P = (size_t)p.pitch, plane = P * (size_t)p.ny;
  switch (which) {
    case 0: return density_lines<R>(p, complex_field, p.ny, P, p.nz, plane, p.hz, out, st);
    case 1: return density_lines<R>(p, complex_field, p.nz, plane, p.ny, P, p.hy, out, st);
    case 3: return density_lines<R>(p, complex_field, 1, 0, p.ny * p.nz, P, p.hy * p.hz, out, st);
    default: break;
  }
  const double w = which == 2 ? p.hx : which == 4 ? p.hx * p.hz : p.hx * p.hy;
  const long long rows = (long long)p.ny * p.nz;
  double* sums = which == 2 ? out : out + std::max(p.ny, p.nz);   // the rows' sums
  const unsigned int blocks = (unsigned int)((rows + 63) / 64);   // eight warps of eight rows
  if (complex_field)
    k_density_sum_rows<R, true><<<blocks, 256, 0, st>>>(p, w, sums);
  else
    k_density_sum_rows<R, false><<<blocks, 256, 0, st>>>(p, w, sums);
  if (which == 4) {   // over z: column j of [nz][ny]
    launch_combine(sums, p.nz, p.ny, 1.0, nullptr, out, st);
  } else if (which == 5) {   // over y: row k of [nz][ny]
    k_rows_sum<<<(unsigned int)((p.nz + 7) / 8), 256, 0, st>>>(sums, p.nz, p.ny, 1.0, out);
  }
  return cudaGetLastError();
}

#define GP_INSTANTIATE(R)                                                                      \
  template cudaError_t launch_observables<R>(const FieldParams&, bool, bool, cudaStream_t);   \
  template cudaError_t launch_norm_to_scale<R>(const FieldParams&, cudaStream_t);             \
  template cudaError_t launch_half_pointwise<R>(const FieldParams&, bool, const void*,       \
                                                const void*, double, bool, bool, cudaStream_t); \
  template cudaError_t launch_init_gaussian<R>(const FieldParams&, double, double, double,    \
                                               cudaStream_t);                                  \
  template cudaError_t launch_import<R>(const FieldParams&, const double*, bool, cudaStream_t); \
  template cudaError_t launch_export<R>(const FieldParams&, double*, bool, bool, cudaStream_t); \
  template cudaError_t launch_density<R>(const FieldParams&, bool, int, double*, cudaStream_t);
GP_INSTANTIATE(double)
GP_INSTANTIATE(float)
#undef GP_INSTANTIATE

}  // namespace gpk
