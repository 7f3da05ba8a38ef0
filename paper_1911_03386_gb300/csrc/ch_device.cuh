// ch_device.cuh -- device helpers shared by the kernel translation units: block reductions,
// sample partials and finalisation, thread-block cluster access.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ch_internal.h"

namespace chk {
namespace {

using i64 = long long;
constexpr unsigned kAll = 0xffffffffu;

// -------------------------------------------------------------------------------------
// 64-bit fixed point
// -------------------------------------------------------------------------------------
// a b + c, 32 x 32 -> 64 bits, signed.
__device__ __forceinline__ i64 madw(int a, int b, i64 c) {
  i64 d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// v = h 2^32 + l with l signed (so that every partial product is a signed one).
__device__ __forceinline__ FxLimb limbs(i64 v) {
  FxLimb q;
  q.l = (int)v;
  q.h = (int)(v >> 32) + (int)((unsigned)q.l >> 31);
  return q;
}

// a b / 2^64 for |a| <= 2^62, |b| < 2^63, to about one unit: the product of the low limbs (at most
// 1/4 unit) is left out, the middle products are rounded.
__device__ __forceinline__ i64 mul_top(FxLimb a, FxLimb b) {
  const i64 mid = madw(a.l, b.h, madw(a.h, b.l, 1ll << 31));
  return madw(a.h, b.h, mid >> 32);
}

// v / 2^r (1 <= r <= 62), rounded to nearest, halves away from zero (a rounding that is not odd
// in v would bias every point of a field the same way, and the mean is the mode that the solves
// damp least).
__device__ __forceinline__ i64 shift_down(i64 v, int r) { return (v + ((1ll << r) >> 1) + (v >> 63)) >> r; }

// v 2^s for |s| <= 62: f(operation) with the operation for the sign of s (s the same in a warp).
template <class F>
__device__ __forceinline__ void with_shift(int s, const F& f) {
  if (s >= 0)
    f([s](i64 v) { return v << s; });
  else
    f([s](i64 v) { return shift_down(v, -s); });
}


// r + p1 a + p2 b for |a|, |b|, |result| < 2^62, coefficients given / 2^X times 2^64, to about a unit.
// X = 3: |p1| < 2, |p2| < 1, the products of the low limbs (below 2 units) left out; X = 6: both
// below 15, with them.  The middle products are at most 2^61 (l p.h) and 2^61 (h p.l) each, less for
// the smaller coefficient, so their sum stays below 2^63.  They start at 2^63 + 2^(31 - X), so that
// the sum is unsigned and its shift rounds; the high products take the 2^63 back.
template <int X>
__device__ __forceinline__ i64 fixed_dot(FxLimb p1, FxLimb p2, FxLimb a, FxLimb b, i64 r) {
  i64 lo = madw(b.l, p2.h, (i64)((1ull << 63) + (1ull << (31 - X))));
  if (X > 3) lo += (madw(b.l, p2.l, 0) >> 32) + (madw(a.l, p1.l, 0) >> 32);
  lo = madw(b.h, p2.l, lo);
  i64 hi = madw(b.h, p2.h, -(1ll << 31));
  lo = madw(a.l, p1.h, lo);
  lo = madw(a.h, p1.l, lo);
  hi = madw(a.h, p1.h, hi);
  return r + (hi << X) + (i64)((unsigned long long)lo >> (32 - X));
}

// x 2^(59 - E) for |x| < 2^E, E = emax - 1022, from the fields of the binary64 value: the
// 53-bit significand moved up by 6 bits, then down by the distance of its exponent from emax.
__device__ __forceinline__ i64 to_fixed(i64 bits, int emax) {
  const int hi = (int)(bits >> 32);
  const int e = (hi >> 20) & 0x7ff;
  const i64 m = ((i64)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)bits) << 6;
  const i64 v = m >> min(emax - e, 63);
  const i64 s = hi >> 31;
  return (v ^ s) - s;
}

// Binary64 -> binary32 with the significand truncated, from the two formats' fields (IEEE
// 754: binary64 = sign, 11-bit exponent biased by 1023, 52-bit fraction; binary32 = sign,
// 8-bit exponent biased by 127, 23-bit fraction): the exponent is rebiased by 896 and the
// top 23 fraction bits kept, so the relative error is below 2^-23.  |x| < 2^-126 gives a
// signed zero, |x| >= 2^128 (and NaN) a signed infinity.  Integer operations only: the
// FP32 heads of the FP64 pre-rolls leave the FP64 pipe to the FP64 part.
__device__ __forceinline__ float f32_trunc(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned mag = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  const unsigned body = __funnelshift_l(lo, mag - (896u << 20), 3);  // (exp - 896) << 23 | fraction >> 29
  const unsigned bits = mag < (897u << 20) ? sign : (mag >= (1151u << 20) ? (sign | 0x7f800000u) : (sign | body));
  return __uint_as_float(bits);
}

// A line on its way to L2.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }

// Fixed-order block reduction of two FP64 sums (deterministic for a given block size).
__device__ __forceinline__ void block_sum2(double& a, double& b, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) {
    red[2 * warp] = a;
    red[2 * warp + 1] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sa = 0.0, sb = 0.0;
    for (int w = 0; w < nw; ++w) {
      sa += red[2 * w];
      sb += red[2 * w + 1];
    }
    a = sa;
    b = sb;
  }
}

// FP32 form: FP64 partial sums of the F and dF/dt densities over the band's nr rows (C
// tile rows 2..nr+1) with mu recomputed in FP64 from the stored field once per point.  A
// warp walks a strip of rows down a chunk of 31 columns, carrying three C rows and two mu
// rows in registers; lane 31 holds the column after the chunk, so east neighbours come
// from the next lane.  The work is split over the first nwarps warps and added in their order, so the
// sums depend on nwarps but on no other property of the CTA.
template <typename T>
__device__ void band_partials_mu64(const DevView& v, const Tile& tl, int nx, int nr, const MemberParams& P,
                                   double2* slot, double* red, int nwarps) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double a = P.a, bx = P.bx, by = P.by;
  // the stored field in FP64 (hi + lo for compensated members), read from global memory:
  // band row q of the tile is field row j0 - 2 + q (periodic)
  const T* Hg = static_cast<const T*>(v.C) + P.offset;
  const T* Lg = P.comp ? static_cast<const T*>(v.C) + P.lo_offset : nullptr;
  const int ny = P.ny;
  // field row of band row q (q from -1 to nr + 3, j0 - 3 .. j0 + nr + 1): one wrap at most
  auto at = [&](int q, int ii) {
    int j = tl.start - 2 + q;
    j = j < 0 ? j + ny : (j >= ny ? j - ny : j);
    const int64_t k = (int64_t)j * nx + ii;
    return Lg ? (double)Hg[k] + (double)Lg[k] : (double)Hg[k];
  };
  const int nchunk = (nx + 30) / 31;
  const int nstrip = max(1, nwarps / nchunk);
  const int hs = (nr + nstrip - 1) / nstrip;
  // unscaled sums: (C^2 - 1)^2, (D+x C)^2, (D+y C)^2, (D+x mu)^2, (D+y mu)^2 (the grid
  // spacings and prefactors are applied once per thread at the end)
  double sw = 0.0, sdx = 0.0, sdy = 0.0, smx = 0.0, smy = 0.0;
  for (int item = warp < nwarps ? warp : nchunk * nstrip; item < nchunk * nstrip; item += nwarps) {
    const int k = item % nchunk, r0 = (item / nchunk) * hs, r1 = min(nr, r0 + hs);
    if (r0 >= r1) continue;
    const int i = (31 * k + lane) % nx;
    const bool own = lane < 31 && 31 * k + lane < nx;
    const int iw = i == 0 ? nx - 1 : i - 1, ie = i + 1 == nx ? 0 : i + 1;
    // C at tile row q in FP64, and its west / east neighbours (shuffles inside the chunk)
    auto cload = [&](int q) { return at(q, i); };
    auto mu_row = [&](int q, double cq, double cdn, double cup) {
      double w = __shfl_up_sync(full, cq, 1), e = __shfl_down_sync(full, cq, 1);
      if (lane == 0) w = at(q, iw);
      if (lane == 31) e = at(q, ie);
      return cq * (cq * cq - a) - bx * (e + w) - by * (cup + cdn);
    };
    const int q0 = r0 + 2;
    double cm = cload(q0 - 1), c0 = cload(q0), c1 = cload(q0 + 1), c2 = cload(q0 + 2);
    double mu0 = mu_row(q0, c0, cm, c1);
    double mu1 = mu_row(q0 + 1, c1, c0, c2);
    for (int r = r0; r < r1; ++r) {
      const double ce = __shfl_down_sync(full, c0, 1);
      const double mue = __shfl_down_sync(full, mu0, 1);
      if (own) {
        const double w = c0 * c0 - 1.0, gx = ce - c0, gy = c1 - c0, mx = mue - mu0, my = mu1 - mu0;
        sw += w * w;
        sdx += gx * gx;
        sdy += gy * gy;
        smx += mx * mx;
        smy += my * my;
      }
      if (r + 1 < r1) {  // advance: row q+3 enters, mu of row q+2
        const double c3 = cload(r + 5);
        const double mu2 = mu_row(r + 4, c2, c1, c3);
        c0 = c1;
        c1 = c2;
        c2 = c3;
        mu0 = mu1;
        mu1 = mu2;
      }
    }
  }
  const double hxi2 = 1.0 / (P.hx * P.hx), hyi2 = 1.0 / (P.hy * P.hy);
  double sF = 0.25 * sw + 0.5 * P.gamma * (hxi2 * sdx + hyi2 * sdy);
  double sD = hxi2 * smx + hyi2 * smy;
  block_sum2(sF, sD, red);
  if (threadIdx.x == 0) *slot = make_double2(sF, sD);
}

// x 2^(59 - E) of a binary32 value, as to_fixed (zero and subnormal values count as zero).
__device__ __forceinline__ i64 to_fixed(float x, int emax) {
  const int b = __float_as_int(x), e = (b >> 23) & 0xff;
  if (e == 0) return 0;
  const i64 m = (i64)((b & 0x7fffff) | 0x800000) << 35;  // leading one at bit 58, as in to_fixed(i64)
  const i64 v = m >> min(max(emax - (e + 896), 0), 63);
  const i64 s = b >> 31;
  return (v ^ s) - s;
}

// A sum of squares of up to 15 fixed-point values |v| < 2^60, exact: v = h 2^32 + l, the sums of
// h h, h l (below 2^59 each) and the high words of l l.
struct SquareSum {
  i64 hh = 0, hl = 0;
  unsigned long long ll = 0;
  __device__ __forceinline__ void add(i64 v) {
    const FxLimb q = limbs(v);
    hh = madw(q.h, q.h, hh);
    hl = madw(q.h, q.l, hl);
    ll += (unsigned long long)madw(q.l, q.l, 0) >> 32;
  }
  // the lanes' sums / 2^16, rounded down, added over the warp: hi 2^64 + lo, in every lane
  __device__ __forceinline__ void warp_total(i64& hi, unsigned long long& lo) const {
    const unsigned long long l1 = (unsigned long long)hl << 33, l2 = ll << 32;
    lo = l1 + l2;
    hi = hh + (hl >> 31) + (i64)(ll >> 32) + (lo < l1 ? 1 : 0);
    lo = (lo >> 16) | ((unsigned long long)hi << 48);
    hi >>= 16;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long x = __shfl_xor_sync(kAll, lo, o);
      const i64 y = __shfl_xor_sync(kAll, hi, o);
      lo += x;
      hi += y + (lo < x ? 1 : 0);
    }
  }
};

// v / 2^r of a constant, r >= 0, rounded.
__device__ __forceinline__ FxLimb cut_limb(FxLimb q, int r) {
  const i64 v = ((i64)q.h << 32) + q.l;
  return r > 0 ? limbs(shift_down(v, r)) : q;
}

__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// Partial sums of the F and dF/dt densities (in thread 0) over nr rows of a field of nx columns in
// fixed point: load(r, i) = field row r (-1 .. nr + 1, relative to the first row) at column i,
// conv(value, emax) its fixed-point form, mag(r, i) = a biased binary64 exponent not below the
// value's.  On sample steps these sums took the FP64 pipe 25 operations per point, 64 clocks each per
// warp and scheduler: a sample cost as much as 7 FP64 or 30 FP32 steps.  In integers (the arithmetic
// of the step's mu, sums of squares of 128 bits per strip and lane added exactly, so the result does
// not depend on the CTA's size) it costs about one.  A warp takes 29 columns (lanes 0, 30 and 31 are their neighbours) of a
// strip of 4 or 8 rows.  sums: 80 bytes of shared memory; ends with every thread past a barrier;
// false (nothing summed) where the values' range does not fit, the same in every thread.  MAXE: |C| <
// 2^MAXE fits, 1 for CH_FP32 (with the exponents of the CH_FP64 step the resident kernel around it took
// 48.6 us per step of 256 x 256^2 instead of 47.5, samples or not).
template <int MAXE, class Load, class Conv, class Mag>
__device__ __noinline__ bool fixed_partials(const MemberParams& P, int nx, int nr, unsigned long long* sums, Load load,
                                            Conv conv, Mag mag, double& sF, double& sD) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nchunk = (nx + 28) / 29;
  const int hs = nx <= 64 ? 4 : 8, nstrip = (nr + hs - 1) / hs;
  unsigned* slots = reinterpret_cast<unsigned*>(sums);
  int top = 0;
  for (int item = warp; item < nchunk * nstrip; item += nw) {
    const int k = item % nchunk, r0 = (item / nchunk) * hs, r1 = min(nr, r0 + hs);
    const int i = (29 * k + lane + nx - 1) % nx;
#pragma unroll 6
    for (int r = r0 - 1; r < r1 + 2; ++r) top = max(top, mag(r, i));
  }
  top = __reduce_max_sync(kAll, top);
  if (lane == 0) slots[warp] = (unsigned)top;
  __syncthreads();
  const int emax = __reduce_max_sync(kAll, lane < nw ? (int)slots[lane] : 0);
  __syncthreads();
  if (!P.fx_mu || emax > 1022 + MAXE || emax < 823) return false;
  if (threadIdx.x < 10) sums[threadIdx.x] = 0;
  __syncthreads();
  const int E = emax - 1022, cut = MAXE > 1 && E > 1 ? P.fx_cut[E - 2] : 0;
  const int wb = MAXE > 1 ? 60 - 2 * max(E, 1) : 58, sh = max(2 * E + wb - 54, -63);  // C^2 - 1 is held times 2^wb
  const i64 one = 1ll << wb;
  const FxLimb bx = cut_limb(P.fx_bx, cut), by = cut_limb(P.fx_by, cut);
  const int su = P.fx_su + cut + wb - 60;  // the cubic term from (C^2 - 1) 2^wb
  auto scaled = [](i64 v, int s) { return s >= 0 ? v << s : v >> -s; };
  for (int item = warp; item < nchunk * nstrip; item += nw) {
    const int k = item % nchunk, r0 = (item / nchunk) * hs, r1 = min(nr, r0 + hs);
    if (r0 >= r1) continue;
    const int i = (29 * k + lane + nx - 1) % nx;
    const bool own = lane >= 1 && lane <= 29 && 29 * k + lane - 1 < nx;
    auto mu_of = [&](i64 c, i64 e, i64 w, i64 n, i64 s, i64& q) {
      const FxLimb cl = limbs(c);
      q = scaled(mul_top(cl, cl), sh) - one;
      const i64 u = mul_top(cl, limbs(scaled(q, -su)));
      return u - mul_top(limbs(e + w - 2 * c), bx) - mul_top(limbs(n + s - 2 * c), by);
    };
    SquareSum w2, gx2, gy2, mx2, my2;
    const auto vm = load(r0 - 1, i), v0 = load(r0, i), v1 = load(r0 + 1, i);
    auto next = load(r0 + 2, i);
    const i64 cm = conv(vm, emax);
    i64 c0 = conv(v0, emax), c1 = conv(v1, emax), q0, q1;
    i64 e0 = __shfl_down_sync(kAll, c0, 1);
    i64 mu0 = mu_of(c0, e0, __shfl_up_sync(kAll, c0, 1), cm, c1, q0);
    for (int r = r0; r < r1; ++r) {
      const i64 c2 = conv(next, emax);
      if (r + 1 < r1) next = load(r + 3, i);  // in flight while this row is summed
      const i64 e1 = __shfl_down_sync(kAll, c1, 1);
      const i64 mu1 = mu_of(c1, e1, __shfl_up_sync(kAll, c1, 1), c0, c2, q1);
      const i64 mue = __shfl_down_sync(kAll, mu0, 1);
      if (own) {
        w2.add(q0);
        gx2.add(e0 - c0);
        gy2.add(c1 - c0);
        mx2.add(mue - mu0);
        my2.add(mu1 - mu0);
      }
      c0 = c1;
      c1 = c2;
      e0 = e1;
      mu0 = mu1;
      q0 = q1;
    }
    i64 hi, th;
    unsigned long long lo, tlo;
    w2.warp_total(hi, lo);
    auto take = [&](const SquareSum& q, int at) {
      q.warp_total(th, tlo);
      if (lane == at) {
        hi = th;
        lo = tlo;
      }
    };
    take(gx2, 1);
    take(gy2, 2);
    take(mx2, 3);
    take(my2, 4);
    if (lane < 5) {
      const unsigned long long old = atomicAdd(sums + 2 * lane, lo);
      atomicAdd(sums + 2 * lane + 1, (unsigned long long)hi + (old + lo < old ? 1 : 0));
    }
  }
  __syncthreads();
  if (warp == 0) {
    // lane q: sum q: (C^2 - 1)^2 / 4, gamma / 2 of (D+x C)^2 and (D+y C)^2, (D+x mu)^2, (D+y mu)^2
    const int q = min(lane, 4);
    const double hinv = (q & 1) ? P.ihx2 : P.ihy2;
    const double weight = q == 0 ? pow2(14 - 2 * wb) : q < 3 ? 0.5 * P.gamma * pow2(16 + 2 * (E - 59)) * hinv
                                                          : pow2(16 + 2 * (E - P.fx_kmu + cut)) * hinv;
    const double s = weight * fma((double)sums[2 * q + 1], 18446744073709551616.0, (double)sums[2 * q]);
    sF = s + (__shfl_sync(kAll, s, 1) + __shfl_sync(kAll, s, 2));
    sD = __shfl_sync(kAll, s, 3) + __shfl_sync(kAll, s, 4);
  }
  __syncthreads();
  return true;
}

// The band's partial sums (tile tl) from the stored field in global memory, FP64 values or FP32 ones
// (hi + lo for compensated members): in fixed point, or in FP64 where the range does not fit (split over
// nwarps warps, all of the CTA's if 0).
template <typename T>
__device__ void band_partials_field(const DevView& v, const Tile& tl, int nx, int nr, const MemberParams& P,
                                    double2* slot, double* red, int nwarps = 0) {
  const T* H = static_cast<const T*>(v.C) + P.offset;
  const T* Lo = P.comp ? static_cast<const T*>(v.C) + P.lo_offset : nullptr;
  const int ny = P.ny, j0 = tl.start;
  auto index = [=](int r, int i) {
    int j = j0 + r;
    j = j < 0 ? j + ny : (j >= ny ? j - ny : j);
    return (int64_t)j * nx + i;
  };
  double sF, sD;
  const bool ok = fixed_partials<sizeof(T) == 8 ? kFxMaxE : 1>(
      P, nx, nr, reinterpret_cast<unsigned long long*>(red),
      [=](int r, int i) {
        const int64_t k = index(r, i);
        if constexpr (sizeof(T) == 8)
          return (i64)__double_as_longlong(H[k]);
        else
          return make_float2((float)H[k], Lo ? (float)Lo[k] : 0.0f);
      },
      [=](auto x, int emax) -> i64 {
        if constexpr (sizeof(T) == 8)
          return to_fixed(x, emax);
        else
          return Lo ? to_fixed(x.x, emax) + to_fixed(x.y, emax) : to_fixed(x.x, emax);
      },
      [=](int r, int i) -> int {
        const int64_t k = index(r, i);
        if constexpr (sizeof(T) == 8) return (int)(__double2hiint(H[k]) >> 20) & 0x7ff;
        const int e = (__float_as_int((float)H[k]) >> 23) & 0xff;
        return e == 255 ? 2047 : e == 0 ? 0 : e + 896;
      },
      sF, sD);
  if (!ok) {
    band_partials_mu64<T>(v, tl, nx, nr, P, slot, red, nwarps ? nwarps : (int)(blockDim.x >> 5));
    return;
  }
  if (threadIdx.x == 0) *slot = make_double2(sF, sD);
}

// Active flag and sample decision of a stencil-phase CTA.
__device__ __forceinline__ bool stencil_prologue(const Tile& tl, MemberState* st, const MemberParams& P, bool& sample) {
  const bool active = st->remaining > 0;
  if (tl.index == 0 && threadIdx.x == 0) st->active = active ? 1 : 0;
  sample = (st->step % P.every) == 0;
  return active;
}

__device__ __forceinline__ double* red_buffer(unsigned char* smem, size_t tile_bytes) {
  return reinterpret_cast<double*>(smem + ((tile_bytes + 15) & ~(size_t)15));
}

// The sample itself from the member's summed partials (sF, sD): F, dF/dt, beta, the series
// ring and the window average; then the step counter and horizon advance.
__device__ __forceinline__ void finalize_sums(const DevView& v, int member, MemberState* st, const MemberParams& P,
                                              double sF, double sD) {
  const int64_t n = st->step;
  if (n % P.every == 0) {
    const double hh = P.hx * P.hy;
    const double F = hh * sF;
    const double dFdt = -(hh * sD);
    const double t = (double)n * P.dt;
    const double beta = -(t / F) * dFdt;
    st->F = F;
    st->dFdt = dFdt;
    st->beta = beta;
    if (!isfinite(F) || !isfinite(dFdt)) st->nonfinite = 1;
    if (P.series_cap > 0) {
      double* s = v.series + ((size_t)member * P.series_cap + (size_t)(st->nsamples % P.series_cap)) * 4;
      s[0] = t;
      s[1] = F;
      s[2] = dFdt;
      s[3] = beta;
    }
    st->nsamples += 1;
    if (t >= P.t1) {
      st->beta_sum += beta;
      st->beta_count += 1;
    }
  }
  st->step = n + 1;
  if (st->remaining != kUnbounded) st->remaining -= 1;
}

// Sample finalisation of one member (called once per member and step by the column phase,
// after the stencil phase wrote the band partials): the partials summed in band order, then
// finalize_sums.
__device__ __forceinline__ void finalize_sample(const DevView& v, int member, MemberState* st, const MemberParams& P) {
  double sF = 0.0, sD = 0.0;
  if (st->step % P.every == 0) {
    for (int b = 0; b < P.nbands; ++b) {
      const double2 pr = v.partials[P.partial_base + b];
      sF += pr.x;
      sD += pr.y;
    }
  }
  finalize_sums(v, member, st, P, sF, sD);
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Shared-memory address of p in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned peer_addr(const void* p, unsigned rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

__device__ __forceinline__ float ld_peer(unsigned addr, float) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(addr) : "memory");
  return x;
}
__device__ __forceinline__ double ld_peer(unsigned addr, double) {
  double x;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(addr) : "memory");
  return x;
}

}  // namespace
}  // namespace chk
