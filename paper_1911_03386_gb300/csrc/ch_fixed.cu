// ch_fixed.cu -- the CH_FP64 step in 64-bit fixed point (sm_103a).
//
// GB300's FP64 pipe takes 2 operations per SM and clock, so an FP64 recurrence step (2 FMA)
// costs a warp 38 SM clocks; the same step in 64-bit fixed point (six 32 x 32 -> 64 bit
// multiply-adds and a few adds) costs 8.7 (measured, 16 or more warps per SM).  The step of a
// CH_FP64 member is therefore formed in 64-bit integers with power-of-two scales taken from
// the data: C enters with 59 bits below its band's scale, the solves hold 62 bits less the
// recurrences' gain (2^1 at s = 0.9, 2^5 at s = 900, 2^8 at s = 5e4), where FP64 holds 53; the
// fields stay FP64 in memory and the update C += kappa Z is one FP64 FMA.
//
//   fx_rows_kernel   a band of rows: C -> mu -> R' -> both row recurrences -> W (64-bit
//                    integers, one exponent per row)
//   fx_cols_kernel   a panel of up to 32 columns: both column recurrences of W, C += kappa Z
//
// Measured (a step of a whole ensemble; in brackets the FP64 kernels): 256 x 256^2 rows 212 + columns
// 138 us, 0.352 ms (0.650 ms), 16 x 1024^2 0.402 ms (1.16 ms), 64^2 alone 14.7 us (58 us).  At 256^2 a
// point takes 331 instructions of the row kernel and 175 of the column kernel; both are bound by issue
// slots and the integer multiply pipe (65 % and 53 % of the issue slots, 59 % and 52 % of that pipe),
// not by HBM (40 bytes per point, 0.1 ms).  Oblong grids (hx != hy) pay 2 % for the precision of R'.
//
// Scales.  x = C / 2^E with 2^E just above the band's largest |C| (E from an integer maximum
// over the loaded values); C enters as x 2^59, mu as mu 2^(kmu - E), where kmu leaves room for
// the largest R' the stencil can form from such a band (so mu's unit is a few bits below the
// rounding of the FP64 formula, whose terms 4 (bx + by) C are as large), R' is formed in units
// of the closer spacing, from mu exactly where hx = hy.  Each recurrence y_i = r_i + p1 y_{i-1}
// + p2 y_{i-2} then runs on r shifted so that its row's (or panel's) largest value sits g bits
// below 2^62, 2^g a bound of the recurrence's gain (the l1 norm of its impulse response), and
// its result is shifted the same way before the backward one.
//
// A band whose largest |C| is outside [2^-200, 8), or not finite, is taken through the same code
// in FP64 arithmetic (the Fp policy: 0.91 ms per step of 256 x 256^2 where every band is, FP64
// kernels 0.65; 16 x 1024^2 1.01 and 1.15; 64^2 alone 24 and 55 us), its rows marked kBadRow;
// the columns of a member with such a row run in FP64 too.  So do a band in which some block of
// 32 columns (16 to 32 at the end of a row) by 4 rows (halo rows included) holds only values
// below 2^-10 of the band's largest, and the columns of a member whose bands' largest values
// differ by that much: a value that far below the one that sets its scale would keep fewer bits
// than in FP64, which shows in regions so quiet beside others (a field grown from a local seed:
// 1e-12 noise beside it had a relative error of 7e-3 after a step, now FP64's 2e-12). Above that
// line the error is FP64's or less relative to the run's largest |C|, and within a factor of 16
// of it relative to a block's.  Four rows: a nodal line of one or two rows is no quiet region,
// and the two rows next to an active one take its flux within the step.
//
// Lines of n points are split into G = ceil(n / S) segments of S points (the last one may be
// shorter), one lane (rows) or warp (columns) per segment.  Each recurrence is a pass from a
// zero state over every segment, a Kogge-Stone scan of the end states (in the same arithmetic: in
// FP64 it took the FP64 pipe a fifth of the kernels' time) and a pass from the exact periodic
// start state.
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "ch_device.cuh"
#include "ch_internal.h"

namespace chk {
namespace {

// Asynchronous global -> shared copy of one value.
__device__ __forceinline__ void copy8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

__device__ __forceinline__ i64 double_bits(double x) { return __double_as_longlong(x); }

// Arithmetic of the recurrences: fixed point ...
struct Fx {
  using State = FxLimb;
  FxLimb p1, p2;  // p / 8, times 2^64
  unsigned top = 0;  // OR of the magnitudes' high words
  __device__ __forceinline__ Fx(const FxCoef& c, double, double) : p1(c.p1), p2(c.p2) {}
  static __device__ __forceinline__ State zero() { return FxLimb{0, 0}; }
  __device__ __forceinline__ i64 step(State a, State b, i64 r) const { return fixed_dot<3>(p1, p2, a, b, r); }
  // row[0] x0 + row[1] x1 + r of the scans
  static __device__ __forceinline__ i64 dot(const FxLimb* row, i64 x0, i64 x1, i64 r) {
    return fixed_dot<6>(row[0], row[1], limbs(x0), limbs(x1), r);
  }
  static constexpr bool kFixed = true;
  static __device__ __forceinline__ State state(i64 y) { return limbs(y); }
  static __device__ __forceinline__ i64 value(State s) { return ((i64)s.h << 32) + s.l; }
  __device__ __forceinline__ void track(i64 y) {
    const int h = (int)(y >> 32);
    top |= (unsigned)(h ^ (h >> 31));
  }
};

// ... and FP64 (values held as their bits).
struct Fp {
  using State = double;
  double p1, p2;
  unsigned top = 0;
  __device__ __forceinline__ Fp(const FxCoef&, double q1, double q2) : p1(q1), p2(q2) {}
  static __device__ __forceinline__ State zero() { return 0.0; }
  __device__ __forceinline__ i64 step(State a, State b, i64 r) const {
    return double_bits(fma(p1, a, fma(p2, b, __longlong_as_double(r))));
  }
  static constexpr bool kFixed = false;
  static __device__ __forceinline__ State state(i64 y) { return __longlong_as_double(y); }
  static __device__ __forceinline__ i64 value(State s) { return double_bits(s); }
  // (a table of fp64_tables)
  static __device__ __forceinline__ i64 dot(const FxLimb* row, i64 x0, i64 x1, i64 r) {
    const double* m = reinterpret_cast<const double*>(row);
    return double_bits(fma(m[0], __longlong_as_double(x0), fma(m[1], __longlong_as_double(x1), __longlong_as_double(r))));
  }
  __device__ __forceinline__ void track(i64) {}
};

// One pass of a recurrence over a segment of len values in shared memory, `es` elements apart
// (p: its first value in the pass's direction, es negative for the backward one), from the
// state (a, b); the loads of four values are issued ahead of the chain.  PRE: each value is first
// replaced by pre(value).  STORE: the solution replaces the values.
template <bool STORE, bool PRE, class A, class Pre>
__device__ __forceinline__ void pass(A& ar, i64* p, int es, int len, typename A::State& a, typename A::State& b,
                                     const Pre& pre) {
  auto one = [&](i64 r, i64* at) {
    if constexpr (PRE) {
      r = pre(r);
      *at = r;
    }
    const i64 t = ar.step(a, b, r);
    if constexpr (STORE) {
      *at = t;
      ar.track(t);
    }
    b = a;
    a = A::state(t);
  };
  int k = 0;
#pragma unroll 1
  for (; k + 4 <= len; k += 4) {
    i64 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = p[u * es];
#pragma unroll
    for (int u = 0; u < 4; ++u) one(v[u], p + u * es);
    p += 4 * es;
  }
#pragma unroll 1
  for (; k < len; ++k) {
    one(*p, p);
    p += es;
  }
}
// The zero-state pass over the values shifted by sl (FP64: unshifted), and the pass from a state.
template <class A>
__device__ __forceinline__ void pass_end(A& ar, i64* p, int es, int len, int sl, typename A::State& a,
                                         typename A::State& b) {
  a = A::zero();
  b = A::zero();
  if constexpr (A::kFixed)
    with_shift(sl, [&](auto sh) { pass<false, true>(ar, p, es, len, a, b, sh); });
  else
    pass<false, false>(ar, p, es, len, a, b, 0);
}
template <class A>
__device__ __forceinline__ void pass_full(A& ar, i64* p, int es, int len, typename A::State a, typename A::State b) {
  ar.top = 0;
  pass<true, false>(ar, p, es, len, a, b, 0);
}

// Start states of the segments of one line from their end states, one lane per segment (the
// first G of gw consecutive lanes, gw a power of two; l = lane within them).  The line's last
// segment may be shorter than the others; tab.A[d] = M^(S 2^d), tab.P = M^(length of the last
// segment), tab.B[l] = M^(S l) P, tab.B[32 + pos] = M^(distance from the line's end) P with P
// = (I - M^n)^-1, all in shared memory.  (a, b): end state in, start state out.
struct alignas(16) ScanTab {
  FxLimb A[5][4], P[4], B[64][4];  // entries / 64, times 2^64, row-major
};
// The table into shared memory (16-byte asynchronous copies: Ax, Px, Bx lie like A, P, B).
__device__ __forceinline__ void load_tab(ScanTab& t, const SegTable& g) {
  static_assert(sizeof(ScanTab) % 16 == 0, "whole pieces");
  for (int k = threadIdx.x; k < (int)(sizeof(ScanTab) / 16); k += blockDim.x)
    copy16(reinterpret_cast<char*>(&t) + 16 * k, reinterpret_cast<const char*>(&g.Ax[0][0]) + 16 * k);
}

// The Fp policy's tables in place of the fixed-point ones, whose entries are exact to 2^-59: not enough
// for values that differ by more, which is why a band is in FP64.  Warp 0, lane l segment l; the caller's
// barriers order it.  The scans take all levels: no power vanishes.
__device__ __forceinline__ void fp64_tables(ScanTab& t, const SegTable& g) {
  if (threadIdx.x < 32) {
    const int l = threadIdx.x;
    auto put = [](FxLimb* to, double a, double b, double c, double d) {
      double* q = reinterpret_cast<double*>(to);
      q[0] = a;
      q[1] = b;
      q[2] = c;
      q[3] = d;
    };
    const double *tail = g.Dx[5], *own = g.Dx[6 + l], *before = g.Dx[6 + max(l - 1, 0)];
    if (l < 5) put(t.A[l], g.Dx[l][0], g.Dx[l][1], g.Dx[l][2], g.Dx[l][3]);
    if (l == 5) put(t.P, tail[0], tail[1], tail[2], tail[3]);
    put(t.B[l], own[0], own[1], own[2], own[3]);
    if (l == 0)
      put(t.B[32], own[0], own[1], own[2], own[3]);
    else  // the last segment's own length, then the others
      put(t.B[32 + l], fma(tail[0], before[0], tail[1] * before[2]), fma(tail[0], before[1], tail[1] * before[3]),
          fma(tail[2], before[0], tail[3] * before[2]), fma(tail[2], before[1], tail[3] * before[3]));
  }
}
__device__ __forceinline__ int all_levels(int G) { return 32 - __clz(G - 1); }

// Programmatic dependent launch: a step kernel lets its successor start (its CTAs take the SMs'
// free slots, read their constant tables and wait) and waits itself until its predecessor has
// finished and its writes are visible.  What is read before the wait -- the tiles and the scan
// tables -- must therefore not come from the predecessor (tables_ready, launch_fx_rows).  64^2 alone:
// 20.2 us per step without it, 14.7 with it.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.launch_dependents;\ngriddepcontrol.wait;\n" ::: "memory");
}

template <bool REV, class A>
__device__ __forceinline__ void scan_states(const ScanTab& tab, i64& a, i64& b, int l, int G, int gw, int levels, bool full) {
  const int pos = REV ? G - 1 - l : l;
  const i64 e0 = a, e1 = b;
#pragma unroll 1
  for (int d = 0, delta = 1; d < levels; ++d, delta *= 2) {
    const i64 ya = REV ? __shfl_down_sync(kAll, a, delta, gw) : __shfl_up_sync(kAll, a, delta, gw);
    const i64 yb = REV ? __shfl_down_sync(kAll, b, delta, gw) : __shfl_up_sync(kAll, b, delta, gw);
    if (pos >= delta) {
      a = A::dot(tab.A[d], ya, yb, a);
      b = A::dot(tab.A[d] + 2, ya, yb, b);
    }
  }
  i64 xa = REV ? __shfl_down_sync(kAll, a, 1, gw) : __shfl_up_sync(kAll, a, 1, gw);
  i64 xb = REV ? __shfl_down_sync(kAll, b, 1, gw) : __shfl_up_sync(kAll, b, 1, gw);
  if (pos == 0) xa = xb = 0;
  i64 ta = a, tb = b;
  if (!REV && !full) {  // the last segment's own length
    ta = A::dot(tab.P, xa, xb, e0);
    tb = A::dot(tab.P + 2, xa, xb, e1);
  }
  ta = __shfl_sync(kAll, ta, REV ? 0 : G - 1, gw);
  tb = __shfl_sync(kAll, tb, REV ? 0 : G - 1, gw);
  const FxLimb* B = tab.B[REV ? 32 + max(pos, 0) : min(l, 31)];
  a = A::dot(B, ta, tb, xa);
  b = A::dot(B + 2, ta, tb, xb);
}

__device__ __forceinline__ int bit_length_hi(unsigned top) { return 64 - __clz((int)top); }  // >= 32

// -------------------------------------------------------------------------------------
// Rows
// -------------------------------------------------------------------------------------
// mu at c with neighbours e, w, n, s (SQ: hx = hy, one product for both directions).  The cubic
// term: (C^2 - 1) 2^(60 - su) from C^2's product by one shift (sh = 2 E + 6 - su), times C.
template <bool SQ, class Shift>
struct MuFx {
  FxLimb pbx, pby;
  i64 one;
  Shift sh;
  __device__ __forceinline__ i64 operator()(i64 c, i64 e, i64 w, i64 n, i64 s) const {
    const FxLimb cl = limbs(c);
    const i64 u = mul_top(cl, limbs(sh(mul_top(cl, cl)) - one));
    const i64 lx = e + w - 2 * c, ly = n + s - 2 * c;
    if (SQ) return u - mul_top(limbs(lx + ly), pbx);
    return u - mul_top(limbs(lx), pbx) - mul_top(limbs(ly), pby);
  }
};
struct MuFp {
  double a, bx, by;
  __device__ __forceinline__ i64 operator()(i64 c_, i64 e_, i64 w_, i64 n_, i64 s_) const {
    const double c = __longlong_as_double(c_), e = __longlong_as_double(e_), w = __longlong_as_double(w_),
                 n = __longlong_as_double(n_), s = __longlong_as_double(s_);
    return double_bits(fma(-by, s + n, fma(-bx, e + w, c * fma(c, c, -a))));
  }
};
// R' at m with neighbours e, w, n, s, in units of the closer spacing (FORM 0: hx = hy, exact; 1: hx <
// hy, dx + ratio dy; 2: hx > hy, ratio dx + dy).  The product's rounding is the one rounding in R'
// that no difference damps afterwards, so forms 1 and 2 first move the differences up by the `up`
// bits that the band's largest |mu| leaves free (mu of a smooth field is far below the bound that
// sets its unit).
template <int FORM>
struct RhsFx {
  FxLimb ratio;
  int er, up = 0;
  __device__ __forceinline__ i64 operator()(i64 m, i64 e, i64 w, i64 n, i64 s) const {
    const i64 dx = e + w - 2 * m, dy = n + s - 2 * m;
    if (FORM == 0) return dx + dy;
    const i64 d = FORM == 1 ? dx : dy, q = FORM == 1 ? dy : dx;
    return (d << up) + mul_top(limbs(q << (er + up)), ratio);
  }
};
struct RhsFp {
  bool tall;
  double ratio, w0;
  __device__ __forceinline__ i64 operator()(i64 m_, i64 e_, i64 w_, i64 n_, i64 s_) const {
    const double m = __longlong_as_double(m_), e = __longlong_as_double(e_), w = __longlong_as_double(w_),
                 n = __longlong_as_double(n_), s = __longlong_as_double(s_);
    const double x = e + w, y = s + n, p = tall ? x : y, q = tall ? y : x;
    return double_bits(fma(w0, m, fma(ratio, p, q)));
  }
};

// One band of nr rows (up to TH / gw).  The band's C rows (with two halo rows on each side) go to
// a shared-memory tile whose rows are padded by one value per segment of S, so that lanes S + 1
// values apart fall in distinct banks.  Warps take strips of 32 columns down the rows, twice and
// in place: mu from three C rows in registers and the neighbouring lanes, written over the C row
// above, then R' from three mu rows the same way (strip edges of both through shared memory).
// Then gw lanes take each row for both recurrences.  All of it runs in short loops over shared
// memory: fully unrolled register forms of this kernel spent a third of their cycles fetching
// instructions, and their registers held an SM to 16 warps.
struct Band {
  i64* tile;
  int pitch, ls;       // tile pitch; log2 S: column i at i + (i >> ls)
  int nx, ns, nr;      // columns, strips, band rows
};

// First element of an edge column (rows values) of a strip.
__device__ __forceinline__ int edge_index(int rows, int strip, int side) { return (2 * strip + side) * rows; }

// A walk of every strip down `rows` output rows: out row r = f(c, e, w, n, s) with n, c, s the
// input rows r, r + 1, r + 2 (conv applied on entry), written over input row r.  Ein: edge columns
// of the input rows; each output row goes to `sink` (value, row, valid lane) before it is stored.
template <class Conv, class F, class Sink>
__device__ __forceinline__ void walk_strips(const Band& b, int rows, const i64* Ein, const Conv& conv, const F& f,
                                            const Sink& sink) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int s = threadIdx.x >> 5; s < b.ns; s += nw) {
    const int last = min(31, b.nx - 1 - 32 * s);
    const int i = 32 * s + min(lane, last);
    i64* col = b.tile + i + (i >> b.ls);
    // west edge of lane 0: right edge of the strip before; east edge of the last lane: left edge
    // of the strip after
    const i64* ew = Ein + edge_index(rows + 2, s == 0 ? b.ns - 1 : s - 1, 1) + 1;
    const i64* ee = Ein + edge_index(rows + 2, s + 1 == b.ns ? 0 : s + 1, 0) + 1;
    i64 n = conv(col[0]), c = conv(col[b.pitch]);
#pragma unroll 2
    for (int r = 0; r < rows; ++r) {
      const i64 so = conv(col[2 * b.pitch]);
      i64 w = __shfl_up_sync(kAll, c, 1), e = __shfl_down_sync(kAll, c, 1);
      if (lane == 0) w = ew[r];
      if (lane == last) e = ee[r];
      const i64 m = f(c, e, w, n, so);
      sink(m, s, r, lane, last);
      if (lane <= last) col[0] = m;
      col += b.pitch;
      n = c;
      c = so;
    }
  }
}

// OR of `top` over the CTA (slots: one per warp, not in use; ends with every thread past it).
template <int NW>
__device__ __forceinline__ unsigned cta_or(unsigned top, unsigned* slots) {
  const int lane = threadIdx.x & 31;
  top = __reduce_or_sync(kAll, top);
  if (lane == 0) slots[threadIdx.x >> 5] = top;
  __syncthreads();
  return __reduce_or_sync(kAll, lane < NW ? slots[lane] : 0u);
}

// mu, then R' (with the OR of its magnitudes in top), over the tile.  FORM: of RhsFx, or -1 in FP64;
// slots: one word per warp, not in use.
template <int NW, int FORM, class Mu, class Rhs>
__device__ __forceinline__ void band_rhs(const Band& b, i64* Es, i64* Em, unsigned& top, int emax, const Mu& mu, Rhs& rhs,
                                         unsigned* slots) {
  constexpr bool FIXED = FORM >= 0;
  const auto magnitude = [](i64 m) {
    const int h = (int)(m >> 32);
    return (unsigned)(h ^ (h >> 31));
  };
  top = 0;
  walk_strips(
      b, b.nr + 2, Es, [emax](i64 c) { return FIXED ? to_fixed(c, emax) : c; }, mu,
      [&](i64 m, int s, int r, int lane, int last) {
        if (lane == 0) Em[edge_index(b.nr + 2, s, 0) + r] = m;
        if (lane == last) Em[edge_index(b.nr + 2, s, 1) + r] = m;
        if (FORM > 0 && lane <= last) top |= magnitude(m);
      });
  // a difference is at most 4 |mu|: below 2^62 moved up by er + up, R' (twice that) below 2^62 by up
  if constexpr (FORM > 0)
    rhs.up = max(0, 60 - max(rhs.er, 1) - bit_length_hi(cta_or<NW>(top, slots)));
  else
    __syncthreads();
  top = 0;
  walk_strips(
      b, b.nr, Em, [](i64 m) { return m; }, rhs,
      [&](i64 m, int, int, int lane, int last) {
        if (FIXED && lane <= last) top |= magnitude(m);
      });
}

// Both recurrences of a row: segment seg (len points) of lane l of gw, G of them in use; top: OR of
// the band's |R'|.  The band shares its shifts, so a band of W has one exponent.
template <int NW, class A>
__device__ __forceinline__ void row_solve(i64* seg, int len, int l, int G, int gw, int levels, bool full, A ar,
                                          const ScanTab& tab, int gain, unsigned top, unsigned* slots, int& e_lsb,
                                          int& e_top) {
  const int sl = 62 - gain - bit_length_hi(cta_or<NW>(top, slots));
  typename A::State a, b;
  pass_end(ar, seg, 1, len, sl, a, b);
  i64 ea = A::value(a), eb = A::value(b);
  scan_states<false, A>(tab, ea, eb, l, G, gw, levels, full);
  pass_full(ar, seg, 1, len, A::state(ea), A::state(eb));
  const int sl2 = 62 - gain - bit_length_hi(cta_or<NW>(ar.top, slots + NW));
  i64* end = seg + max(len - 1, 0);
  pass_end(ar, end, -1, len, sl2, a, b);
  ea = A::value(a);
  eb = A::value(b);
  scan_states<true, A>(tab, ea, eb, l, G, gw, levels, full);
  pass_full(ar, end, -1, len, A::state(ea), A::state(eb));
  e_lsb = -sl - sl2;
  e_top = e_lsb + bit_length_hi(cta_or<NW>(ar.top, slots + 2 * NW));
}

// Warps that share a sample's FP64 sums (a band out of the scaled range): those of the row class's own
// CTA, so that a member's samples do not depend on the CTA size that its company leads to.
__device__ __forceinline__ int sample_warps(const MemberParams& P) { return P.fx == 1 ? 2 : P.fx == 2 ? 4 : 8; }

// Exponents by which a block's largest |C| may lie below the band's (a band's below the member's) of
// |C| < 2^E: less where the cubic term takes bits from mu.
__device__ __forceinline__ int quiet_line(int E) { return 10 - 3 * max(0, E - 1); }

template <int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) fx_rows_kernel(DevView v, int tile_base) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned wtop[5 * (TH / 32)];
  const Tile tl = v.row_tiles[tile_base + blockIdx.x];
  const MemberParams& P = v.mp[tl.member];
  MemberState* st = v.ms + tl.member;
  load_tab(*reinterpret_cast<ScanTab*>(smem), v.seg[tl.member]);
  after_previous();
  bool sample;
  if (!stencil_prologue(tl, st, P, sample)) return;
  constexpr int NW = TH / 32;
  const int nx = P.nx, ny = P.ny, j0 = tl.start, nr = tl.count, S = P.fx_sx, G = P.fx_gx, gw = P.fx_gwx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ScanTab& tab = *reinterpret_cast<ScanTab*>(smem);
  Band b;
  b.tile = reinterpret_cast<i64*>(smem + sizeof(ScanTab));
  b.pitch = G * (S + 1);
  b.ls = __ffs(S) - 1;
  b.nx = nx;
  b.ns = (nx + 31) >> 5;
  b.nr = nr;
  i64* Es = b.tile + (nr + 4) * b.pitch;
  i64* Em = Es + 2 * b.ns * (nr + 4);
  double* red = reinterpret_cast<double*>(Em + 2 * b.ns * (nr + 2));

  // C rows j0 - 2 .. j0 + nr + 1 (periodic) into the tile
  {
    const i64* Cg = static_cast<const i64*>(v.C) + P.offset;
    for (int s = warp; s < b.ns; s += NW) {
      const int i = min(32 * s + lane, nx - 1);
      i64* col = b.tile + i + (i >> b.ls);
      int j = j0 - 2 < 0 ? j0 - 2 + ny : j0 - 2;
      const i64* src = Cg + (int64_t)j * nx + i;
#pragma unroll 4
      for (int t = 0; t < nr + 4; ++t) {
        copy8(col, src);
        col += b.pitch;
        src += nx;
        if (++j == ny) {
          j = 0;
          src = Cg + i;
        }
      }
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  unsigned top = 0, low = ~0u;  // of the blocks' largest |C|, the largest and the least (high words)
  for (int s = warp; s < b.ns; s += NW) {  // this thread's own copies
    const int i = min(32 * s + lane, nx - 1);
    const int2* col = reinterpret_cast<const int2*>(b.tile + i + (i >> b.ls));
    const bool wide = 32 * s + 16 <= nx;  // a last strip of a few columns may lie along a nodal line
#pragma unroll 2
    for (int t = 0; t < nr + 4; t += 4) {
      const int2* at = col + min(t, nr) * b.pitch;  // the last block may overlap the one before
      unsigned block = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) block = max(block, (unsigned)at[q * b.pitch].y & 0x7fffffffu);
      block = __reduce_max_sync(kAll, block);
      top = max(top, block);
      if (wide) low = min(low, block);
    }
  }
  if (lane == 0) {
    wtop[warp] = top;
    wtop[NW + warp] = low;
  }
  __syncthreads();
  top = __reduce_max_sync(kAll, lane < NW ? wtop[lane] : 0u);
  low = __reduce_min_sync(kAll, lane < NW ? wtop[NW + lane] : ~0u);
  const int emax = (int)(top >> 20);  // biased exponent of the largest |C|
  const bool bad = emax > 1022 + kFxMaxE || emax < 823 || (int)(low >> 20) + quiet_line(emax - 1022) < emax;
  auto cut_bits = [&] { return emax > 1023 ? P.fx_cut[emax - 1024] : 0; };  // (in range)
  // the strips' edge columns
  for (int k = threadIdx.x; k < 2 * b.ns * (nr + 4); k += TH) {
    const int e = k / (nr + 4), t = k - e * (nr + 4);
    const int i = min(16 * (e & ~1) + 31 * (e & 1), nx - 1);
    const i64 c = b.tile[t * b.pitch + i + (i >> b.ls)];
    Es[k] = bad ? c : to_fixed(c, emax);
  }
  __syncthreads();
  int up = 0;  // R' is held times 2^(kmu + up - E)
  if (bad) {
    fp64_tables(tab, v.seg[tl.member]);
    RhsFp rhs{P.fx_tall != 0, P.fx_ratio, P.fx_w0};
    band_rhs<NW, -1>(b, Es, Em, top, emax, MuFp{P.a, P.bx, P.by}, rhs, wtop + 4 * NW);
  } else {
    const int cut = cut_bits(), su = P.fx_su + cut;
    with_shift(max(-62, 2 * (emax - 1022) + 6 - su), [&](auto sh) {  // C^2 vanishes long before -62
      const i64 one = 1ll << (60 - su);
      const FxLimb bx = cut_limb(P.fx_bx, cut), by = cut_limb(P.fx_by, cut);
      auto fixed = [&](auto mu, auto rhs, auto form) {
        band_rhs<NW, decltype(form)::value>(b, Es, Em, top, emax, mu, rhs, wtop + 4 * NW);
        up = rhs.up;
      };
      if (P.fx_square)
        fixed(MuFx<true, decltype(sh)>{bx, by, one, sh}, RhsFx<0>{P.fx_rl, P.fx_er},
              std::integral_constant<int, 0>());
      else if (!P.fx_tall)
        fixed(MuFx<false, decltype(sh)>{bx, by, one, sh}, RhsFx<1>{P.fx_rl, P.fx_er},
              std::integral_constant<int, 1>());
      else
        fixed(MuFx<false, decltype(sh)>{bx, by, one, sh}, RhsFx<2>{P.fx_rl, P.fx_er},
              std::integral_constant<int, 2>());
    });
  }
  if (sample)
    band_partials_field<double>(v, tl, nx, nr, P, v.partials + P.partial_base + tl.index, red, sample_warps(P));

  // rows: gw lanes per row (row_solve starts with a barrier: R' is complete)
  const int l = lane & (gw - 1), row = threadIdx.x / gw, r = min(row, nr - 1);
  const int len = l < G && row < nr ? min(S, nx - l * S) : 0;
  i64* seg = b.tile + r * b.pitch + l * (S + 1);
  const bool full = nx % S == 0;
  int e_lsb, e_top;
  if (bad)
    row_solve<NW>(seg, len, l, G, gw, all_levels(G), full, Fp(P.fx_cx, P.p1x, P.p2x), tab, 0, 0u, wtop + NW, e_lsb, e_top);
  else
    row_solve<NW>(seg, len, l, G, gw, P.fx_lvx, full, Fx(P.fx_cx, 0.0, 0.0), tab, P.fx_gainx, top, wtop + NW, e_lsb, e_top);
  if (row < nr && l == 0) {
    const int eb = bad ? 0 : emax - 1022 - P.fx_kmu + cut_bits() - up;
    v.wexp[P.fx_wexp + j0 + row] = bad ? RowExp{0, (short)kBadRow, (short)(emax - 1022), 0}
                                       : RowExp{(short)(e_lsb + eb), (short)(e_top + eb), (short)(emax - 1022), 0};
  }
  // W to HBM as whole rows (row_solve ends with a barrier)
  i64* Wg = static_cast<i64*>(v.W) + P.offset + (int64_t)j0 * nx;
  for (int q = warp; q < nr; q += NW) {
    const i64* src = b.tile + q * b.pitch;
    i64* dst = Wg + q * nx;
#pragma unroll 4
    for (int i = lane; i < nx; i += 32) dst[i] = src[i + (i >> b.ls)];
  }
}

// Observables of the current fields (ch_observables): the partials of one band.
__global__ void __launch_bounds__(256) fx_observe_kernel(DevView v, int tile_base) {
  __shared__ double red[16];
  const Tile tl = v.row_tiles[tile_base + blockIdx.x];
  const MemberParams& P = v.mp[tl.member];
  band_partials_field<double>(v, tl, P.nx, tl.count, P, v.partials + P.partial_base + tl.index, red, sample_warps(P));
}

// -------------------------------------------------------------------------------------
// Columns
// -------------------------------------------------------------------------------------
// A CTA of 256 threads takes a panel of cw columns (32, 16 or 8), thread = segment tid / cw of S
// rows of column tid % cw, its values in shared memory (value u of thread t at u 256 + t: no bank
// conflicts).  The first pass runs as W arrives, the last one updates C.
constexpr int kColThreads = 256;
constexpr int kXsMax = 32 * 9;  // state exchange: G x (cw + 1), G cw <= 256

template <class A>
__device__ __forceinline__ int col_solve(A& ar, i64* y, int len, const ScanTab& tab, longlong2* xs, unsigned* wtop, int G,
                                         int gw, int levels, bool full, int cw, int gain, typename A::State& a, typename A::State& b) {
  const int seg = threadIdx.x / cw, c = threadIdx.x - seg * cw;
  const int l = threadIdx.x & (gw - 1), sc = threadIdx.x / gw;  // scan: segment l of column sc
  auto exchange = [&](bool rev) {  // end state of this thread's segment in, its start state out
    if (seg < G) xs[seg * (cw + 1) + c] = make_longlong2(A::value(a), A::value(b));
    __syncthreads();
    longlong2* p = xs + min(l, G - 1) * (cw + 1) + min(sc, cw - 1);
    longlong2 e = *p;
    i64 ea = e.x, eb = e.y;
    if (rev)
      scan_states<true, A>(tab, ea, eb, l, G, gw, levels, full);
    else
      scan_states<false, A>(tab, ea, eb, l, G, gw, levels, full);
    e = make_longlong2(ea, eb);
    if (l < G && sc < cw) *p = e;
    __syncthreads();
    e = xs[min(seg, G - 1) * (cw + 1) + c];
    a = A::state(e.x);
    b = A::state(e.y);
  };
  exchange(false);
  pass_full(ar, y, kColThreads, len, a, b);
  // the panel's largest |y| sets the shift before the backward recurrence
  const int sl = 62 - gain - bit_length_hi(cta_or<kColThreads / 32>(ar.top, wtop));
  pass_end(ar, y + max(len - 1, 0) * kColThreads, -kColThreads, len, sl, a, b);
  exchange(true);
  return sl;
}

// The backward pass from its start state and the update C += kap x (y, Cg: the segment's last row),
// 4 rows at a time, the next 4 rows of C in flight.
template <class A, class Conv>
__device__ __forceinline__ void col_update(const A& ar, const i64* y, int len, double* Cg, int nx, double kap, bool cv,
                                           typename A::State a, typename A::State b, Conv conv) {
  double nc[4];
  const double* q = Cg;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (u < len && cv) nc[u] = *q;
    q -= nx;
  }
#pragma unroll 1
  for (int k = len; k > 0; k -= 4) {
    double cc[4];
    i64 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      cc[u] = nc[u];
      if (u < k) v[u] = y[-u * kColThreads];
      if (u + 4 < k && cv) nc[u] = *q;
      q -= nx;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < k) {
        const i64 t = ar.step(a, b, v[u]);
        b = a;
        a = A::state(t);
        if (cv) *Cg = fma(kap, conv(t), cc[u]);
        Cg -= nx;
      }
    y -= 4 * kColThreads;
  }
}

// The scaled forward pass from a zero state over W as its copies arrive, in 4 groups of 8 rows per
// segment.  Rows come in bands of one exponent that start at multiples of 8 (ws: the segment's
// row exponents).
template <class A, class Scaled>
__device__ __forceinline__ void col_first(const A& ar, i64* y, int len, int S, const RowExp* ws,
                                          typename A::State& a, typename A::State& b, const Scaled& scaled) {
  a = A::zero();
  b = A::zero();
#pragma unroll 1
  for (int k = 0; k < S; k += 8) {
    if (k == 0)
      asm volatile("cp.async.wait_group 3;\n" ::: "memory");
    else if (k == 8)
      asm volatile("cp.async.wait_group 2;\n" ::: "memory");
    else if (k == 16)
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    else
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    if (k < len)
      scaled(ws[k], [&](auto sh) {
        i64 w[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k + u < len) w[u] = y[u * kColThreads];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k + u < len) {
            const i64 r = sh(w[u]);
            y[u * kColThreads] = r;
            const i64 t = ar.step(a, b, r);
            b = a;
            a = A::state(t);
          }
      });
    y += 8 * kColThreads;
  }
}

__global__ void __launch_bounds__(kColThreads, 3) fx_cols_kernel(DevView v, int tile_base) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) longlong2 xs[kXsMax];
  __shared__ __align__(16) ScanTab tab;
  __shared__ unsigned wtop[kColThreads / 32];
  const Tile tl = v.colseg_tiles[tile_base + blockIdx.x];
  MemberState* st = v.ms + tl.member;
  load_tab(tab, v.segy[tl.member]);
  after_previous();
  if (!st->active) return;
  const MemberParams& P = v.mp[tl.member];
  const int nx = P.nx, ny = P.ny, G = P.fx_gy, gw = P.fx_gwy, gain = P.fx_gainy, S = P.fx_sy, cw = P.fx_cw;
  const int lane = threadIdx.x & 31;
  const int seg = threadIdx.x / cw, c = threadIdx.x - seg * cw;
  const bool cv = c < tl.count;
  const int len = cv && seg < G ? min(S, ny - seg * S) : 0;  // 0: nothing to do, and no say in the panel's scale
  const int64_t base = (int64_t)min(seg, G - 1) * S * nx + tl.start + (cv ? c : 0);
  i64* y = reinterpret_cast<i64*>(smem) + threadIdx.x;
  double* Cg = static_cast<double*>(v.C) + P.offset + base;
  const RowExp* we = v.wexp + P.fx_wexp;
  const RowExp* ws = we + min(seg, G - 1) * S;
  // All of the panel's W in flight in up to 4 groups of rows of every segment (value u of segment g
  // at u 256 + g cw, so a row piece of the panel is contiguous on both sides), in 16-byte pieces
  // where the rows allow it; C on its way to L2 for the update.
  // the bands' exponents (of every eighth row: bands start at multiples of 8), 4 loads ahead of the copies
  RowExp we4[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) we4[k] = we[min(8 * (lane + 32 * k), ny - 1)];
  {
    i64* Y = reinterpret_cast<i64*>(smem);
    const bool wide = !((nx | tl.count) & 1);
    const int half = wide ? cw >> 1 : cw, cols = wide ? tl.count >> 1 : tl.count;
    const int tc = threadIdx.x % half, tr = threadIdx.x / half;
    // a thread copies column piece tc of rows u0 + (tr & 7) of segments tr / 8, + step, ...
    const int step = kColThreads / half / 8, u = tr & 7, s0 = tr >> 3, E = wide ? 2 : 1;
    const i64* Wm = static_cast<const i64*>(v.W) + P.offset + tl.start + E * tc;
    const int64_t dsrc = (int64_t)step * S * nx;
    for (int u0 = 0; u0 < 32; u0 += 8) {
      if (u0 < S && tc < cols) {
        const i64* src = Wm + (int64_t)(s0 * S + u0 + u) * nx;
        i64* dst = Y + (u0 + u) * kColThreads + s0 * cw + E * tc;
        for (int q = s0, j = s0 * S + u0 + u; q < G && j < ny; q += step, j += step * S) {
          if (wide)
            copy16(dst, src);
          else
            copy8(dst, src);
          src += dsrc;
          dst += step * cw;
        }
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    const char* Cm = static_cast<const char*>(v.C) + 8 * (P.offset + tl.start);
    for (int j = threadIdx.x; j < ny; j += kColThreads) {
      const char* p = Cm + (int64_t)j * nx * 8;
      prefetch_l2(p);
      prefetch_l2(p + 8 * (tl.count - 1));
      if (tl.count > 16) prefetch_l2(p + 128);
    }
  }
  int emax = -32768, Emax = -32768, Emin = 32767;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    emax = max(emax, (int)we4[k].top);
    Emax = max(Emax, (int)we4[k].E);
    Emin = min(Emin, (int)we4[k].E);
  }
  emax = __reduce_max_sync(kAll, emax);
  Emax = __reduce_max_sync(kAll, Emax);
  Emin = __reduce_min_sync(kAll, Emin);
  const bool bad = emax == kBadRow || Emin + quiet_line(Emax) < Emax;
  i64* const ye = y + max(len - 1, 0) * kColThreads;
  double* const Ce = Cg + (int64_t)max(len - 1, 0) * nx;
  if (bad) {
    Fp ar(P.fx_cy, P.p1y, P.p2y);
    double a, b;
    col_first(ar, y, len, S, ws, a, b, [](RowExp e, auto f) {
      if (e.top == kBadRow) {
        f([](i64 w) { return w; });
      } else {
        const double unit = pow2(e.unit);  // above -500: no subnormal
        f([unit](i64 w) { return double_bits(unit * (double)w); });
      }
    });
    fp64_tables(tab, v.segy[tl.member]);
    col_solve(ar, y, len, tab, xs, wtop, G, gw, all_levels(G), ny % S == 0, cw, 0, a, b);
    col_update(ar, ye, len, Ce, nx, P.fx_kappa, cv, a, b, [](i64 t) { return __longlong_as_double(t); });
  } else {
    Fx ar(P.fx_cy, 0.0, 0.0);
    FxLimb a, b;
    const int up = 62 - gain - emax;
    col_first(ar, y, len, S, ws, a, b, [up](RowExp e, auto f) { with_shift(max(-62, min(62, up + (int)e.unit)), f); });
    const int sl = col_solve(ar, y, len, tab, xs, wtop, G, gw, P.fx_lvy, ny % S == 0, cw, gain, a, b);
    col_update(ar, ye, len, Ce, nx, P.fx_kappa * ldexp(1.0, -up - sl), cv, a, b, [](i64 t) { return (double)t; });
  }
  if (tl.index == 0 && threadIdx.x == 0) finalize_sample(v, tl.member, st, P);
}

template <int TH, int MINB>
cudaError_t rows_limit() {
  return cudaFuncSetAttribute(fx_rows_kernel<TH, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
}

}  // namespace

// A step kernel; as a dependent launch up to one CTA per SM (above, CTAs that start in the slots their
// predecessor happens to leave free are spread unevenly: 64 x 128^2 51 us per step with it, 39
// without, 8 x 512^2 76 and 68).
constexpr int kDependentCtas = 152;  // the GPU's SMs

template <class K>
void launch_dependent(K kernel, int grid, int block, size_t smem, cudaStream_t st, const DevView& v, int base, bool ready) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)block, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ready && grid <= kDependentCtas ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, v, base);
}

cudaError_t launch_fx_rows(const DevView& v, const LaunchShape& sh, cudaStream_t st, bool tables_ready) {
  int base = sh.n_row_tiles;
  const int* n = sh.fx_rt;
  const size_t* sm = sh.fx_smem;
  // Classes only set the CTA size (a run's results do not depend on it): where several of the
  // short ones are present they share a launch, since a mix of small runs is bound by its launches
  // (a burst of 24 requests of 64^2 to 256^2 takes 35.2 ms in separate launches, 24.2 ms in one).
  if ((n[0] > 0) + (n[1] > 0) + (n[2] > 0) > 1) {
    const int all = n[0] + n[1] + n[2];
    launch_dependent(fx_rows_kernel<256, 4>, all, 256, max(sm[0], max(sm[1], sm[2])), st, v, base, tables_ready);
    base += all;
    if (n[3] > 0) launch_dependent(fx_rows_kernel<256, 2>, n[3], 256, sm[3], st, v, base, tables_ready);
    return cudaPeekAtLastError();
  }
  // few tiles of one short class (so none of the next): larger CTAs (a sample's sums then take 8 warps)
  if (n[0] + n[1] > 0 && n[0] + n[1] <= kDependentCtas) {
    launch_dependent(fx_rows_kernel<256, 4>, n[0] + n[1], 256, max(sm[0], sm[1]), st, v, base, tables_ready);
    base += n[0] + n[1];
    if (n[3] > 0) launch_dependent(fx_rows_kernel<256, 2>, n[3], 256, sm[3], st, v, base, tables_ready);
    return cudaPeekAtLastError();
  }
  if (n[0] > 0) launch_dependent(fx_rows_kernel<64, 14>, n[0], 64, sm[0], st, v, base, tables_ready);
  base += n[0];
  if (n[1] > 0) launch_dependent(fx_rows_kernel<128, 7>, n[1], 128, sm[1], st, v, base, tables_ready);
  base += n[1];
  if (n[2] > 0) launch_dependent(fx_rows_kernel<256, 4>, n[2], 256, sm[2], st, v, base, tables_ready);
  base += n[2];
  if (n[3] > 0) launch_dependent(fx_rows_kernel<256, 2>, n[3], 256, sm[3], st, v, base, tables_ready);
  return cudaPeekAtLastError();
}

cudaError_t launch_fx_observe(const DevView& v, const LaunchShape& sh, cudaStream_t st) {
  if (sh.fx_tiles > 0) fx_observe_kernel<<<sh.fx_tiles, 256, 0, st>>>(v, sh.n_row_tiles);
  return cudaGetLastError();
}

cudaError_t launch_fx_cols(const DevView& v, const LaunchShape& sh, cudaStream_t st, bool tables_ready) {
  const int base = sh.cst_n[0] + sh.cst_n[1] + sh.cst_n[2] + sh.cst_n[3];
  if (sh.fx_ct > 0) launch_dependent(fx_cols_kernel, sh.fx_ct, kColThreads, sh.fx_cols_smem, st, v, base, tables_ready);
  return cudaPeekAtLastError();
}

size_t fx_rows_smem(int nr, int nx, int S) {
  const int G = (nx + S - 1) / S, ns = (nx + 31) / 32;
  return sizeof(ScanTab) + 8 * ((size_t)(nr + 4) * G * (S + 1) + (size_t)2 * ns * (2 * nr + 6) + 32);
}

size_t fx_cols_smem(int S) { return (size_t)S * kColThreads * 8; }

cudaError_t set_fx_smem_limits() {
  cudaError_t e;
  if ((e = rows_limit<64, 14>()) != cudaSuccess || (e = rows_limit<128, 7>()) != cudaSuccess ||
      (e = rows_limit<256, 4>()) != cudaSuccess || (e = rows_limit<256, 2>()) != cudaSuccess)
    return e;
  return cudaFuncSetAttribute(fx_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
}

}  // namespace chk
