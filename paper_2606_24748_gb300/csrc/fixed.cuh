// FP64 block products on two pipes at once: some products of each block by FP64
// FMA, the others in fixed point on the integer pipes.
//
// A GB300 SM retires two FP64 FMA per clock but some 60 integer operations and
// 13 wide (32 x 32 + 64 bit) integer multiply-adds (measured), so a product
// that takes every entry through the FP64 pipe is bound by it below the rate of
// HBM.  A fixed-point product takes three wide multiply-adds and no FP64
// operation:
//  - every scalar row has a scale of its own, the exponent sum of its largest
//    product |a| |x| so far (when a larger one comes its sums are shifted down);
//  - a's 53 bits stand in two 28-bit limbs as they are; x's are shifted down by
//    what the product's exponent sum lacks to the row's scale, and cut to 56
//    bits below it;
//  - the limb products high x high and high x low + low x high are summed in
//    two 64-bit integers; low x low is dropped.
// With 2^E the scale, some product of the row is 2^E or larger.  A product loses
// at most 2^(E-54) by the cut of x and 2^(E-54) by the dropped limb product, the
// shifts of the sums lose at most 2^(E-53) together, and integer sums do not
// round: n products of a scalar row are off by at most (n + 1) 2^-53 of the
// largest |a| |x| among them, and by one rounding to a double.  FP64 FMA may be
// off by n 2^-53 of the sum of |a| |x|, which is no less, so values of unlike
// size in a block or in x cost no more bits here than there.  Measured against
// 113-bit sums, root mean square of error over sum of |a| |x|, rows of 1 to 90
// 3x3 blocks: 3.3e-17 here (five of nine products in fixed point) and 5.2e-17
// by FP64 FMA; with rows, columns or entries over 24 decades 3.5e-17 to 1.5e-16
// and 5.2e-17 to 2.1e-16.  (One scale for the rows of a block, and one for x's
// entries, would take fewer operations, but lose the small rows and entries of a
// block beside large ones.)  Cuts are symmetric in the sign and move with the
// exponent, so x -> -x and x -> 2^k x give exactly -y and 2^k y.
// Rows with subnormals, Inf or NaN among their operands, or with a scale whose
// sums may not be normal doubles, are done again by FP64 FMA alone.
#pragma once

#include <cstdint>

namespace bamg {

// Products of a block (row-major) that stay on the FP64 pipe; the last row of
// these may be divided.  Four of nine with one lane per row: at 64^3 with three,
// four, five, six of nine y = A x takes 95, 96, 98, 99 us, the fused Chebyshev
// step 108, 106, 106, 110 and the CG product 133 (spills), 109, 107, 109; 16
// vectors at 48^3 442, 447, 474, 518.  With six the FP64 pipe is 0.91 busy where
// products follow one another.  Six of nine for several lanes per row, which have
// few blocks each, so that only one of three rows has fixed-point sums to shift
// and convert (24^3, fine Chebyshev step 16.7 us, 19.2 with five).
template <int BR, int BC>
constexpr int fx_fma_products(int lanes) { return BR * BC * (lanes == 1 ? 4 : 6) / 9; }

// Exponents are biased, less one.  A zero's is so far below all others that a
// product with it is shifted out at every scale and does not raise one (kFxNone:
// no product yet); that of a subnormal, Inf or NaN so far above that any product
// with it, even by zero, takes the scale out of the range that covers() accepts.
constexpr int kFxZero = -5000, kFxNone = -2500, kFxOdd = 10000;

// A double taken apart.
struct FxParts {
  int sign;     // 1 or -1
  int e;        // exponent
  unsigned m;   // leading 28 bits
  unsigned lo;  // the other 25, from the top of the word
};
__device__ __forceinline__ FxParts fx_parts(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned t = (hi - 0x00100000u) & 0x7fffffffu;
  const bool special = t >= 0x7fe00000u;  // exponent 0 or 2047
  const int e = special ? (((hi & 0x7fffffffu) | lo) != 0 ? kFxOdd : kFxZero) : (int)(t >> 20);
  return {((int)hi >> 31) | 1, e, (__funnelshift_l(lo, hi, 7) & 0x07ffffffu) | 0x08000000u, lo << 7};
}
// The same as limbs with the sign: (h 2^28 + l) 2^(e - 1077).
struct FxLimbs {
  int h, l, e;
};
__device__ __forceinline__ FxLimbs fx_limbs(double v) {
  const FxParts p = fx_parts(v);
  return {(int)p.m * p.sign, (int)(p.lo >> 4) * p.sign, p.e};
}

// v / 2^d toward zero, so that -v gives exactly the opposite.
__device__ __forceinline__ long long fx_down(long long v, int d) {
  return (v + ((v >> 63) & ((1LL << d) - 1))) >> d;
}

// The entries of a block whose products are formed in fixed point: the last
// BR * BC - F0.
template <int BR, int BC, int F0>
struct FxBlock {
  static constexpr int N = BR * BC - F0;
  FxLimbs a[N];
  // v(r, q): the block's entries
  template <typename F>
  __device__ __forceinline__ void take(F v) {
#pragma unroll
    for (int e = 0; e < N; ++e) a[e] = fx_limbs(v((F0 + e) / BC, (F0 + e) % BC));
  }
};

// A block as it is kept where many threads read it: its first F0 values, the
// others' limbs, and their exponents as 16-bit numbers, in 16-byte words.
template <int BR, int BC, int F0>
struct FxCut {
  using Block = FxBlock<BR, BC, F0>;
  static constexpr int N = Block::N;
  static constexpr int kWords = (2 * F0 + 2 * N + (N + 1) / 2 + 3) / 4;  // 16-byte words
  // v(r, q): the block's entries
  template <typename F>
  __device__ __forceinline__ static void pack(F v, uint4 (&out)[kWords]) {
    unsigned w[4 * kWords];
#pragma unroll
    for (int k = 0; k < 4 * kWords; ++k) w[k] = 0;
#pragma unroll
    for (int e = 0; e < F0; ++e) {
      w[2 * e] = (unsigned)__double2loint(v(e / BC, e % BC));
      w[2 * e + 1] = (unsigned)__double2hiint(v(e / BC, e % BC));
    }
    Block b;
    b.take(v);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      w[2 * (F0 + e)] = (unsigned)b.a[e].h;
      w[2 * (F0 + e) + 1] = (unsigned)b.a[e].l;
      w[2 * (F0 + N) + e / 2] |= ((unsigned)b.a[e].e & 0xffffu) << (e % 2 * 16);
    }
#pragma unroll
    for (int k = 0; k < kWords; ++k) out[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
  }
  __device__ __forceinline__ static void load(const uint4* __restrict__ p, double (&v)[F0], Block& b) {
    unsigned w[4 * kWords];
#pragma unroll
    for (int k = 0; k < kWords; ++k) {
      const uint4 q = __ldg(p + k);
      w[4 * k] = q.x;
      w[4 * k + 1] = q.y;
      w[4 * k + 2] = q.z;
      w[4 * k + 3] = q.w;
    }
#pragma unroll
    for (int e = 0; e < F0; ++e) v[e] = __hiloint2double((int)w[2 * e + 1], (int)w[2 * e]);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const unsigned x = w[2 * (F0 + N) + e / 2];
      b.a[e] = {(int)w[2 * (F0 + e)], (int)w[2 * (F0 + e) + 1], e % 2 ? (int)x >> 16 : (int)(short)(x & 0xffffu)};
    }
  }
};

// Sums of one row (all its components) over its blocks for one vector.
template <int BR, int BC, int F0>
struct FxRow {
  // rows R0 .. BR - 1 have products in fixed point, the first of them perhaps only some
  static constexpr int R0 = F0 / BC, NI = BR - R0;
  // Limb products are below 2^56, so `mid` (two per term) holds 60 terms
  // before it is carried into `hh`, and `hh` 120 before it goes to `acc`.
  static constexpr int kCarry = 60 / BC;
  double acc[BR];
  long long hh[NI], mid[NI];
  int E[NI];  // hh and mid are on the scale 2^(E - 2154 + 56) and 2^(E - 2154 + 28)

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int r = 0; r < BR; ++r) acc[r] = 0.0;
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      hh[r] = mid[r] = 0;
      E[r] = kFxNone;
    }
  }
  // v(r, q): the block's entries
  template <typename F>
  __device__ __forceinline__ void add(F v, const FxBlock<BR, BC, F0>& a, const double (&x)[BC]) {
#pragma unroll
    for (int e = 0; e < F0; ++e) acc[e / BC] = fma(v(e / BC, e % BC), x[e % BC], acc[e / BC]);
    FxParts xn[BC];
#pragma unroll
    for (int q = 0; q < BC; ++q) xn[q] = fx_parts(x[q]);
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      const int q0 = r == 0 ? F0 - R0 * BC : 0, first = (R0 + r) * BC - F0;
      int top = E[r];
#pragma unroll
      for (int q = q0; q < BC; ++q) top = __viaddmax_s32(a.a[first + q].e, xn[q].e, top);
      if (top > E[r]) {
        const int d = min(top - E[r], 62);
        E[r] = top;
        hh[r] = fx_down(hh[r], d);
        mid[r] = fx_down(mid[r], d);
      }
#pragma unroll
      for (int q = q0; q < BC; ++q) {
        const FxLimbs& p = a.a[first + q];
        const int s = min(top - p.e - xn[q].e, 63);  // 60 and more: nothing is left
        const unsigned long long w = (((unsigned long long)xn[q].m << 32) | xn[q].lo) >> s;
        const int h = (int)(w >> 32) * xn[q].sign, l = (int)((unsigned)w >> 4) * xn[q].sign;
        hh[r] += (long long)p.h * h;
        mid[r] += (long long)p.h * l;
        mid[r] += (long long)p.l * h;
      }
    }
  }
  __device__ __forceinline__ void carry() {
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      const long long up = fx_down(mid[r], 28);
      hh[r] += up;
      mid[r] -= up << 28;
    }
  }
  // The sums as doubles, rounded to nearest, by integer operations: an FP64
  // conversion or add holds the SM sub-partition for 64 cycles, and a row of
  // four blocks would spend as many of them here as on its products.  Exact in
  // the sign; needs covers().
  __device__ __forceinline__ double value(int r) const {
    const unsigned long long low = ((unsigned long long)hh[r] << 28) + (unsigned long long)mid[r];
    long long high = (hh[r] >> 36) + (mid[r] >> 63) + (low < (unsigned long long)mid[r] ? 1 : 0);
    unsigned long long lo = low;
    const bool neg = high < 0;
    if (neg) {
      lo = 0 - lo;
      high = ~high + (lo == 0);
    }
    unsigned long long m = (unsigned long long)high;
    int e = 64;
    if (m == 0) {
      m = lo;
      lo = 0;
      e = 0;
    }
    if (m == 0) return 0.0;
    const int z = __clzll((long long)m);
    m = z ? (m << z) | (lo >> (64 - z)) : m;
    // the sum is m 2^(e - z) 2^(E - 2126)
    const unsigned long long mant = (m >> 11) + ((m >> 10) & 1);
    const unsigned long long bits = ((unsigned long long)(E[r] - 2126 + 63 + e - z + 1022) << 52) + mant;
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0)));
  }
  __device__ __forceinline__ void flush() {  // after carry()
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      if (covers(r)) acc[R0 + r] += value(r);
      else E[r] = 2 * kFxOdd;  // these sums are lost: the row is not valid
      hh[r] = mid[r] = 0;
    }
  }
  // The row's sums; flushed: whether flush() has been called before.
  __device__ __forceinline__ bool finish(double (&out)[BR], bool flushed) {  // false: not valid
    carry();
    bool ok = true;
#pragma unroll
    for (int r = 0; r < NI; ++r) ok = ok && covers(r);
#pragma unroll
    for (int r = 0; r < R0; ++r) out[r] = acc[r];
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      const double v = ok ? value(r) : 0.0;
      out[R0 + r] = flushed || (R0 + r) * BC < F0 ? acc[R0 + r] + v : v;
    }
    return ok;
  }
  // The scale gives normal doubles (kFxNone: all products are zero).
  __device__ __forceinline__ bool covers(int r) const { return E[r] == kFxNone || (unsigned)(E[r] - 1104) < 1950u; }
};

// One row's sums over a stream of blocks.
template <int BR, int BC, int F0>
struct FxSum {
  using Row = FxRow<BR, BC, F0>;
  Row row;
  int left, carries;
  __device__ __forceinline__ void init() {
    row.init();
    left = Row::kCarry;
    carries = 0;
  }
  // v(r, q): the block's entries
  template <typename F>
  __device__ __forceinline__ void add(F v, const double (&x)[BC]) {
    FxBlock<BR, BC, F0> a;
    a.take(v);
    add(v, a, x);
  }
  template <typename F>
  __device__ __forceinline__ void add(F v, const FxBlock<BR, BC, F0>& a, const double (&x)[BC]) {
    row.add(v, a, x);
    if (--left == 0) {
      left = Row::kCarry;
      row.carry();
      if ((++carries & 1) == 0) row.flush();
    }
  }
  // False: the values are not covered, and the sums have to be formed by FP64 FMA.
  __device__ __forceinline__ bool finish(double (&out)[BR]) {
    return row.finish(out, carries >= 2);
  }
};

}  // namespace bamg
