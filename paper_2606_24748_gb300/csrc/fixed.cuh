// FP64 block products on two pipes at once: some rows of each block by FP64
// FMA, the others in block-scaled fixed point on the integer pipes.
//
// A GB300 SM retires two FP64 FMA per clock but some 60 integer operations and
// 13 wide (32 x 32 + 64 bit) integer multiply-adds (measured), so a product
// that takes every row through the FP64 pipe is bound by it below the rate of
// HBM.  A fixed-point product takes three wide multiply-adds and no FP64
// operation:
//  - a block's values are cut, each with its sign, into two 28-bit limbs on the
//    scale of the block's largest value; x's entries likewise on a scale that
//    gives every product of a row one common exponent, the largest seen so far
//    (when a larger one comes the row's sums are shifted down to it);
//  - the limb products high x high and high x low + low x high are summed in
//    two 64-bit integers; low x low (2^-56 of the largest product) is dropped.
// Integer sums do not round, so a row's error is that of the cut operands, at
// most 2^-55 of the largest |block| |x| of the row per product; an FP64 sum
// rounds at 2^-53 of each partial sum.  Measured against 80-bit sums on a
// 27-block row with values over two decades: 1.6e-16 in the fixed-point rows,
// 3.0e-16 by FP64 FMA.  Every cut is symmetric in the sign and moves with the
// exponent, so x -> -x and x -> 2^k x give exactly -y and 2^k y.
// Rows with values that the scales do not cover (Inf, NaN, or a largest entry
// beyond 2^+-767) are done again by FP64 FMA alone.
#pragma once

#include <cstdint>

namespace bamg {

// Rows of a block that stay on the FP64 pipe.  With one of three there, the two
// pipes are busy for about as long (3x3 products, 65^3 nodes, 27 blocks per
// row: 141.8 us with three, 102 with one, 116 with none).
template <int BR>
constexpr int fx_fma_rows() { return BR / 3; }

__device__ __forceinline__ unsigned fx_shr(unsigned a, unsigned s) {  // 0 for s > 31
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(s));
  return r;
}
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long a, unsigned s) {  // 0 for s > 63
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}

struct FxBits {  // a double's words
  unsigned hi, lo;
};
__device__ __forceinline__ FxBits fx_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return {(unsigned)(b >> 32), (unsigned)b};
}

// (h 2^28 + l) 2^(top - 1078) is v cut toward zero, for a biased exponent
// top >= v's; 0 when top is 60 or more above it (so for v = 0, top >= 60).
__device__ __forceinline__ void fx_limbs(FxBits v, int top, int& h, int& l) {
  const unsigned s = (unsigned)(top - (int)((v.hi & 0x7fffffffu) >> 20));
  const unsigned m = (__funnelshift_l(v.lo, v.hi, 7) & 0x07ffffffu) | 0x08000000u;
  const unsigned long long w = ((unsigned long long)m << 32) | (v.lo << 7);
  const int sign = ((int)v.hi >> 31) | 1;
  h = (int)fx_shr(m, s) * sign;
  l = (int)((unsigned)fx_shr(w, s) >> 4) * sign;
}

// v / 2^d toward zero, so that -v gives exactly the opposite.
__device__ __forceinline__ long long fx_down(long long v, int d) {
  return (v + ((v >> 63) & ((1LL << d) - 1))) >> d;
}

// Smallest biased exponent a scale is taken from: zeros, and values this far
// down, then cut to 0 on it.
constexpr int kFxMinExp = 64;

// A block's values cut to limbs: rows fx_fma_rows() .. BR - 1.
template <int BR, int BC>
struct FxBlock {
  static constexpr int R0 = fx_fma_rows<BR>(), N = (BR - R0) * BC;
  int h[N], l[N];
  unsigned top;  // largest high word without sign (0: all values zero)
  int exp;       // exponent of the scale
  __device__ __forceinline__ void cut(const double (&v)[BR * BC]) {
    top = 0;
#pragma unroll
    for (int e = 0; e < N; ++e) top = max(top, fx_bits(v[R0 * BC + e]).hi & 0x7fffffffu);
    if (top == 0) {  // zeros, or subnormals below the high word
      unsigned low = 0;
#pragma unroll
      for (int e = 0; e < N; ++e) low |= fx_bits(v[R0 * BC + e]).lo;
      top = low != 0;
    }
    exp = max((int)(top >> 20), kFxMinExp);
#pragma unroll
    for (int e = 0; e < N; ++e) fx_limbs(fx_bits(v[R0 * BC + e]), exp, h[e], l[e]);
  }
};

// A block as it is kept where many threads read it: the FP64 rows, the others'
// limbs and the largest high word, in 16-byte words.
template <int BR, int BC>
struct FxCut {
  using Block = FxBlock<BR, BC>;
  static constexpr int F = Block::R0 * BC, N = Block::N;
  static constexpr int kWords = (2 * F + 2 * N + 1 + 3) / 4;  // 16-byte words
  __device__ __forceinline__ static void pack(const double (&v)[BR * BC], uint4 (&out)[kWords]) {
    unsigned w[4 * kWords];
#pragma unroll
    for (int e = 0; e < F; ++e) {
      w[2 * e] = fx_bits(v[e]).lo;
      w[2 * e + 1] = fx_bits(v[e]).hi;
    }
    Block a;
    a.cut(v);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      w[2 * (F + e)] = (unsigned)a.h[e];
      w[2 * (F + e) + 1] = (unsigned)a.l[e];
    }
    w[2 * (F + N)] = a.top;
#pragma unroll
    for (int k = 2 * (F + N) + 1; k < 4 * kWords; ++k) w[k] = 0;
#pragma unroll
    for (int k = 0; k < kWords; ++k) out[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
  }
  __device__ __forceinline__ static void load(const uint4* __restrict__ p, double (&v)[F], Block& a) {
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
    for (int e = 0; e < F; ++e) v[e] = __hiloint2double((int)w[2 * e + 1], (int)w[2 * e]);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      a.h[e] = (int)w[2 * (F + e)];
      a.l[e] = (int)w[2 * (F + e) + 1];
    }
    a.top = w[2 * (F + N)];
    a.exp = max((int)(a.top >> 20), kFxMinExp);
  }
};

// Sums of one row (all its components) over its blocks for one vector.
template <int BR, int BC>
struct FxRow {
  static constexpr int R0 = fx_fma_rows<BR>(), NI = BR - R0;
  // Limb products are below 2^56, so `mid` (two per term) holds 60 terms
  // before it is carried into `hh`, and `hh` 120 before it goes to `acc`.
  static constexpr int kCarry = 60 / BC, kFlush = 2 * kCarry;
  double acc[BR];
  long long hh[NI], mid[NI];
  int E;              // hh and mid are on the scale 2^(E - 2156 + 56) and 2^(E - 2156 + 28)
  unsigned amax, xmax;  // largest high words of the blocks' and of x's values

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int r = 0; r < BR; ++r) acc[r] = 0.0;
#pragma unroll
    for (int r = 0; r < NI; ++r) hh[r] = mid[r] = 0;
    E = 0;
    amax = xmax = 0;
  }
  // v: the block's values, at least its first R0 rows
  template <int M>
  __device__ __forceinline__ void add(const double (&v)[M], const FxBlock<BR, BC>& a, const double (&x)[BC]) {
    static_assert(M >= R0 * BC, "the FP64 rows come first");
#pragma unroll
    for (int r = 0; r < R0; ++r)
#pragma unroll
      for (int q = 0; q < BC; ++q) acc[r] = fma(v[r * BC + q], x[q], acc[r]);
    unsigned mx = 0;
#pragma unroll
    for (int q = 0; q < BC; ++q) mx = max(mx, fx_bits(x[q]).hi & 0x7fffffffu);
    if (mx == 0) {
      unsigned low = 0;
#pragma unroll
      for (int q = 0; q < BC; ++q) low |= fx_bits(x[q]).lo;
      mx = low != 0;
    }
    amax = max(amax, a.top);
    xmax = max(xmax, mx);
    const int need = (a.top != 0 && mx != 0) ? a.exp + max((int)(mx >> 20), kFxMinExp) : 0;
    if (need > E) {
      const int d = min(need - E, 62);
      E = need;
#pragma unroll
      for (int r = 0; r < NI; ++r) {
        hh[r] = fx_down(hh[r], d);
        mid[r] = fx_down(mid[r], d);
      }
    }
    const int top = mx != 0 ? E - a.exp : 2200;
#pragma unroll
    for (int q = 0; q < BC; ++q) {
      int h, l;
      fx_limbs(fx_bits(x[q]), top, h, l);
#pragma unroll
      for (int r = 0; r < NI; ++r) {
        hh[r] += (long long)a.h[r * BC + q] * h;
        mid[r] += (long long)a.h[r * BC + q] * l;
        mid[r] += (long long)a.l[r * BC + q] * h;
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
  // the sign; needs valid().
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
    // the sum is m 2^(e - z) 2^(E - 2128)
    const unsigned long long mant = (m >> 11) + ((m >> 10) & 1);
    const unsigned long long bits = ((unsigned long long)(E - 2128 + 63 + e - z + 1022) << 52) + mant;
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0)));
  }
  __device__ __forceinline__ void flush() {  // after carry()
    if (!covers()) amax = 0x7fffffffu;  // these sums are lost: the row is not valid
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      if (covers()) acc[R0 + r] += value(r);
      hh[r] = mid[r] = 0;
    }
  }
  // The row's sums; flushed: whether flush() has been called before.
  __device__ __forceinline__ bool finish(double (&out)[BR], bool flushed) {  // false: not valid
    carry();
    const bool ok = valid();
#pragma unroll
    for (int r = 0; r < R0; ++r) out[r] = acc[r];
#pragma unroll
    for (int r = 0; r < NI; ++r) {
      const double v = ok ? value(r) : 0.0;
      out[R0 + r] = flushed ? acc[R0 + r] + v : v;
    }
    return ok;
  }
  // The exponent gives normal doubles (E = 0: no product yet).
  __device__ __forceinline__ bool covers() const { return E == 0 || (unsigned)(E - 1106) < 1950u; }
  // Whether the sums are the row's products; otherwise these have to be formed by FP64 FMA.
  __device__ __forceinline__ bool valid() const {
    auto covered = [](unsigned m) { return m == 0 || m - 0x10000000u < 0x60000000u; };
    return covered(amax) && covered(xmax) && covers();
  }
};

// One row's sums over a stream of blocks.
template <int BR, int BC>
struct FxSum {
  FxRow<BR, BC> row;
  int left, carries;
  __device__ __forceinline__ void init() {
    row.init();
    left = FxRow<BR, BC>::kCarry;
    carries = 0;
  }
  __device__ __forceinline__ void add(const double (&v)[BR * BC], const double (&x)[BC]) {
    FxBlock<BR, BC> a;
    a.cut(v);
    add(v, a, x);
  }
  template <int M>
  __device__ __forceinline__ void add(const double (&v)[M], const FxBlock<BR, BC>& a, const double (&x)[BC]) {
    row.add(v, a, x);
    if (--left == 0) {
      left = FxRow<BR, BC>::kCarry;
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
