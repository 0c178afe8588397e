// Fixed-point product sums in place of FP64 ones (sm_103a).  GB300 issues one FP64 FMA per 64 clocks and SM
// partition (measured: 18.7 clocks per warp instruction and SM), but two 32 x 32 + 64 bit integer
// multiply-adds per clock and SM (measured 1.92), so a product sum in exact integers costs a ninth of the FP64 one.
// H and the real and the imaginary part of a tile are scaled by a power of two each (the largest element's)
// and cut to 2 LB - 1 bits, kept as two signed limbs of LB bits; sums of limb products are exact in 64 bits (LB = 29
// for up to 32 terms, 28 for up to 128), and the total, again below 2^62, is rounded once to FP64.  The idea is
// the splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012), with integers in place of short
// floating-point slices.
// What is cut off an element is below 2^(1 - 2 LB) of the largest one's binade (2^-57 or 2^-55; FP64 itself rounds
// that element at 2^-54), and no sum rounds on the way.  Measured against 64-bit torch (relative 2-norm): four steps of
// 1,344,904 ADOs of 14 x 14 from a site 1.7e-16 and 1.9e-16 on two inputs, with FP64 FMAs 2.1e-16 and 1.1e-16; 400 steps of 3060 ADOs of 7 x 7 1.6e-15
// both.  Where elements of very different size share a scale and the small ones matter (general runs: Re and Im of
// the two-exciton space under a pulse share it, populations beside weak coherences), the longer form below keeps 28
// more bits of H, the tile and the sum: with the short one the error of ten steps grew from 1.2e-16 to 1.2e-15.
// A tile with Inf, NaN or exponents near the ends of the range takes the FMA chain.
#pragma once
#include <cuda_runtime.h>

namespace heom {

// |x| as an ordered integer (0 only for zero): the high word, its last bit set if only the low word is not zero.
__device__ __forceinline__ int fx_key(double x) {
  const int h = __double2hiint(x) & 0x7fffffff;
  return h | (h == 0 && __double2loint(x) != 0);
}
__device__ __forceinline__ int fx_exp(int key) { return max(key >> 20, 1); }

// x as limbs of lb bits, |x| = (hi 2^lb + lo) 2^(e - 1022 - (2 lb - 1)) with the sign on both limbs, for
// |x| < 2^(e - 1022), cut below the last bit; |lo| <= 2^(lb - 1), |hi| <= 2^(lb - 1).  32-bit funnel shifts: about 25
// instructions (with 64-bit shifts by a variable and rounding to nearest it took about 90).
__device__ __forceinline__ int2 fx_split(double x, int e, int lb) {
  const int h = __double2hiint(x), l = __double2loint(x);
  const int ex = (h >> 20) & 0x7ff;
  unsigned mh = __funnelshift_l((unsigned)l, (unsigned)h, 11) | 0x80000000u, ml = (unsigned)l << 11;  // 1.fraction
  int n = e + 65 - 2 * lb - ex;  // shift right by n >= 7
  if (n >= 32) {
    ml = mh;
    mh = 0;
    n -= 32;
  }
  const unsigned xl = __funnelshift_rc(ml, mh, n), xh = __funnelshift_rc(mh, 0u, n);
  int lo = (int)(xl << (32 - lb)) >> (32 - lb);
  int hi = (int)__funnelshift_r(xl, xh, lb) + (int)((unsigned)lo >> 31);
  if (ex == 0) hi = lo = 0;  // zero; subnormals are below the last bit wherever fx_ok holds
  const int sg = h >> 31;
  return make_int2((hi ^ sg) - sg, (lo ^ sg) - sg);
}

// k 2^p rounded to nearest (|k| < 2^62); the caller keeps the result in FP64's normal range.
__device__ __forceinline__ double fx_double(long long k, int p) {
  const int sg = (int)(k >> 63);
  unsigned long long u = (unsigned long long)((k ^ sg) - sg);
  const int lz = __clzll((long long)u);
  u <<= (lz & 63);
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1);  // the carry of all ones moves into the exponent
  unsigned long long b = ((unsigned long long)(unsigned)(1085 - lz + p) << 52) + m;
  if (u == 0) b = 0;
  return __hiloint2double((int)(b >> 32) | (sg & (int)0x80000000), (int)b);
}

// The same by two FP64 additions, where that pipe has room: the words of k as the low bits of 2^84 and 2^52 (scaled by
// 2^p), the first addition exact.  |k| < 2^62, result and scales in the normal range.
__device__ __forceinline__ double fx_double_add(long long k, int p) {
  const int e = p << 20;
  const double a = __hiloint2double(0x45300000 + e, (int)(k >> 32) ^ (int)0x80000000);  // 2^84 + (hi + 2^31) 2^32
  const double b = __hiloint2double(0x43300000 + e, (int)k);                             // 2^52 + lo
  const double c = __hiloint2double(0x45300000 + e, (int)0x80100000);                    // 2^84 + 2^63 + 2^52
  return (a - c) + b;
}

// acc + a b in one integer multiply-add.  (Written as acc += (long long)a * b the compiler widened the operands first
// and took about seven instructions for each product.)
__device__ __forceinline__ void fx_mad(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// a product sum in parts: hi hi, the two cross sums, lo lo
struct FxSum {
  long long hh, x, y, ll;
  __device__ __forceinline__ FxSum() : hh(0), x(0), y(0), ll(0) {}
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    fx_mad(hh, ah, bh);
    fx_mad(x, ah, bl);
    fx_mad(y, al, bh);
    fx_mad(ll, al, bl);
  }
  __device__ __forceinline__ long long total(int lb) const {  // in units of hi hi, rounded
    return hh + ((x + y + (ll >> lb) + (1ll << (lb - 1))) >> lb);
  }
};

// ---- the longer form (general runs): three limbs of 28 bits, the sum kept to 90 bits ------------------------

constexpr int kFxLong = 28;

// As fx_split with lb = kFxLong, and the next 28 bits in `rest`, balanced too (|rest| <= 2^27): exact for elements down to
// 2^-30 of the largest.
__device__ __forceinline__ int2 fx_split3(double x, int e, int &rest) {
  const int h = __double2hiint(x), l = __double2loint(x);
  const int ex = (h >> 20) & 0x7ff;
  unsigned mh = __funnelshift_l((unsigned)l, (unsigned)h, 11) | 0x80000000u, ml = (unsigned)l << 11, mz = 0;
  int n = e + 65 - 2 * kFxLong - ex;  // >= 9
  if (n >= 32) {
    mz = ml;
    ml = mh;
    mh = 0;
    n -= 32;
  }
  if (n >= 32) {
    mz = ml;
    ml = 0;
    n -= 32;
  }
  const unsigned xl = __funnelshift_rc(ml, mh, n), xh = __funnelshift_rc(mh, 0u, n), xz = __funnelshift_rc(mz, ml, n);
  const int up = (int)(xz >> 31);  // the upper half of the third limb counts as one more of the second
  int lo = (int)(xl << (32 - kFxLong)) >> (32 - kFxLong);
  int hi = (int)__funnelshift_r(xl, xh, kFxLong) + (int)((unsigned)lo >> 31);
  int rs = (int)(xz >> 4) - (up << kFxLong);
  lo += up;
  if (ex == 0) hi = lo = rs = 0;
  const int sg = h >> 31;
  rest = (rs ^ sg) - sg;
  return make_int2((hi ^ sg) - sg, (lo ^ sg) - sg);
}

// Sums of up to 128 products of three-limb numbers: hi hi, the two cross sums, and the three of the next weight (at
// most 128 * 3 * 2^54 < 2^63); what is left out is below 2^-82 of the largest product.
struct FxLong {
  long long hh, x, y, ll;
  __device__ __forceinline__ FxLong() : hh(0), x(0), y(0), ll(0) {}
  __device__ __forceinline__ void add(int ah, int al, int ar, int bh, int bl, int br) {
    fx_mad(hh, ah, bh);
    fx_mad(x, ah, bl);
    fx_mad(y, al, bh);
    fx_mad(ll, al, bl);
    fx_mad(ll, ah, br);
    fx_mad(ll, ar, bh);
  }
  // the sum times 2^p in FP64 (p counts units of the cross sums): hh 2^28 + x + y + ll 2^-28 in 128 bits, normalised
  __device__ __forceinline__ double value(int p) const {
    const long long t = x + y + (ll >> kFxLong);
    unsigned long long lo = (unsigned long long)hh << kFxLong;
    long long hi = hh >> (64 - kFxLong);
    const unsigned long long s = lo + (unsigned long long)t;
    hi += (t >> 63) + (s < lo ? 1 : 0);
    lo = s;
    const bool neg = hi < 0;
    if (neg) {
      lo = 0ull - lo;
      hi = ~hi + (lo == 0 ? 1 : 0);
    }
    const int l1 = __clzll(hi);
    unsigned long long u;
    if (hi != 0) {
      u = (unsigned long long)hi << l1 | lo >> (64 - l1);  // hi < 2^40: l1 >= 24
      p += 64 - l1;
    } else {
      const int l2 = __clzll((long long)lo);
      u = lo << (l2 & 63);
      p -= l2;
    }
    const unsigned long long m = (u >> 11) + ((u >> 10) & 1);
    unsigned long long b = ((unsigned long long)(unsigned)(1085 + p) << 52) + m;
    if (u == 0) b = 0;
    return __hiloint2double((int)(b >> 32) | (neg ? (int)0x80000000 : 0), (int)b);
  }
};

// Limb bits: sums of 2 n (real H) or 4 n products stay below 2^63.
__device__ __forceinline__ int fx_bits(int n, bool cplx) { return !cplx && n <= 16 ? 29 : 28; }

// Whether the fixed-point commutator of a tile with this key stays in FP64's normal range (or is exactly zero).
__device__ __forceinline__ bool fx_ok(int hkey, int key) {
  const int e = (hkey >> 20) + (key >> 20);
  return hkey < 0x7ff00000 && key < 0x7ff00000 && (hkey == 0 || key == 0 || (e >= 1120 && e <= 3000));
}

}  // namespace heom
