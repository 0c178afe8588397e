// Fixed-point product sums in place of FP64 ones (sm_103a).  GB300 issues one FP64 FMA per 64 clocks and SM
// partition (measured: 18.7 clocks per warp instruction and SM), but two 32 x 32 + 64 bit integer
// multiply-adds per clock and SM (measured 1.92), so a product of six limb products costs a sixth of the FP64 FMA.
// H and the real and the imaginary part of a tile (of a column in stage_col.cuh) are scaled by a power of two each (the
// largest element's) and kept as three signed limbs of 28 bits, cut below 2^-83 of the scale; the six limb products of
// weight 2^-56 and more are summed exactly in 64 bits (up to 128 terms), put together in 90 bits and rounded to FP64 at
// the end.  The idea is the splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012), with integers in
// place of short floating-point slices.
// Precision: elements down to 2^-30 of the largest are exact, no sum rounds on the way, and what is cut stays below a
// few units of 2^-82 of the largest product -- but it is an absolute error, where an FP64 chain's is relative to the terms of its own
// sum.  So a sum below 2^-28 of the largest product, where that chain is the more precise, is taken from the chain
// (fx_weak).  Error of a commutator element in units of 2^-53 of the sum of its terms' magnitudes, states of 7, 10 and 14
// sites after 0 to 40 steps: at most 1.0 (rms 0.2 to 0.4), FP64 chain 5.7 (0.6 to 0.8).  (Two limbs of 29 bits,
// one rounding at 2^-56 of the largest product, were faster -- 135 ms against 177 at the LHCII size -- but kept fewer bits of
// small elements than FP64 does: up to 1e6 of these units.)
// A tile with Inf, NaN or exponents near the ends of the range takes the FMA chain too.
#pragma once
#include <cuda_runtime.h>

namespace heom {

constexpr int kFxBits = 28;  // bits of a limb

// |x| as an ordered integer (0 only for zero): the high word, its last bit set if only the low word is not zero.
__device__ __forceinline__ int fx_key(double x) {
  const int h = __double2hiint(x) & 0x7fffffff;
  return h | (h == 0 && __double2loint(x) != 0);
}
__device__ __forceinline__ int fx_exp(int key) { return max(key >> 20, 1); }

// x as limbs, |x| = (hi 2^28 + lo + rest 2^-28) 2^(e - 1022 - 55) with the sign on all limbs, for
// |x| < 2^(e - 1022), cut below the last bit; |lo|, |rest|, |hi| <= 2^27.  32-bit funnel shifts: with 64-bit shifts by a
// variable and rounding to nearest two limbs took about 90 instructions, three take about 40 so.
__device__ __forceinline__ int2 fx_split(double x, int e, int &rest) {
  const int h = __double2hiint(x), l = __double2loint(x);
  const int ex = (h >> 20) & 0x7ff;
  unsigned mh = __funnelshift_l((unsigned)l, (unsigned)h, 11) | 0x80000000u, ml = (unsigned)l << 11, mz = 0;  // 1.fraction
  int n = e + 65 - 2 * kFxBits - ex;  // shift right by n >= 9
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
  int lo = (int)(xl << (32 - kFxBits)) >> (32 - kFxBits);
  int hi = (int)__funnelshift_r(xl, xh, kFxBits) + (int)((unsigned)lo >> 31);
  int rs = (int)(xz >> 4) - (up << kFxBits);
  lo += up;
  if (ex == 0) hi = lo = rs = 0;  // zero; subnormals are below the last bit wherever fx_ok holds
  const int sg = h >> 31;
  rest = (rs ^ sg) - sg;
  return make_int2((hi ^ sg) - sg, (lo ^ sg) - sg);
}

// acc + a b in one integer multiply-add.  (Written as acc += (long long)a * b the compiler widened the operands first
// and took about seven instructions for each product.)
__device__ __forceinline__ void fx_mad(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// A sum of up to 128 products of three-limb numbers: hi hi, the cross products, and the three of the next weight (at
// most 128 * 3 * 2^54 < 2^63).
struct FxSum {
  long long hh, x, ll;
  __device__ __forceinline__ FxSum() : hh(0), x(0), ll(0) {}
  __device__ __forceinline__ void add(int ah, int al, int ar, int bh, int bl, int br) {
    fx_mad(hh, ah, bh);
    fx_mad(x, ah, bl);
    fx_mad(x, al, bh);
    fx_mad(ll, al, bl);
    fx_mad(ll, ah, br);
    fx_mad(ll, ar, bh);
  }
  // w 2^28 + f, 0 <= f < 2^28, in units of the cross products (2^-82 of the largest product that the scales allow)
  __device__ __forceinline__ long long whole(unsigned &f) const {
    const long long t = x + (ll >> kFxBits);
    f = (unsigned)t & ((1u << kFxBits) - 1);
    return hh + (t >> kFxBits);
  }
};

// Whether a sum is below 2^54 units.  What was cut from its terms adds up to about a unit (rms 0.13 per product; an
// element's cut weighs half a unit at most), an FP64 chain of terms of that size rounds by about 0.7 2^-53 2^54: the line
// lies where the two meet.
__device__ __forceinline__ bool fx_weak(long long w) { return (unsigned long long)(w + (1ll << 26)) < (1ull << 27); }

// The sum times 2^p rounded to nearest, in integers; not for weak sums.  The caller keeps the result in FP64's normal range.
__device__ __forceinline__ double fx_double(long long w, unsigned f, int p) {
  const long long sg = w >> 63;
  unsigned long long u = (unsigned long long)(w ^ sg);
  const unsigned g = (f ^ (unsigned)sg) & ((1u << kFxBits) - 1);
  const int lz = __clzll((long long)u);  // 1..38
  u = u << lz | ((unsigned long long)g << (64 - kFxBits)) >> (64 - lz);
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1);  // the carry of all ones moves into the exponent
  const unsigned long long b = ((unsigned long long)(unsigned)(1085 + kFxBits - lz + p) << 52) + m;
  return __hiloint2double((int)(b >> 32) | ((int)sg & (int)0x80000000), (int)b);
}

// The same by two FP64 additions, where that pipe has room: w 2^28 + f cut at bit 52 into the low bits of 2^104 and of 2^52
// (a device long used by compilers' run-time libraries for 64-bit integers), the first addition exact.
__device__ __forceinline__ double fx_double_add(long long w, unsigned f, int p) {
  const int e = p << 20;
  const long long t = w >> 24;
  const double a = __hiloint2double(0x46780000 + e + (int)(t >> 32), (int)t);  // 2^104 + (2^51 + t) 2^52
  const double b = __hiloint2double(0x43300000 + e + (int)(((unsigned)w >> 4) & 0xfffff), (int)((unsigned)w << 28 | f));
  const double c = __hiloint2double(0x46780000 + e, 1);                        // 2^104 + 2^103 + 2^52
  return (a - c) + b;
}

// 2^p of the unit for the scales of two keys.
__device__ __forceinline__ int fx_unit(int hkey, int key) { return fx_exp(hkey) + fx_exp(key) - 2042 - 3 * kFxBits; }

// Re C and Im C from their sums (keys of H and of the parts) where those are not weak; returns which are (bits 0 and 1).  A
// zero part (or H) gives exactly zero.
__device__ __forceinline__ int fx_finish(const FxSum &r, const FxSum &m, int hk, int kx, int ky, double &cr, double &ci) {
  unsigned fr, fm;
  const long long wr = r.whole(fr), wm = m.whole(fm);
  const bool no_r = fx_weak(wr), no_m = fx_weak(wm);
  cr = no_r ? 0.0 : fx_double(wr, fr, fx_unit(hk, kx));
  ci = no_m ? 0.0 : fx_double(wm, fm, fx_unit(hk, ky));
  return (no_r && hk && kx ? 1 : 0) | (no_m && hk && ky ? 2 : 0);
}

// Whether the fixed-point sums of operands with these keys stay in FP64's normal range (or are exactly zero), and what is
// subnormal in them lies below the last limb.
__device__ __forceinline__ bool fx_ok(int hkey, int key) {
  const int e = (hkey >> 20) + (key >> 20);
  const bool h = hkey == 0 || (unsigned)(hkey - (86 << 20)) < ((2047u - 86u) << 20);
  const bool k = key == 0 || (unsigned)(key - (86 << 20)) < ((2047u - 86u) << 20);
  return h && k && (hkey == 0 || key == 0 || (e >= 1120 && e <= 3000));
}

}  // namespace heom
