// Block fixed point: sums of products evaluated in 58-bit integers on the
// integer pipe instead of the FP64 pipe.
//
// This GPU retires two FP64 thread operations per SM and clock and about sixty
// 32-bit integer ones (measured: fma.f64 2.1, mad.wide.s32 58, shifts and logic
// 62 per SM and clock), so a sum of products whose factors share a scale is
// cheaper as integer arithmetic, conversions included.  A block of values (the
// fluxes of one element and variable class) is written as X 2^s with one common
// exponent and |X| < 2^58, X = h 2^29 + l; a fixed matrix (the DFR derivative
// rows) likewise.  A product then needs three widening multiply-adds: h h', and
// h l' + l h' (l l' is below 2^-57 of the largest product).  The sums are exact
// in 64 bits for up to twenty terms: |h|, |l| <= 2^29, so the h h' sum stays
// below 20 2^58 < 2^63, and with the matrix' l' centred (|l'| <= 2^28) the
// mixed sum below 20 (2^57 + 2^58) < 2^63.  A block's largest value carries 58 bits
// and the sum is rounded once, where an FP64 chain rounds every partial sum to 53:
// against its largest terms a sum is more accurate (measured against a 64-bit
// reference; see the kernels).  A value k bits below its block's largest one holds
// 58 - k bits, so a sum of such values alone can hold fewer than an FP64 chain's.
//
// Blocks the format cannot hold faithfully -- a NaN, an infinity, a largest
// magnitude outside 2^-623 .. 2^677 -- are left to the FP64 chain (fx_usable).
#pragma once

#include <cuda_runtime.h>

namespace swepi {

constexpr int kFxBits = 58;                      // magnitude bits of a block value
constexpr int kFxLimb = 29;                      // bits of the low limb
constexpr int kFxExpMin = 400, kFxExpMax = 1700; // biased exponents of the largest magnitude the format takes
constexpr int kFxPackMin = 58;                   // smallest block exponent a value is packed for (fx_pack)
// largest exponent of a packed coefficient class of the split product (lin_node_kernel)
constexpr int kFxCoefMax = 1020 + kFxExpMin + 2 - kFxPackMin;

// the magnitude key a block's maximum is taken over: the high word without the
// sign (ordered as the magnitudes are, NaN and infinities above all others)
__device__ __forceinline__ unsigned fx_key(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// whether a block whose largest key is m can be held (m = 0: all zero)
__device__ __forceinline__ bool fx_usable(unsigned m) {
  const unsigned e = m >> 20;
  return m == 0u || (e >= (unsigned)kFxExpMin && e <= (unsigned)kFxExpMax);
}
// the block's biased exponent
__device__ __forceinline__ int fx_exp(unsigned m) { return m == 0u ? 1023 : (int)(m >> 20); }

__device__ __forceinline__ unsigned shr_clamped(unsigned x, int s) {   // 0 for shifts of 32 and more
  unsigned r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
}

// x as block value for the block exponent E (>= the exponent of x): h and l
// packed as the high and low word of a double (a container, never an operand
// of FP64 arithmetic).  X = trunc(|x| 2^(58 - (E - 1022))), the sign on both
// limbs.  Zeros and subnormals (exponent field 0) become 0: E is at least kFxPackMin.
__device__ __forceinline__ double fx_pack(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int d = E - (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  // the significand at the top of 64 bits (th:tl); X = (th:tl) >> (6 + d)
  const unsigned th = __funnelshift_l(lo, mh, 11), tl = lo << 11;
  const unsigned xh = shr_clamped(th, d + 3);
  const unsigned xl = shr_clamped(__funnelshift_rc(tl, th, d + 6), max(d - 26, 0)) & 0x1fffffffu;
  const int s = (int)hi >> 31;
  return __hiloint2double(((int)xh ^ s) - s, ((int)xl ^ s) - s);
}

// the FP64 value of a packed one (rounded to 53 bits)
__device__ __forceinline__ double fx_unpack(double p, int E) {
  const double x = fma((double)__double2hiint(p), 536870912.0, (double)__double2loint(p));
  return x * __hiloint2double((E - 57) << 20, 0);   // 2^(E - 1080)
}

// sum of products of packed values
struct FxAcc {
  long long hh = 0, mid = 0;
};
__device__ __forceinline__ void fx_mac(FxAcc& a, double x, double m) {
  const int xh = __double2hiint(x), xl = __double2loint(x), mh = __double2hiint(m), ml = __double2loint(m);
  a.hh += (long long)xh * mh;
  a.mid += (long long)xh * ml;
  a.mid += (long long)xl * mh;
}
// the sum in units of 2^58 times the product of the two blocks' units
__device__ __forceinline__ double fx_sum(const FxAcc& a) {
  return (double)(a.hh + ((a.mid + (1ll << (kFxLimb - 1))) >> kFxLimb));
}

// the same sum as an integer, and as a packed value (|sum| < 2^58)
__device__ __forceinline__ long long fx_int(const FxAcc& a) {
  return a.hh + ((a.mid + (1ll << (kFxLimb - 1))) >> kFxLimb);
}
__device__ __forceinline__ double fx_repack(long long y) {
  return __hiloint2double((int)(y >> kFxLimb), (int)y & 0x1fffffff);
}

// s 2^k for an integer-valued s (a converted sum), through the exponent field
__device__ __forceinline__ double fx_ldexp(double s, int k) {
  const int hi = __double2hiint(s);
  return hi == 0 ? 0.0 : __hiloint2double(hi + k * 1048576, __double2loint(s));
}

// sum_k w_k x_k with the block exponent of the N values x: w as packed integers
// wq (units in swepi_internal.h) and, for a block the format cannot hold, as
// FP64 values (w0 where lo, else w1).  One FP64 instruction, the conversion,
// takes the place of N; the packing and the multiply-adds are integer work.
template <int N>
__device__ __forceinline__ double fx_dot(const double (&x)[N], const double (&wq)[N], int wexp, bool lo,
                                         const double* w0, const double* w1) {
  if constexpr (N == 1) return (lo ? w0[0] : w1[0]) * x[0];   // one FP64 instruction either way
  unsigned m = 0u;
#pragma unroll
  for (int k = 0; k < N; ++k) m = max(m, fx_key(x[k]));
  if (!fx_usable(m)) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) s = fma(lo ? w0[k] : w1[k], x[k], s);
    return s;
  }
  const int E = fx_exp(m);
  FxAcc a;
#pragma unroll
  for (int k = 0; k < N; ++k) fx_mac(a, fx_pack(x[k], E), wq[k]);
  return fx_ldexp(fx_sum(a), E + wexp);
}

// Largest keys (two classes) of the EPB elements of a tile of whole elements
// with NN threads each (thread t belongs to element t / NN): reduced over each
// warp's threads of one element, then one shared-memory maximum per warp and
// element.  All BLOCK threads call it; sE [EPB][2] starts at zero and is valid
// after the next barrier.
template <int NN, int EPB, int BLOCK>
__device__ __forceinline__ void fx_block_max(unsigned (*sE)[2], int le, unsigned m0, unsigned m1) {
  if constexpr (NN >= 16) {
    const int base = threadIdx.x & ~31;
    const int lanes = BLOCK - base;
    const unsigned mask = lanes >= 32 ? 0xffffffffu : (1u << lanes) - 1u;
    const int first = base / NN, last = min((base + 31) / NN, EPB - 1);
    for (int s = first; s <= last; ++s) {   // uniform over the warp
      const unsigned r0 = __reduce_max_sync(mask, le == s ? m0 : 0u), r1 = __reduce_max_sync(mask, le == s ? m1 : 0u);
      if ((threadIdx.x & 31) == 0) {
        atomicMax(&sE[s][0], r0);
        atomicMax(&sE[s][1], r1);
      }
    }
  } else {
    if (le < EPB) {
      atomicMax(&sE[le][0], m0);
      atomicMax(&sE[le][1], m1);
    }
  }
}

}  // namespace swepi
