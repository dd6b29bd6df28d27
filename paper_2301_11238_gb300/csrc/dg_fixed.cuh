// Block fixed-point contractions for the FP64 kernels.
//
// GB300 retires two FP64 operations per clock and SM, but 64 IMAD.WIDE (32 x 32
// + 64 bit multiply-adds), on a pipe that runs beside the FP64 pipe: one FP64
// operation takes the time of 32 of them (measured 2.0 against 55-64 lanes per
// clock and SM; both together take no longer than the FP64 part alone).  The
// reference-element contractions sum_a c_a x_a, with constant c and a handful
// of nodal values x of similar size, therefore run in integers: the x of one
// sum share an exponent (that of the largest), each is held as two signed
// parts h 2^28 + l (58 bits with the sign), the constants likewise, and a term
// takes three IMAD.WIDE:
//   a += x.h c.h ;  b += x.h c.l + x.l c.h      (x.l c.l, below one unit, is left out)
// with sum = a + b 2^-28, exact otherwise.  What is rounded: x when it is aligned
// (below 2^-57 of the group's largest), a constant to half the table's unit 2^-cs
// (cs 52 to 60, so that the table's largest row sum is just below 2^62 units), and
// the result when it returns to a double.  A sum of n terms is off by less than
// 1.5 n 2^-cs max|x| + 2^-57 sum |c| max|x|.  Against sum |c| max|x| that is far below
// a floating-point sum's several roundings of 2^-53 for rows of the table's own size,
// and comparable with it for the smallest: 2D p = 3 (n = 25), worst case 2^-48 for
// w_q l_a beside w_q dl_a/dr in one table and 2^-47 for the smallest mass products.
// The measured errors of dV/dt and E in units of their terms are those of the
// floating-point kernels or less (p = 3, rough states: h 1.04 against 1.07, u 0.45
// against 0.46, E 13.1 in both).
//
// max|x| is the group's: operands that share an exponent have to be of one kind.
// Metric terms have one exponent a direction and residual rows one unit a field,
// so that a stretched element or a small momentum component keeps its bits.
//
// Ranges.  A group whose largest value is below 2^-823 is taken as zero; one
// with a value of 2^957 or above (infinities and NaN among them) makes its
// results NaN, so a non-finite state stays non-finite.
#pragma once
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace dgswe {

struct Fx {
  int32_t h, l;  // h 2^28 + l, |h| < 2^30, |l| < 2^28
};
struct FxAcc {
  long long a, b;
};
// How results leave: exponent step kk (in the high word), and masks that make
// every result of the group zero (am = 0) or NaN (om).
struct FxScale {
  int kk, am, om;
};

constexpr int kFxLo = 28;
constexpr int kFxMinExp = 200, kFxMaxExp = 1980;  // biased exponents of a group's largest value

__device__ __forceinline__ int fx_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// x in units of 2^(E - 1075 - SH), E the group's largest biased exponent:
// |x| < 2^(53 + SH).  SH = 5 uses the format's full range; smaller SH leave
// room for sums of x.
template <int SH>
__device__ __forceinline__ Fx fx_from(double v, int E) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  // mantissa at bit 62, then down to 53 + SH bits and to the group's exponent;
  // a shift of 63 leaves nothing (zeros, tiny values, a group below kFxMinExp)
  const int sh = min((E < kFxMinExp ? 4096 : E) - ((hi >> 20) & 0x7ff) + (10 - SH), 63);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = (((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10)) >> sh;
  const int s = hi >> 31;
  Fx r;
  r.h = ((int)(m >> kFxLo) ^ s) - s;
  r.l = ((int)((unsigned)m & ((1u << kFxLo) - 1)) ^ s) - s;
  return r;
}

__device__ __forceinline__ long long fx_wide(int a, int b) { return (long long)a * (long long)b; }

__device__ __forceinline__ void fx_mac(FxAcc& s, Fx x, Fx c) {
  s.a += fx_wide(x.h, c.h);
  s.b += fx_wide(x.h, c.l);
  s.b += fx_wide(x.l, c.h);
}
// The sum in units of (unit of x)(unit of c) 2^56.
__device__ __forceinline__ long long fx_sum(const FxAcc& s) { return s.a + (s.b >> kFxLo); }
// Moves what b has above one unit of a into a: sums of more than 15 terms do
// this every 15, so that b (two products below 2^58 a term) stays below 2^63.
__device__ __forceinline__ void fx_fold(FxAcc& s) {
  s.a += s.b >> kFxLo;
  s.b &= (1ll << kFxLo) - 1;
}
// A sum |r| < 2^RB as an operand |x| < 2^58 again, in units of r's 2^(RB - 58), rounded.
template <int RB>
__device__ __forceinline__ Fx fx_operand(long long r) {
  const long long t = r + (1ll << (RB - 59));
  Fx x;
  x.h = (int)(t >> (RB - 30));
  x.l = (int)((unsigned)(t >> (RB - 58)) & ((1u << kFxLo) - 1));
  return x;
}
// Left shift that brings the sums whose magnitudes were or-ed into m (fx_mag)
// up to 2^61 .. 2^62.
__device__ __forceinline__ unsigned long long fx_mag(long long r) { return (unsigned long long)(r ^ (r >> 63)); }
__device__ __forceinline__ int fx_norm(unsigned long long m) { return max(__clzll((long long)(m | 1)) - 2, 0); }

// Scale of results r 2^k (k in binary orders) whose groups' largest exponents
// were lo..hi (several groups for a product of groups).
__device__ __forceinline__ FxScale fx_scale(int k, bool finite) {
  FxScale s;
  s.kk = (int)((unsigned)k << 20);
  s.am = k < -1022 ? 0 : -1;
  s.om = (!finite || k > 960) ? 0x7ff80000 : 0;
  return s;
}
// Normalized by integer shifts and rounded to nearest (halves up): the
// conversion instruction takes the FP64 pipe (face 788 -> 750 us, volume 929 ->
// 898 us, E-step 115 -> 121 us on 524,288 triangles at p = 2).
__device__ __forceinline__ double fx_to(long long r, const FxScale& s) {
  const int sg = (int)(r >> 63);
  const unsigned long long m = (unsigned long long)((r ^ (long long)sg) - (long long)sg);
  const int lz = __clzll((long long)m);
  const unsigned long long t = ((m << (lz & 63)) >> 10) + 1;  // 53 bits and half of the last one
  const int hi = (int)(t >> 33) + ((1022 + 63 - lz) << 20) + s.kk;  // the leading bit adds one to the exponent
  const int keep = m != 0 ? s.am : 0;
  return __hiloint2double(((hi | (sg & (int)0x80000000u)) & keep) | s.om, (int)(unsigned)(t >> 1) & keep);
}

// ------------------------------------------------------------------ host: constant tables

// A constant in units of 2^-cs.
inline Fx fx_const(double c, int cs) {
  const long long m = std::llround(std::ldexp(c, cs));
  Fx r;
  r.h = (int32_t)(m >> kFxLo);
  r.l = (int32_t)(m - ((long long)r.h << kFxLo));
  return r;
}
// Largest cs at which the constants are below 2^58 units and a row of absolute
// sum `row` keeps |sum| below 2^62 for operands below 2^xbits.
inline int fx_table_scale(double cmax, double row, int xbits) {
  int e1 = 0, e2 = 0;
  std::frexp(cmax, &e1);
  std::frexp(row, &e2);
  const int a = 58 - e1, b = 62 + 56 - xbits - e2;
  return a < b ? a : b;
}

}  // namespace dgswe
