// Fixed-point sums of products on the integer pipe, for kernels that the FP64
// pipe would bound. GB300 issues 1.6 FP64 operations per clock and SM (measured
// with independent FMA chains), against 57 multiply-adds 32 x 32 + 64; three of
// the latter make one product of two numbers of up to 59 bits held as two limbs.
//
// A value is an integer t of at most 56 bits in units of a power of two chosen
// per element from its largest input, a coefficient c the integer round(c 2^56).
// Both are split as h 2^28 + l with a signed low limb, and c t 2^-56 = h h' +
// (h l' + l h') 2^-28 up to the product of the low limbs, at most a quarter of the
// last place. A sum carries the two parts apart and is rounded once.
//
// The bound: inputs are truncated below a unit of 2^-55 to 2^-56 of the largest,
// exact from 2^-3 of it up. A sum of n products, |c| < 2, is off by at most a unit
// times the sum of |c| (the inputs), half a unit each (the coefficients), a quarter
// each (the low limbs) and half for the sum: sum|c| + 0.75 n + 0.5 units, a unit
// times the row's scale (2^scale for a largest coefficient of 1 to 2). An FMA chain
// is off by up to n/2 2^-52 of its partial sums. So a row whose largest coefficients
// meet the element's largest values comes out two to three times as accurate as in
// double (by rational arithmetic, p = 1 to 6: 4e-17 to 6e-17 against 1e-16 to 2e-16
// on random inputs); a value or a coefficient 2^-k of the largest of its group keeps
// 56 - k of its own bits, where a double keeps 53. The scales (of rows, of groups of
// columns, of elements) are chosen so that operators whose blocks differ in size, by
// a small time step or by a velocity nearly along a face, lose nothing to it.
// (Rounding the inputs to nearest changed no error against a 64-bit solution and
// took 8% at 256 x 256 elements with an operator each, p = 4.)
#pragma once

#include <cuda_runtime.h>

#include <cstring>

// (the integer parts compile for the host too, where a test checks the bound)
#define FX_INLINE __host__ __device__ __forceinline__

namespace ehdg {

// coefficient c as the limbs of round(c 2^56)
struct Cfx {
  int h, l;
};

constexpr int kW = 28;                                  // bits of a low limb
constexpr long long kHalf = 1LL << (kW - 1);

// t = h 2^28 + l with l in [-2^27, 2^27)
struct Limb {
  int h, l;
};
FX_INLINE Limb fx_split(long long t) {
  Limb x;
  x.h = (int)((t + kHalf) >> kW);
  x.l = (int)((unsigned)t - ((unsigned)x.h << kW));
  return x;
}

FX_INLINE long long fx_pack(const Limb& x) {
  return (long long)((unsigned long long)(unsigned)x.h << 32 | (unsigned)x.l);
}
FX_INLINE Limb fx_limb(long long v) {
  return Limb{(int)(v >> 32), (int)v};
}

// a += c x as one multiply-add; the compiler makes more of the C++ product and sum
FX_INLINE void fx_mad(long long& a, int c, int x) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(c), "r"(x), "l"(a));
  a = r;
#else
  a += (long long)c * x;
#endif
}

// a sum of products c x 2^56 as hi 2^56 + mid 2^28 (the products of two low
// limbs, below a quarter of the last place each, are left out)
struct Acc {
  long long hi, mid;
  FX_INLINE explicit Acc(long long y) : hi(y), mid(kHalf) {}
  FX_INLINE void mac(const Cfx& c, const Limb& x) {
    fx_mad(hi, c.h, x.h);
    fx_mad(mid, c.h, x.l);
    fx_mad(mid, c.l, x.h);
  }
  FX_INLINE long long get() const { return hi + (mid >> kW); }
};

// 2^e as a double, e in [-1022, 1023]
__device__ __forceinline__ double fx_pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// m 2^e: one conversion on the FP64 pipe, the scale added to the exponent field
__device__ __forceinline__ double fx_value(long long m, int e) {
  const double x = (double)m;
  if (e > -1000 && e < 900)
    return m == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + e * (1 << 20), __double2loint(x));
  const int a = max(-1022, min(1023, e / 2)), b = max(-1022, min(1023, e - e / 2));
  return x * fx_pow2(a) * fx_pow2(b);
}

// the high and low words of a double
FX_INLINE int fx_high(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  long long v;
  memcpy(&v, &x, sizeof v);
  return (int)(v >> 32);
#endif
}
FX_INLINE unsigned fx_low(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  long long v;
  memcpy(&v, &x, sizeof v);
  return (unsigned)v;
#endif
}
FX_INLINE int fx_max(int a, int b) { return a > b ? a : b; }
FX_INLINE int fx_min(int a, int b) { return a < b ? a : b; }

FX_INLINE int fx_exponent(double x) { return (fx_high(x) >> 20) & 0x7ff; }

// x in units of 2^(emax - 1078), truncated, for biased exponents up to emax (that
// of zero and the subnormals counts as 1): |result| < 2^56
FX_INLINE long long fx_from_double(double x, int emax) {
  const int hi = fx_high(x), e = fx_exponent(x);
  const unsigned long long m =
      (unsigned long long)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32 | fx_low(x);
  const long long v = (long long)((m << 3) >> fx_min(63, emax - fx_max(e, 1)));
  const long long sg = (long long)(hi >> 31);
  return (v ^ sg) - sg;
}

// v 2^-s rounded, for s >= 0 and |v| < 2^61
FX_INLINE long long fx_shift(long long v, int s) {
  s = fx_min(s, 62);
  return (v + ((1LL << s) >> 1)) >> s;
}

// A shared operator's rows as limbs in blocks of four rows, [rows / 4][cols][4]
// (the last block zero-padded), with scales of either sign: 2^col[a] for the
// columns of group a (an axis's faces), and for each row one for each of its ng
// parts, the columns whose values have units of their own (the fields of the state),
// scale[row * ng + f]. entry = 2^(col + scale - 56) (h 2^28 + l); with col divided
// out the limbs' value is below 2 and its sum over the part below 32, so that a
// part's products with 56-bit values sum below 2^62.
struct FxOp {
  const int2* x;
  const int* scale;
  int col[3];
};
// a value that is not finite in the exponent of a set of values
constexpr int kNotFinite = 1 << 16;
// the scale of a group of columns that are zero, so low that its values do not
// raise the others' unit
constexpr int kZeroGroup = -4096;
__host__ __device__ inline int64_t fx_blocked(int rows, int cols) {
  return (int64_t)((rows + 3) / 4) * 4 * cols;
}

// four rows (blk) times the column of packed limbs X[c * 32]
__device__ __forceinline__ void fx_rows4(const int2* blk, const long long* X, int cols,
                                         long long (&y)[4]) {
  Acc t[4] = {Acc(0), Acc(0), Acc(0), Acc(0)};
  const int4* b = reinterpret_cast<const int4*>(blk);
#pragma unroll 4
  for (int c = 0; c < cols; ++c) {
    const int4 p = b[2 * c], q = b[2 * c + 1];
    const Limb x = fx_limb(X[c * 32]);
    t[0].mac(Cfx{p.x, p.y}, x);
    t[1].mac(Cfx{p.z, p.w}, x);
    t[2].mac(Cfx{q.x, q.y}, x);
    t[3].mac(Cfx{q.z, q.w}, x);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) y[i] = t[i].get();
}

}  // namespace ehdg
