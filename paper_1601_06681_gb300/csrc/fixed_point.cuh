// Fixed-point sums of products on the integer pipe, for kernels that the FP64
// pipe would bound. GB300 issues 1.6 FP64 operations per clock and SM (measured
// with independent FMA chains), against 57 multiply-adds 32 x 32 + 64; three of
// the latter make one product of two numbers of up to 59 bits held as two limbs.
//
// A value is an integer t in units of a power of two chosen per element from
// its largest input, a coefficient c the integer round(c 2^56). Both are split
// as h 2^28 + l with a signed low limb, and c t 2^-56 = h h' + (h l' + l h') 2^-28
// up to the product of the low limbs, below a quarter of the last place. A sum
// carries the two parts apart and is rounded once. Against double: an FMA chain
// rounds every partial sum at 2^-53 of itself, this form its inputs and results
// at 2^-56 to 2^-57 of the element's largest value.
#pragma once

#include <cuda_runtime.h>

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
__device__ __forceinline__ Limb fx_split(long long t) {
  Limb x;
  x.h = (int)((t + kHalf) >> kW);
  x.l = (int)((unsigned)t - ((unsigned)x.h << kW));
  return x;
}

__device__ __forceinline__ long long fx_pack(const Limb& x) {
  return (long long)((unsigned long long)(unsigned)x.h << 32 | (unsigned)x.l);
}
__device__ __forceinline__ Limb fx_limb(long long v) {
  return Limb{(int)(v >> 32), (int)v};
}

// a += c x. As mad.wide: from the C++ product and sum the compiler made 10
// instructions of an Acc::mac, from three of these 6.
__device__ __forceinline__ void fx_mad(long long& a, int c, int x) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(c), "r"(x), "l"(a));
  a = r;
}

// a sum of products c x 2^56 as hi 2^56 + mid 2^28 (the products of two low
// limbs, below a quarter of the last place each, are left out)
struct Acc {
  long long hi, mid;
  __device__ __forceinline__ explicit Acc(long long y) : hi(y), mid(kHalf) {}
  __device__ __forceinline__ void mac(const Cfx& c, const Limb& x) {
    fx_mad(hi, c.h, x.h);
    fx_mad(mid, c.h, x.l);
    fx_mad(mid, c.l, x.h);
  }
  __device__ __forceinline__ long long get() const { return hi + (mid >> kW); }
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

__device__ __forceinline__ int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x in units of 2^(emax - 1078), for biased exponents up to emax >= 1:
// |result| < 2^56, truncated below the last place
__device__ __forceinline__ long long fx_from_double(double x, int emax) {
  const int hi = __double2hiint(x), e = fx_exponent(x);
  const unsigned long long m =
      (unsigned long long)(unsigned)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32 |
      (unsigned)__double2loint(x);
  const long long v = (long long)((m << 3) >> min(63, emax - max(e, 1)));
  const long long sg = (long long)(hi >> 31);
  return (v ^ sg) - sg;
}

// A shared operator's rows as limbs in blocks of four rows, [rows / 4][cols][4]
// (the last block zero-padded). The columns are in nf groups (the fields of the
// state, which may differ in size by orders), and each row has a scale for each
// group, scale[row * nf + f]: entry = 2^(scale - 56) (h 2^28 + l), the limbs'
// value below 2 and its sum over the group below 32, so that a group's products
// with 56-bit values sum below 2^62.
struct FxOp {
  const int2* x;
  const int* scale;
};
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
