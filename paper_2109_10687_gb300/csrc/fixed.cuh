// Fixed-point complex 3x3 matrices with float64-like accuracy on the integer
// multipliers: a number is an integer times 2^-58, kept as two limbs
// hi 2^29 + lo.  A product of two numbers is three 32x32 -> 64 multiply-adds
// (lo lo, below 2^-59 of one, is left out); sums of products are exact in 64
// bits.  This GPU has two float64 lanes per SM and cycle, so for matrices
// whose entries are bounded by about one (SU(3) links) this is several times
// faster than float64 at an absolute error of a few 2^-58.
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

constexpr int FX_LIMB = 29;          // bits of the low limb
constexpr int FX_FRAC = 2 * FX_LIMB; // a value is an integer times 2^-58

struct FxMat {  // limbs of re and im, |hi| <= 2^30, |lo| <= 2^28
  int rh[3][3], rl[3][3], ih[3][3], il[3][3];
};
struct FxSum {  // full 64-bit values
  long long re[3][3], im[3][3];
};

// v = hi 2^29 + lo with lo rounded to the nearest
__device__ __forceinline__ void fx_split(long long v, int& hi, int& lo) {
  hi = (int)((v + (1LL << (FX_LIMB - 1))) >> FX_LIMB);
  lo = (int)((unsigned)v - ((unsigned)hi << FX_LIMB));
}
__device__ __forceinline__ void fx_limbs(const FxSum& s, FxMat& m) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      fx_split(s.re[i][j], m.rh[i][j], m.rl[i][j]);
      fx_split(s.im[i][j], m.ih[i][j], m.il[i][j]);
    }
}

// float64 -> round(d 2^58), for |d| < 2^3, on the bit fields (the float64
// pipe is the scarce one here)
__device__ __forceinline__ long long fx_from_double(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0) return 0;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = e - 1023 - 52 + FX_FRAC;  // value = m 2^sh units
  unsigned long long v;
  if (sh >= 0) v = m << sh;
  else if (sh > -54) v = (m + (1ull << (-sh - 1))) >> -sh;
  else v = 0;
  return (b >> 63) ? -(long long)v : (long long)v;
}

// C = A B, each complex product by three real ones,
//   k = ar (br + bi),  re = k - bi (ar + ai),  im = k + br (ai - ar),
// exact in the limbs: nine multiply-adds instead of twelve (they are the
// bound, one warp instruction per cycle and SM).  For |A entries| <= 1 and
// |B entries| <= 2 the limbs' sums stay below 2^31 and the sums of three
// products below 2^62.
__device__ __forceinline__ void fx_mul(const FxMat& A, const FxMat& B, FxSum& C) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    int ph[3], pl[3], mh[3], ml[3];  // ar + ai, ai - ar
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ph[k] = A.rh[i][k] + A.ih[i][k];
      pl[k] = A.rl[i][k] + A.il[i][k];
      mh[k] = A.ih[i][k] - A.rh[i][k];
      ml[k] = A.il[i][k] - A.rl[i][k];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // hi hi products (h), and the hi lo and lo hi ones 2^29 below them (x)
      long long kh = 0, kx = 1LL << (FX_LIMB - 1), uh = 0, ux = 0, vh = 0, vx = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int sh = B.rh[k][j] + B.ih[k][j], sl = B.rl[k][j] + B.il[k][j];
        kh += (long long)A.rh[i][k] * sh;
        uh += (long long)ph[k] * B.ih[k][j];
        vh += (long long)mh[k] * B.rh[k][j];
        kx += (long long)A.rh[i][k] * sl;
        ux += (long long)ph[k] * B.il[k][j];
        vx += (long long)mh[k] * B.rl[k][j];
        kx += (long long)A.rl[i][k] * sh;
        ux += (long long)pl[k] * B.ih[k][j];
        vx += (long long)ml[k] * B.rh[k][j];
      }
      C.re[i][j] = (kh - uh) + ((kx - ux) >> FX_LIMB);
      C.im[i][j] = (kh + vh) + ((kx + vx) >> FX_LIMB);
    }
  }
}

// a single complex number as limbs, and a sum of products of such
struct FxCx {
  int rh, rl, ih, il;
};
struct FxAcc {
  long long rh, rx, ih, ix;
};
// acc + a b; neg: acc - a b
__device__ __forceinline__ FxAcc fx_cmac(FxAcc s, FxCx a, FxCx b, bool neg) {
  if (neg) a = FxCx{-a.rh, -a.rl, -a.ih, -a.il};
  s.rh += (long long)a.rh * b.rh - (long long)a.ih * b.ih;
  s.rx += (long long)a.rh * b.rl + (long long)a.rl * b.rh - (long long)a.ih * b.il - (long long)a.il * b.ih;
  s.ih += (long long)a.rh * b.ih + (long long)a.ih * b.rh;
  s.ix += (long long)a.rh * b.il + (long long)a.rl * b.ih + (long long)a.ih * b.rl + (long long)a.il * b.rh;
  return s;
}
__device__ __forceinline__ long long fx_re(const FxAcc& s) {
  return s.rh + ((s.rx + (1LL << (FX_LIMB - 1))) >> FX_LIMB);
}
__device__ __forceinline__ long long fx_im(const FxAcc& s) {
  return s.ih + ((s.ix + (1LL << (FX_LIMB - 1))) >> FX_LIMB);
}
__device__ __forceinline__ FxCx fx_entry(const FxMat& m, int i, int j) {
  return FxCx{m.rh[i][j], m.rl[i][j], m.ih[i][j], m.il[i][j]};
}

}  // namespace qcd
