// Clover term and its inverse (App. A of arXiv:2109.10687), to float64.
//
// F_mu,nu(n) = (Q_mu,nu - Q_mu,nu^dag) / 8 with Q the sum of the four
// plaquettes ("leaves") in the mu-nu plane through n, all oriented the same
// way; C = i kappa c_SW sum_{mu<nu} sigma_mu,nu F_mu,nu.  In the chiral basis
// sigma_mu,nu is block diagonal, so 1 + C splits into two 6x6 Hermitian
// blocks per site:
//   upper: sigma_1 (F_xt - F_yz) + sigma_2 (F_xz + F_yt) + sigma_3 (F_zt - F_xy)
//   lower: sigma_1 (-F_xt - F_yz) + sigma_2 (F_xz - F_yt) + sigma_3 (-F_zt - F_xy)
// (sigma_k (x) A = [[A_3, A_1 - i A_2], [A_1 + i A_2, -A_3]] on (spin, colour)),
// each multiplied by i kappa c_SW.
//
// One block of the build kernel takes 32 sites in three phases: a warp per
// plane computes F of its plane (a thread per site); a warp per chiral block
// packs 1 + C and inverts it in float64; all six warps write every copy of
// both that the library keeps, each a coalesced stream, from shared memory.
//
// What bounds it: this GPU has two float64 lanes per SM and cycle, and the
// leaves and inverses in float64 (11.2 k fused multiply-adds per site, one
// thread per site) took 17.3 ms on 24^3 x 48, and the staging copies another
// 0.64 ms; this kernel takes 5.4 ms for both.  Links of SU(3) are bounded by one, so their products are done
// in fixed point instead, on the integer multipliers: a number is
// (hi 2^29 + lo) 2^-58 with 30-bit signed hi and lo, a product of two is
// three 32x32 -> 64 multiply-adds (lo lo, below 2^-59 of one, is left out),
// and a sum of products stays in 64 bits.  The error of a matrix product is
// a few units of 2^-58 of the entries' bound, below float64's 2^-53.

#include "qcd_internal.cuh"

namespace qcd {

using C64 = cx<double>;
using M3 = SU3<double>;

__device__ __forceinline__ void mat_mul(const M3& a, const M3& b, M3& c) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      C64 acc = a.m[i][0] * b.m[0][j];
      acc = cmac(acc, a.m[i][1], b.m[1][j]);
      acc = cmac(acc, a.m[i][2], b.m[2][j]);
      c.m[i][j] = acc;
    }
}

__device__ __forceinline__ M3 dagger(const M3& a) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.m[i][j] = conjg(a.m[j][i]);
  return r;
}

// U_mu at site x + off (periodic wrap; links carry no boundary sign)
__device__ __forceinline__ M3 link_at(const Geom& g, const LinkPtr<double>& U, const int x[4], const int off[4],
                                      int mu) {
  int y[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) y[k] = (x[k] + off[k] + g.L[k]) % g.L[k];
  int dom, s;
  coords_to_internal(g, y, dom, s);
  M3 u;
  U.load(g, dom, mu, s, u);
  return u;
}

__device__ M3 prod4(const M3& a, const M3& b, const M3& c, const M3& d) {
  M3 t1, t2, r;
  mat_mul(a, b, t1);
  mat_mul(t1, c, t2);
  mat_mul(t2, d, r);
  return r;
}

// F_mu,nu = (Q - Q^dag) / 8 in float64, for links that need not be SU(3)
// (and so have no bound): the nine reals of field_strength_fx
__device__ __noinline__ void field_strength(const Geom& g, const LinkPtr<double>& U, const int x[4], int mu, int nu,
                                            double f[9]) {
  auto at = [&](int dm, int dn, int dir) {
    int off[4] = {0, 0, 0, 0};
    off[mu] += dm;
    off[nu] += dn;
    return link_at(g, U, x, off, dir);
  };
  const M3 um = at(0, 0, mu), un = at(0, 0, nu);
  M3 q1 = prod4(um, at(1, 0, nu), dagger(at(0, 1, mu)), dagger(un));
  M3 q2 = prod4(un, dagger(at(-1, 1, mu)), dagger(at(-1, 0, nu)), at(-1, 0, mu));
  M3 q3 = prod4(dagger(at(-1, 0, mu)), dagger(at(-1, -1, nu)), at(-1, -1, mu), at(0, -1, nu));
  M3 q4 = prod4(dagger(at(0, -1, nu)), at(0, -1, mu), at(1, -1, nu), dagger(um));
  M3 q;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) q.m[i][j] = q1.m[i][j] + q2.m[i][j] + q3.m[i][j] + q4.m[i][j];
  for (int i = 0; i < 3; ++i) f[i] = 0.25 * q.m[i][i].im;
  int o = 3;
  for (int i = 0; i < 3; ++i)
    for (int j = i + 1; j < 3; ++j) {
      f[o++] = 0.125 * (q.m[i][j].re - q.m[j][i].re);
      f[o++] = 0.125 * (q.m[i][j].im + q.m[j][i].im);
    }
}

// ---------------------------------------------------------------------------
// fixed-point 3x3 complex matrices
// ---------------------------------------------------------------------------
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

// C = op(A) op(B), op the conjugate transpose where DA / DB is set.  Sums of
// six products of |hi| <= 2^29 and 2^30 stay below 2^62.
template <bool DA, bool DB>
__device__ __forceinline__ void fx_mul(const FxMat& A, const FxMat& B, FxSum& C) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    // this row's real parts, imaginary parts, and the two operands whose
    // sign the complex product flips (re: -ai bi, im: +ar bi, with bi -> -bi for DB)
    int ah[3], al[3], bh[3], bl[3], ph[3], pl[3], qh[3], ql[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ah[k] = DA ? A.rh[k][i] : A.rh[i][k];
      al[k] = DA ? A.rl[k][i] : A.rl[i][k];
      const int xh = DA ? A.ih[k][i] : A.ih[i][k], xl = DA ? A.il[k][i] : A.il[i][k];
      bh[k] = DA ? -xh : xh;
      bl[k] = DA ? -xl : xl;
      ph[k] = DB ? bh[k] : -bh[k];
      pl[k] = DB ? bl[k] : -bl[k];
      qh[k] = DB ? -ah[k] : ah[k];
      ql[k] = DB ? -al[k] : al[k];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      long long rh = 0, rx = 1LL << (FX_LIMB - 1), ih = 0, ix = 1LL << (FX_LIMB - 1);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int yrh = DB ? B.rh[j][k] : B.rh[k][j], yrl = DB ? B.rl[j][k] : B.rl[k][j];
        const int yih = DB ? B.ih[j][k] : B.ih[k][j], yil = DB ? B.il[j][k] : B.il[k][j];
        rh += (long long)ah[k] * yrh;
        rh += (long long)ph[k] * yih;
        rx += (long long)ah[k] * yrl;
        rx += (long long)al[k] * yrh;
        rx += (long long)ph[k] * yil;
        rx += (long long)pl[k] * yih;
        ih += (long long)qh[k] * yih;
        ih += (long long)bh[k] * yrh;
        ix += (long long)qh[k] * yil;
        ix += (long long)ql[k] * yih;
        ix += (long long)bh[k] * yrl;
        ix += (long long)bl[k] * yrh;
      }
      C.re[i][j] = rh + (rx >> FX_LIMB);
      C.im[i][j] = ih + (ix >> FX_LIMB);
    }
  }
}

// A -= B^dag
__device__ __forceinline__ void fx_sub_dag(FxSum& A, const FxSum& B) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      A.re[i][j] -= B.re[j][i];
      A.im[i][j] += B.im[j][i];
    }
}
// A -= B
__device__ __forceinline__ void fx_sub(FxSum& A, const FxSum& B) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      A.re[i][j] -= B.re[i][j];
      A.im[i][j] -= B.im[i][j];
    }
}

// links as limbs, int4 (re hi, re lo, im hi, im lo) [dom][mu][9][vd]
__device__ __forceinline__ FxMat fx_link(const Geom& g, const int4* __restrict__ U, const int x[4], int mu, int nu,
                                         int dm, int dn, int dir) {
  int y[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int v = x[k] + (k == mu ? dm : 0) + (k == nu ? dn : 0);
    y[k] = v < 0 ? v + g.L[k] : (v >= g.L[k] ? v - g.L[k] : v);
  }
  int dom, s;
  coords_to_internal(g, y, dom, s);
  const int4* p = U + (((size_t)((dom * 4 + dir) * 9)) << g.logvd) + s;
  FxMat m;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int4 v = __ldg(p + ((size_t)e << g.logvd));
    m.rh[e / 3][e % 3] = v.x;
    m.rl[e / 3][e % 3] = v.y;
    m.ih[e / 3][e % 3] = v.z;
    m.il[e / 3][e % 3] = v.w;
  }
  return m;
}

// F_mu,nu at x, as its nine independent reals: the imaginary parts of the
// diagonal, then (re, im) of the entries 01, 02, 12.  Two leaves share a
// first factor and two a last one up to the conjugate transpose, and only
// Q - Q^dag is needed:
//   Q - Q^dag = M - M^dag,  M = U_mu(n) (A - B^dag) + (C - E) U_mu(n - mu),
// with A, B^dag, C, E products of three links: ten matrix products instead
// of twelve.
__device__ __forceinline__ void field_strength_fx(const Geom& g, const int4* U, const int x[4], int mu, int nu,
                                                  double f[9]) {
  auto at = [&](int dm, int dn, int dir) { return fx_link(g, U, x, mu, nu, dm, dn, dir); };
  FxSum M, S, T;
  FxMat t;
  {  // A - B^dag, with U_nu(n) and then U_nu(n - nu) as the outer factor
    fx_mul<false, true>(at(1, 0, nu), at(0, 1, mu), S);
    fx_limbs(S, t);
    fx_mul<false, true>(t, at(0, 0, nu), S);
    fx_mul<false, false>(at(0, -1, mu), at(1, -1, nu), T);
    fx_limbs(T, t);
    fx_mul<true, false>(at(0, -1, nu), t, T);
    fx_sub_dag(S, T);
    fx_limbs(S, t);
    fx_mul<false, false>(at(0, 0, mu), t, M);
  }
  {  // C - E
    fx_mul<false, true>(at(0, 0, nu), at(-1, 1, mu), S);
    fx_limbs(S, t);
    fx_mul<false, true>(t, at(-1, 0, nu), S);
    fx_mul<true, false>(at(-1, -1, mu), at(-1, -1, nu), T);
    fx_limbs(T, t);
    fx_mul<true, false>(at(0, -1, nu), t, T);
    fx_sub(S, T);
    fx_limbs(S, t);
    fx_mul<false, false>(t, at(-1, 0, mu), S);
  }
  const double u = 1.0 / (double)(1LL << FX_FRAC) / 8.0;  // a power of two
#pragma unroll
  for (int i = 0; i < 3; ++i) f[i] = u * (double)(2 * (M.im[i][i] + S.im[i][i]));
  int o = 3;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      f[o++] = u * (double)((M.re[i][j] + S.re[i][j]) - (M.re[j][i] + S.re[j][i]));
      f[o++] = u * (double)((M.im[i][j] + S.im[i][j]) + (M.im[j][i] + S.im[j][i]));
    }
}

// inverse by Gauss-Jordan with partial pivoting, for blocks that are not
// safely positive definite; returns false if singular
__device__ __noinline__ bool invert6(C64 a[6][6], C64 inv[6][6]) {
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) inv[i][j] = make_cx(i == j ? 1.0 : 0.0, 0.0);
  for (int col = 0; col < 6; ++col) {
    int piv = col;
    double best = 0.0;
    for (int r = col; r < 6; ++r) {
      const double v = a[r][col].re * a[r][col].re + a[r][col].im * a[r][col].im;
      if (v > best) {
        best = v;
        piv = r;
      }
    }
    if (!(best > 1e-200)) return false;
    if (piv != col)
      for (int j = 0; j < 6; ++j) {
        C64 t = a[col][j]; a[col][j] = a[piv][j]; a[piv][j] = t;
        t = inv[col][j]; inv[col][j] = inv[piv][j]; inv[piv][j] = t;
      }
    const C64 p = a[col][col];
    const double pn = p.re * p.re + p.im * p.im;
    const C64 pinv = make_cx(p.re / pn, -p.im / pn);
    for (int j = 0; j < 6; ++j) {
      a[col][j] = a[col][j] * pinv;
      inv[col][j] = inv[col][j] * pinv;
    }
    for (int r = 0; r < 6; ++r) {
      if (r == col) continue;
      const C64 f = a[r][col];
      for (int j = 0; j < 6; ++j) {
        a[r][j] = a[r][j] - f * a[col][j];
        inv[r][j] = inv[r][j] - f * inv[col][j];
      }
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// packed Hermitian 6x6 blocks: six diagonal reals, then (re, im) of i < j
// ---------------------------------------------------------------------------
// In-place inverse of a positive definite block by Gauss-Jordan steps that
// keep it Hermitian (symmetric sweeps): no pivoting is needed there, and a
// step costs a quarter of the full elimination.  Returns false, with m
// overwritten, at a pivot that is not safely positive.
constexpr double kMinPivot = 1e-3;  // 1 + C has eigenvalues of order one
__device__ __forceinline__ bool invert6_packed(double m[36]) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    ok = ok && m[k] > kMinPivot;
    const double p = 1.0 / m[k];
    C64 t[6], s[6];  // column k, and column k times 1 / pivot
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      const int o = 6 + 2 * (i < k ? herm_off(i, k) : herm_off(k, i));
      t[i] = make_cx(m[o], i < k ? m[o + 1] : -m[o + 1]);
      s[i] = p * t[i];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      m[i] = fma(-s[i].re, t[i].re, fma(-s[i].im, t[i].im, m[i]));
#pragma unroll
      for (int j = i + 1; j < 6; ++j) {
        if (j == k) continue;
        const int o = 6 + 2 * herm_off(i, j);  // a_ij -= s_i conj(t_j)
        m[o] = fma(-s[i].re, t[j].re, fma(-s[i].im, t[j].im, m[o]));
        m[o + 1] = fma(-s[i].im, t[j].re, fma(s[i].re, t[j].im, m[o + 1]));
      }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (i == k) continue;
      const int o = 6 + 2 * (i < k ? herm_off(i, k) : herm_off(k, i));
      m[o] = s[i].re;
      m[o + 1] = i < k ? s[i].im : -s[i].im;
    }
    m[k] = -p;
  }
#pragma unroll
  for (int i = 0; i < 36; ++i) m[i] = -m[i];
  return ok;
}

// the same through the pivoted elimination, from r to out (element k at
// k stride; zero if singular)
__device__ __noinline__ bool invert6_general(const double* r, double* out, int stride) {
  C64 m[6][6], inv[6][6];
  for (int i = 0; i < 6; ++i) {
    m[i][i] = make_cx(r[i * stride], 0.0);
    for (int j = i + 1; j < 6; ++j) {
      const int o = 6 + 2 * herm_off(i, j);
      m[i][j] = make_cx(r[o * stride], r[(o + 1) * stride]);
      m[j][i] = conjg(m[i][j]);
    }
  }
  const bool ok = invert6(m, inv);
  for (int i = 0; i < 6; ++i) {
    out[i * stride] = ok ? inv[i][i].re : 0.0;
    for (int j = i + 1; j < 6; ++j) {
      const int o = 6 + 2 * herm_off(i, j);
      out[o * stride] = ok ? 0.5 * (inv[i][j].re + inv[j][i].re) : 0.0;
      out[(o + 1) * stride] = ok ? 0.5 * (inv[i][j].im - inv[j][i].im) : 0.0;
    }
  }
  return ok;
}

// chiral block b of 1 + C from the six F (nine reals each, read by f(plane, e)):
// 1 + [[H_3, H_1 - i H_2], [H_1 + i H_2, -H_3]], H_k = i kc A_k Hermitian
template <typename F>
__device__ __forceinline__ void pack_block(const F& f, int b, double kc, double m[36]) {
  // planes 0 xy, 1 xz, 2 xt, 3 yz, 4 yt, 5 zt
  const double sg = b == 0 ? 1.0 : -1.0;
  double a1[9], a2[9], a3[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    a1[e] = kc * fma(sg, f(2, e), -f(3, e));
    a2[e] = kc * fma(sg, f(4, e), f(1, e));
    a3[e] = kc * fma(sg, f(5, e), -f(0, e));
  }
  // entry (i, j) of i A for A given as the nine reals
  auto h = [](const double a[9], int i, int j) {
    if (i == j) return make_cx(-a[i], 0.0);
    const int o = 3 + 2 * ((i < j ? i + j : j + i) - 1);  // 01 -> 0, 02 -> 1, 12 -> 2
    return i < j ? make_cx(-a[o + 1], a[o]) : make_cx(-a[o + 1], -a[o]);
  };
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    m[i] = 1.0 - a3[i];
    m[i + 3] = 1.0 + a3[i];
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      const C64 v = h(a3, i, j);
      const int o = 6 + 2 * herm_off(i, j), q = 6 + 2 * herm_off(i + 3, j + 3);
      m[o] = v.re;
      m[o + 1] = v.im;
      m[q] = -v.re;
      m[q + 1] = -v.im;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const C64 u = h(a1, i, j), v = h(a2, i, j);
      const int o = 6 + 2 * herm_off(i, j + 3);
      m[o] = u.re + v.im;  // u - i v
      m[o + 1] = u.im - v.re;
    }
  }
}

// ---------------------------------------------------------------------------
// the build kernel
// ---------------------------------------------------------------------------
constexpr int CB_SITES = 32;
constexpr int CB_THREADS = 6 * CB_SITES;  // a warp per plane
constexpr int CB_STRIDE = CB_SITES + 1;   // an odd stride: rows and columns without bank conflicts
constexpr size_t CB_SMEM = sizeof(double) * (54 + 144) * CB_STRIDE + sizeof(size_t) * CB_SITES;

struct CloverOut {
  double2 *clov64, *cinv64;   // [dom][36][vd]
  float4 *clov32, *cinv32;    // [dom][18][vd]
  __half2* cinv16;            // [dom][36][vd]
  float4* clovdf;             // [dom][36][vd], double-float
  uint4* st16;                // staging of the SAP block kernel (4^4 domains, else null): [dom][site][9]
  float4* st32;               // [dom][site][19]
};

template <bool FIXED>
__global__ void __launch_bounds__(CB_THREADS, 2) clover_build_kernel(Geom g, const int4* __restrict__ ufx,
                                                                     LinkPtr<double> U, double kc, CloverOut o,
                                                                     int* status) {
  extern __shared__ double csm[];
  double* sf = csm;                         // F: [plane][9][site]
  double* sm = csm + 54 * CB_STRIDE;        // 1 + C, then its inverse: [2][block][36][site]
  size_t* sbase = reinterpret_cast<size_t*>(sm + 144 * CB_STRIDE);  // (dom, s) of every site
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long n0 = blockIdx.x * (long long)CB_SITES;
  const int live = (int)min((long long)CB_SITES, g.vol - n0);
  {
    // sites in lexicographic-domain order, so that neighbouring domains'
    // links are still in L2; a block's sites past the end repeat its first
    const long long gid = n0 + (lane < live ? lane : 0);
    int x[4], lex = (int)(gid >> g.logvd);
    const int s = (int)(gid & (g.vd - 1));
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int q = lex / g.nd[mu];
      x[mu] = (lex - q * g.nd[mu]) * g.d[mu] + ((s >> g.shift[mu]) & (g.d[mu] - 1));
      lex = q;
    }
    if (warp == 0) sbase[lane] = ((size_t)__ldg(g.lex2dom + (int)(gid >> g.logvd)) << 8) | (size_t)s;
    const int mu = warp < 3 ? 0 : (warp < 5 ? 1 : 2);
    const int nu = warp < 3 ? warp + 1 : (warp < 5 ? warp - 1 : 3);
    double f[9];
    if (FIXED) field_strength_fx(g, ufx, x, mu, nu, f);
    else field_strength(g, U, x, mu, nu, f);
#pragma unroll
    for (int e = 0; e < 9; ++e) sf[(warp * 9 + e) * CB_STRIDE + lane] = f[e];
  }
  __syncthreads();
  if (warp < 2) {
    double m[36];
    pack_block([&](int p, int e) { return sf[(p * 9 + e) * CB_STRIDE + lane]; }, warp, kc, m);
    double* out = sm + warp * 36 * CB_STRIDE + lane;
#pragma unroll
    for (int k = 0; k < 36; ++k) out[k * CB_STRIDE] = m[k];
    double* inv = out + 72 * CB_STRIDE;
    bool ok = invert6_packed(m);
#pragma unroll
    for (int k = 0; k < 36; ++k) inv[k * CB_STRIDE] = m[k];
    if (!ok) ok = invert6_general(out, inv, CB_STRIDE);
    bool finite = true;
    for (int k = 0; k < 36; ++k) finite = finite && isfinite(inv[k * CB_STRIDE]);
    if ((!ok || !finite) && lane < live) atomicExch(status, 1);
  }
  __syncthreads();
  // every copy; lane = site: each component is one stream over the sites
  if (lane < live) {
    const size_t base = sbase[lane];
    const size_t dom = base >> 8, s = base & 255;
    const double* v = sm + lane;
    for (int k = warp; k < 36; k += 6) {
      const size_t i = ((dom * 36 + k) << g.logvd) + s;
      const double c0 = v[2 * k * CB_STRIDE], c1 = v[(2 * k + 1) * CB_STRIDE];
      const double q0 = v[(72 + 2 * k) * CB_STRIDE], q1 = v[(73 + 2 * k) * CB_STRIDE];
      o.clov64[i] = make_double2(c0, c1);
      o.cinv64[i] = make_double2(q0, q1);
      o.cinv16[i] = __floats2half2_rn((float)q0, (float)q1);
      const df64 d0 = df64_from_double_scaled(c0, 0), d1 = df64_from_double_scaled(c1, 0);
      o.clovdf[i] = make_float4(d0.hi, d0.lo, d1.hi, d1.lo);
    }
    for (int k = warp; k < 18; k += 6) {
      const size_t i = ((dom * 18 + k) << g.logvd) + s;
      const double* c = v + 4 * k * CB_STRIDE;
      const double* q = c + 72 * CB_STRIDE;
      o.clov32[i] = make_float4((float)c[0], (float)c[CB_STRIDE], (float)c[2 * CB_STRIDE], (float)c[3 * CB_STRIDE]);
      o.cinv32[i] = make_float4((float)q[0], (float)q[CB_STRIDE], (float)q[2 * CB_STRIDE], (float)q[3 * CB_STRIDE]);
    }
  }
  if (o.st16) {
    // 4^4 domains: the 32 sites are consecutive sites of one domain, and so
    // is their stretch of the site-major staging layouts
    const size_t site0 = (sbase[0] >> 8) * 256 + (sbase[0] & 255);
    for (int i = threadIdx.x; i < CB_SITES * 9; i += CB_THREADS) {
      const double* q = sm + (size_t)(72 + 8 * (i % 9)) * CB_STRIDE + i / 9;
      __half2 h[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        h[e] = __floats2half2_rn((float)q[2 * e * CB_STRIDE], (float)q[(2 * e + 1) * CB_STRIDE]);
      o.st16[site0 * 9 + i] = *reinterpret_cast<const uint4*>(h);
    }
    for (int i = threadIdx.x; i < CB_SITES * 19; i += CB_THREADS) {
      const int k = i % 19;
      float4 w = make_float4(0.f, 0.f, 0.f, 0.f);  // the last one pads the site
      if (k < 18) {
        const double* q = sm + (size_t)(72 + 4 * k) * CB_STRIDE + i / 19;
        w = make_float4((float)q[0], (float)q[CB_STRIDE], (float)q[2 * CB_STRIDE], (float)q[3 * CB_STRIDE]);
      }
      o.st32[site0 * 19 + i] = w;
    }
  }
}

__global__ void links_to_fixed_kernel(const double2* __restrict__ u64, int4* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double2 v = u64[i];
    int4 w;
    fx_split(fx_from_double(v.x), w.x, w.y);
    fx_split(fx_from_double(v.y), w.z, w.w);
    out[i] = w;
  }
}

// The fixed-point path takes links that set_gauge found to be SU(3) to 1e-9
// (their entries are bounded by one); any others, which a caller may set by
// switching that check off, take the float64 products.
void build_clover_launch(qcd_ctx* ctx, cudaStream_t st) {
  const Geom& g = ctx->geom;
  static const bool attr = [] {
    QCD_CUDA_CHECK(cudaFuncSetAttribute(clover_build_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)CB_SMEM));
    QCD_CUDA_CHECK(cudaFuncSetAttribute(clover_build_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)CB_SMEM));
    return true;
  }();
  (void)attr;
  const CloverOut o{ctx->clov64, ctx->cinv64, ctx->clov32, ctx->cinv32, ctx->cinv16, ctx->clovdf,
                    (uint4*)ctx->st_clov16, (float4*)ctx->st_clov32};
  const int grid = grid_for(g.vol, CB_SITES);
  const LinkPtr<double> U{ctx->u64};
  const double kc = ctx->kappa * ctx->csw;
  if (ctx->su3_links) {
    // the limbs lie where the double-float links go once the clover term is built
    int4* ufx = reinterpret_cast<int4*>(ctx->udf);
    {
      LaunchScope ls(ctx, QCD_KC_OTHER, st);
      links_to_fixed_kernel<<<1216, 256, 0, st>>>(ctx->u64, ufx, (size_t)g.vol * 36);
      check_launch();
    }
    LaunchScope ls(ctx, QCD_KC_OTHER, st);
    clover_build_kernel<true><<<grid, CB_THREADS, CB_SMEM, st>>>(g, ufx, U, kc, o, ctx->d_status);
    check_launch();
  } else {
    LaunchScope ls(ctx, QCD_KC_OTHER, st);
    clover_build_kernel<false><<<grid, CB_THREADS, CB_SMEM, st>>>(g, nullptr, U, kc, o, ctx->d_status);
    check_launch();
  }
}

}  // namespace qcd
