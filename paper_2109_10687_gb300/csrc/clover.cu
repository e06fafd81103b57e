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
// Two kernels: F of every site and plane (a thread each; in two shares, one
// of which the neighbouring site's thread forms), then, a thread per site and
// chiral block, 1 + C, its inverse in float64 and every copy of both that the
// library keeps.
//
// What bounds them: this GPU has two float64 lanes per SM and cycle, and the
// leaves and inverses in float64 (11.2 k fused multiply-adds per site, one
// thread per site) took 17.3 ms on 24^3 x 48, and the staging copies another
// 0.64 ms.  Links of SU(3) are bounded by one, so their products are done
// in fixed point instead, on the integer multipliers: a number is
// (hi 2^29 + lo) 2^-58 with 30-bit signed hi and lo, a product of two is
// three 32x32 -> 64 multiply-adds (lo lo, below 2^-59 of one, is left out),
// and a sum of products stays in 64 bits.  The error of a matrix product is
// a few units of 2^-58 of the entries' bound, below float64's 2^-53.
// On 24^3 x 48 F takes 1.56 ms with 12 warps per SM (1.62 with 16, 1.78 with
// 20; 2.81 when a site formed its own four leaves, in pairs, and not the
// staples it shares with its neighbours) and the inversion
// 1.43 ms (the float64 pipe busy 84 %; it also adds the two shares of F).
// One kernel with a barrier between the two took 5.4 ms in the older form.

#include "fixed.cuh"
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
// (and so have no bound) or whose small entries count: the nine reals of
// field_strength_fx
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
// field strength
// ---------------------------------------------------------------------------
// The link of direction dir at x + dm e_mu + dn e_nu, or its adjoint, from
// limbs stored as int4 (re hi, re lo, im hi, im lo) [dom][mu][9][vd]
__device__ __forceinline__ FxMat fx_link(const Geom& g, const int4* __restrict__ U, const int x[4], int mu, int nu,
                                         int dm, int dn, int dir, bool dag) {
  int y[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int v = x[k] + (k == mu ? dm : 0) + (k == nu ? dn : 0);
    y[k] = v < 0 ? v + g.L[k] : (v >= g.L[k] ? v - g.L[k] : v);
  }
  int dom, s;
  coords_to_internal(g, y, dom, s);
  const int4* p = U + (((size_t)((dom * 4 + dir) * 9)) << g.logvd) + s;
  const int row = dag ? 1 : 3, col = dag ? 3 : 1, sg = dag ? -1 : 0;
  FxMat m;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 v = __ldg(p + ((size_t)(i * row + j * col) << g.logvd));
      m.rh[i][j] = v.x;
      m.rl[i][j] = v.y;
      m.ih[i][j] = (v.z ^ sg) - sg;
      m.il[i][j] = (v.w ^ sg) - sg;
    }
  return m;
}

// The link U_mu(x) belongs to two of x's leaves in the mu-nu plane and to two
// of x + e_mu's, through the same two staples: with
//   D = X - Y^dag,  X = U_nu(x+mu) U_mu^dag(x+nu) U_nu^dag(x),
//                   Y = U_nu^dag(x-nu) U_mu(x-nu) U_nu(x+mu-nu),
// Q - Q^dag of a site is [M - M^dag] over M = U_mu D at x and M = D U_mu at
// x - e_mu.  So a thread forms the staples of one link and plane (four matrix
// products) and both its M (one each, as U D and U^dag D^dag, whose
// anti-Hermitian part is minus that of D U): six products per site and plane,
// not the ten of a site's own leaves taken in pairs.  own and next get
// 2^61 times the nine reals of this site's share and of x + e_mu's: the
// imaginary parts of the diagonal, then (re, im) of the entries 01, 02, 12.
// X and Y, and the two M, are loops over the same code, whose instructions
// then fit the cache; X, then D, wait in shared memory (stash, this thread's
// column of a [18][FS_THREADS] array).
constexpr int FS_THREADS = 128;
struct PathLink {  // direction (0 mu, 1 nu), offsets along mu and nu, adjoint
  signed char dir, dm, dn, dag;
};
__constant__ PathLink c_path[6] = {  // X's three links, Y's three
    {1, 1, 0, 0}, {0, 0, 1, 1}, {1, 0, 0, 1}, {1, 0, -1, 1}, {0, 0, -1, 0}, {1, 1, -1, 0}};
template <typename Store>
__device__ __forceinline__ void field_strength_fx(const Geom& g, const int4* U, const int x[4], int mu, int nu,
                                                  long long* stash, const Store& store) {
  auto link = [&](int k) {
    const PathLink q = c_path[k];
    return fx_link(g, U, x, mu, nu, q.dm, q.dn, q.dir ? nu : mu, q.dag != 0);
  };
  FxSum P;
  FxMat t;
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    fx_mul(link(3 * q), link(3 * q + 1), P);
    fx_limbs(P, t);
    fx_mul(t, link(3 * q + 2), P);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        long long *re = stash + 2 * (3 * i + j) * FS_THREADS, *im = re + FS_THREADS;
        if (q == 0) {
          *re = P.re[i][j];
          *im = P.im[i][j];
        } else {  // D = X - Y^dag
          *re -= P.re[j][i];
          *im += P.im[j][i];
        }
      }
  }
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    // U D, then U^dag D^dag
    const int row = h ? 1 : 3, col = h ? 3 : 1;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const long long* d = stash + 2 * (row * i + col * j) * FS_THREADS;
        P.re[i][j] = d[0];
        P.im[i][j] = h ? -d[FS_THREADS] : d[FS_THREADS];
      }
    fx_limbs(P, t);
    fx_mul(fx_link(g, U, x, mu, nu, 0, 0, mu, h != 0), t, P);
    long long f[9];
#pragma unroll
    for (int i = 0; i < 3; ++i) f[i] = 2 * P.im[i][i];
    int o = 3;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i + 1; j < 3; ++j) {
        f[o++] = P.re[i][j] - P.re[j][i];
        f[o++] = P.im[i][j] + P.im[j][i];
      }
    if (h)
#pragma unroll
      for (int e = 0; e < 9; ++e) f[e] = -f[e];
    store(h, f);
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

// the same through the pivoted elimination, in place (element k at
// k stride; zero if singular)
__device__ __noinline__ bool invert6_general(double* r, int stride) {
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
    r[i * stride] = ok ? inv[i][i].re : 0.0;
    for (int j = i + 1; j < 6; ++j) {
      const int o = 6 + 2 * herm_off(i, j);
      r[o * stride] = ok ? 0.5 * (inv[i][j].re + inv[j][i].re) : 0.0;
      r[(o + 1) * stride] = ok ? 0.5 * (inv[i][j].im - inv[j][i].im) : 0.0;
    }
  }
  return ok;
}

// a chiral block of 1 + C from kc A_1, kc A_2, kc A_3 (nine reals each):
// 1 + [[H_3, H_1 - i H_2], [H_1 + i H_2, -H_3]], H_k = i kc A_k Hermitian
__device__ __forceinline__ void pack_block(const double a1[9], const double a2[9], const double a3[9],
                                           double m[36]) {
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
// the kernels
// ---------------------------------------------------------------------------
struct CloverOut {
  double2 *clov64, *cinv64;   // [dom][36][vd]
  float4 *clov32, *cinv32;    // [dom][18][vd]
  __half2* cinv16;            // [dom][36][vd]
  float4* clovdf;             // [dom][36][vd], double-float
  uint4* st16;                // staging of the SAP block kernel (4^4 domains, else null): [dom][site][9]
  float4* st32;               // [dom][site][19]
};

// F between the kernels: a plane's nine reals in five pairs (the last half
// filled), pair 5 plane + k of [dom][36][vd]: float64 in the buffer of 1 + C
// (each site's own entries, which 1 + C overwrites), or fixed point, the
// site's own share there and the next site's in a second buffer
constexpr int F_PAIRS = 5;
__host__ __device__ constexpr int plane_mu(int p) { return p < 3 ? 0 : (p < 5 ? 1 : 2); }
__host__ __device__ constexpr int plane_nu(int p) { return p < 3 ? p + 1 : (p < 5 ? p - 1 : 3); }

// A warp takes 32 consecutive sites (in lexicographic-domain order, so that
// neighbouring domains' links are still in L2) and one plane; the six planes
// of a tile are consecutive warps and share its links through L1.  No
// barrier, so that the warps' loads and products overlap (phases of one fused
// kernel, with its barriers, left the multipliers two thirds idle).
template <bool FIXED>
__global__ void __launch_bounds__(FS_THREADS, 3) field_strength_kernel(Geom g, const int4* __restrict__ ufx,
                                                                       LinkPtr<double> U, double2* out,
                                                                       longlong2* next) {
  __shared__ long long stash[FIXED ? 18 * FS_THREADS : 1];
  const int lane = threadIdx.x & 31;
  const long long item = blockIdx.x * (long long)(FS_THREADS / 32) + (threadIdx.x >> 5);
  const int p = (int)(item % 6);
  const long long gid = item / 6 * 32 + lane;
  if (gid >= g.vol) return;
  int x[4], lex = (int)(gid >> g.logvd);
  const int s = (int)(gid & (g.vd - 1));
  const int dom = __ldg(g.lex2dom + lex);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const int q = lex / g.nd[mu];
    x[mu] = (lex - q * g.nd[mu]) * g.d[mu] + ((s >> g.shift[mu]) & (g.d[mu] - 1));
    lex = q;
  }
  const int mu = plane_mu(p), nu = plane_nu(p);
  const size_t at = (((size_t)(dom * 36 + F_PAIRS * p)) << g.logvd) + s;
  if (FIXED) {
    field_strength_fx(g, ufx, x, mu, nu, stash + threadIdx.x, [&](int h, const long long f[9]) {
      longlong2* q = (h ? next : reinterpret_cast<longlong2*>(out)) + at;
#pragma unroll
      for (int k = 0; k < F_PAIRS; ++k) q[(size_t)k << g.logvd] = make_longlong2(f[2 * k], k < 4 ? f[2 * k + 1] : 0);
    });
  } else {
    double f[10];
    f[9] = 0.0;
    field_strength(g, U, x, mu, nu, f);
#pragma unroll
    for (int k = 0; k < F_PAIRS; ++k) out[at + ((size_t)k << g.logvd)] = make_double2(f[2 * k], f[2 * k + 1]);
  }
}

// float64 rounded to float32 on the bit fields (conversions would queue on
// the float64 pipe); what lies outside float32's normal range is converted
__device__ __forceinline__ float to_float(double d) {
  const unsigned e = ((unsigned)__double2hiint(d) >> 20) & 0x7FFu;
  if (e != 0 && e - (1023 - 126) >= 254) return (float)d;
  return df64_from_double_scaled(d, 0).hi;
}

// F of a plane at a site, fixed point: the site's own share and the one that
// the thread of the site before it along mu left
__device__ __forceinline__ void fx_plane(const Geom& g, const double2* own, const longlong2* __restrict__ next, int dom,
                                         int s, int p, long long f[10]) {
  const int mu = plane_mu(p), step = 1 << g.shift[mu];
  const bool inside = ((s >> g.shift[mu]) & (g.d[mu] - 1)) > 0;
  const int bd = inside ? dom : __ldg(g.nbr + dom * 8 + 2 * mu + 1);
  const int bs = inside ? s - step : s + (g.d[mu] - 1) * step;
  const longlong2* u = reinterpret_cast<const longlong2*>(own) + (((size_t)(dom * 36 + F_PAIRS * p)) << g.logvd) + s;
  const longlong2* v = next + (((size_t)(bd * 36 + F_PAIRS * p)) << g.logvd) + bs;
#pragma unroll
  for (int k = 0; k < F_PAIRS; ++k) {
    const longlong2 a = u[(size_t)k << g.logvd], b = __ldg(v + ((size_t)k << g.logvd));
    f[2 * k] = a.x + b.x;
    f[2 * k + 1] = a.y + b.y;
  }
}

// Threads (site, block): warps 0 and 1 the two blocks of 32 sites, warps 2
// and 3 those of the next 32.  The float64 pipe bounds it (the inversion);
// every component it writes is one stream over the warp's sites, only the
// site-major staging rows go through shared memory.
constexpr int CB_THREADS = 128;
constexpr int CB_SITES = CB_THREADS / 2;
constexpr int CB_ROW = 73;  // floats per site in shared memory, odd: no bank conflicts
template <bool FIXED>
__global__ void __launch_bounds__(CB_THREADS, 4) clover_build_kernel(Geom g, double kc, CloverOut o,
                                                                     const longlong2* __restrict__ next, int* status) {
  __shared__ float stage[CB_SITES * CB_ROW];
  __shared__ double rows[36 * CB_THREADS];  // the pivoted inversion's operand and result
  const int b = (threadIdx.x >> 5) & 1;
  const int local = (threadIdx.x & 31) + (threadIdx.x >> 6) * 32;
  const long long n0 = blockIdx.x * (long long)CB_SITES;
  const bool live = n0 + local < g.vol;
  const long long gid = live ? n0 + local : n0;
  const int dom = (int)(gid >> g.logvd), s = (int)(gid & (g.vd - 1));
  const size_t at = ((size_t)dom * 36 << g.logvd) + s;
  double m[36];
  {
    // A_k = +- F_p + or - F_q, planes 0 xy, 1 xz, 2 xt, 3 yz, 4 yt, 5 zt; the
    // upper sign of F_p in block 0
    constexpr int P[3] = {2, 4, 5}, Q[3] = {3, 1, 0};
    double a[3][9];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (FIXED) {
        // exact sums of 62 bits at most, converted once; 2^-61 comes with kc
        long long f[10], h[10];
        fx_plane(g, o.clov64, next, dom, s, P[k], f);
        fx_plane(g, o.clov64, next, dom, s, Q[k], h);
#pragma unroll
        for (int e = 0; e < 9; ++e) {
          const long long v = b == 0 ? f[e] : -f[e];
          a[k][e] = kc * (double)(k == 1 ? v + h[e] : v - h[e]);
        }
      } else {
        const double sg = b == 0 ? 1.0 : -1.0;
        double f[10], h[10];
#pragma unroll
        for (int i = 0; i < F_PAIRS; ++i) {
          const double2 u = o.clov64[at + ((size_t)(F_PAIRS * P[k] + i) << g.logvd)];
          const double2 v = o.clov64[at + ((size_t)(F_PAIRS * Q[k] + i) << g.logvd)];
          f[2 * i] = u.x; f[2 * i + 1] = u.y;
          h[2 * i] = v.x; h[2 * i + 1] = v.y;
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) a[k][e] = kc * fma(sg, f[e], k == 1 ? h[e] : -h[e]);
      }
    }
    pack_block(a[0], a[1], a[2], m);
  }
  __syncthreads();  // every F of the block is read before 1 + C overwrites it
  if (live) {
#pragma unroll
    for (int k = 0; k < 18; ++k) {
      const size_t i = at + ((size_t)(18 * b + k) << g.logvd);
      o.clov64[i] = make_double2(m[2 * k], m[2 * k + 1]);
      const df64 d0 = df64_from_double_scaled(m[2 * k], 0), d1 = df64_from_double_scaled(m[2 * k + 1], 0);
      o.clovdf[i] = make_float4(d0.hi, d0.lo, d1.hi, d1.lo);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k)
      o.clov32[((size_t)(dom * 18 + 9 * b + k) << g.logvd) + s] =
          make_float4(to_float(m[4 * k]), to_float(m[4 * k + 1]), to_float(m[4 * k + 2]), to_float(m[4 * k + 3]));
  }
  double* row = rows + threadIdx.x;
#pragma unroll
  for (int k = 0; k < 36; ++k) row[k * CB_THREADS] = m[k];
  bool ok = invert6_packed(m);
  if (!ok) {
    ok = invert6_general(row, CB_THREADS);
#pragma unroll
    for (int k = 0; k < 36; ++k) m[k] = row[k * CB_THREADS];
  }
  bool finite = true;
#pragma unroll
  for (int k = 0; k < 36; ++k) finite = finite && isfinite(m[k]);
  if (live && !(ok && finite)) atomicExch(status, 1);
  float* st = stage + local * CB_ROW + 36 * b;
  if (live) {
#pragma unroll
    for (int k = 0; k < 18; ++k) {
      const size_t i = at + ((size_t)(18 * b + k) << g.logvd);
      const float q0 = to_float(m[2 * k]), q1 = to_float(m[2 * k + 1]);
      o.cinv64[i] = make_double2(m[2 * k], m[2 * k + 1]);
      o.cinv16[i] = __floats2half2_rn(q0, q1);
      st[2 * k] = q0;
      st[2 * k + 1] = q1;
    }
#pragma unroll
    for (int k = 0; k < 9; ++k)
      o.cinv32[((size_t)(dom * 18 + 9 * b + k) << g.logvd) + s] =
          make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
  }
  if (!o.st16) return;
  // 4^4 domains: every block is full, its sites are consecutive sites of one
  // domain, and so are their rows in the staging layouts
  __syncthreads();
  for (int i = threadIdx.x; i < CB_SITES * 9; i += CB_THREADS) {
    const float* q = stage + i / 9 * CB_ROW + 8 * (i % 9);
    __half2 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2half2_rn(q[2 * e], q[2 * e + 1]);
    o.st16[n0 * 9 + i] = *reinterpret_cast<const uint4*>(h);
  }
  for (int i = threadIdx.x; i < CB_SITES * 19; i += CB_THREADS) {
    const float* q = stage + i / 19 * CB_ROW + 4 * (i % 19);
    o.st32[n0 * 19 + i] = i % 19 < 18 ? make_float4(q[0], q[1], q[2], q[3]) : make_float4(0.f, 0.f, 0.f, 0.f);
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
// (their entries are bounded by one) and not near the diagonal anywhere; any
// others (fields near the identity, and whatever a caller sets with the check
// switched off) take the float64 products.  24^3 x 48: 3.3 ms in fixed point,
// 10.1 ms in float64.  Error of the off-diagonal part of 1 + C on links
// exp(i eps H), fixed point against float64: 4.9e-16 and 4.8e-16 at eps 0.05,
// 5.0e-16 and 4.8e-16 at 0.02, 2.2e-15 and 4.8e-16 at 1e-3, 2e-12 at 1e-6: in
// steps of 2^-58 whatever the entries' size.
void build_clover_launch(qcd_ctx* ctx, cudaStream_t st) {
  const Geom& g = ctx->geom;
  const CloverOut o{ctx->clov64, ctx->cinv64, ctx->clov32, ctx->cinv32, ctx->cinv16, ctx->clovdf,
                    (uint4*)ctx->st_clov16, (float4*)ctx->st_clov32};
  const int grid = grid_for((g.vol + 31) / 32 * 6, FS_THREADS / 32);
  const LinkPtr<double> U{ctx->u64};
  const double kc = ctx->kappa * ctx->csw;
  const int sites = grid_for(g.vol, CB_SITES);
  auto launch = [&](auto kernel, int blocks, int threads, auto... args) {
    LaunchScope ls(ctx, QCD_KC_OTHER, st);
    kernel<<<blocks, threads, 0, st>>>(args...);
    check_launch();
  };
  if (ctx->fixed_clover) {
    // scratch: the limbs where 1 + C goes in double-float, the next sites'
    // shares of F where the double-float links go once the clover term is built
    int4* ufx = reinterpret_cast<int4*>(ctx->clovdf);
    longlong2* next = reinterpret_cast<longlong2*>(ctx->udf);
    launch(links_to_fixed_kernel, 1216, 256, ctx->u64, ufx, (size_t)g.vol * 36);
    launch(field_strength_kernel<true>, grid, FS_THREADS, g, ufx, U, ctx->clov64, next);
    launch(clover_build_kernel<true>, sites, CB_THREADS, g, kc / (double)(8LL << FX_FRAC), o, next, ctx->d_status);
  } else {
    launch(field_strength_kernel<false>, grid, FS_THREADS, g, nullptr, U, ctx->clov64, nullptr);
    launch(clover_build_kernel<false>, sites, CB_THREADS, g, kc, o, nullptr, ctx->d_status);
  }
}

}  // namespace qcd
