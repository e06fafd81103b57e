// D, D^dag and A = C_inv D (App. A and Sec. 3 of arXiv:2109.10687) in float32
// on several right-hand sides: with one right-hand side per thread
// (dslash.cuh) and with two.  4^4 storage blocks.

#include <cstdio>

#include "dslash.cuh"

namespace qcd {

// Two right-hand sides per thread (kRhs): each link and clover block is read
// through L2 once for both, and the two spinors of a hop are independent
// loads, which keeps more bytes in flight than the fewer warps cost.  An odd
// last right-hand side is computed twice and stored once.  The arithmetic of
// a right-hand side is that of dslash_site, bit for bit.
//
// With several right-hand sides the operator is bound by issue and by the
// latency of the spinor gathers, not by HBM: one per thread with strides
// known at run time issued 2.3 k instructions per site and right-hand side
// in 66 % of the cycles, a quarter of them index arithmetic.  24^3 x 32, 12
// right-hand sides, links as 12 reals: D^dag 0.460 ms with run-time strides,
// 0.443 (128x4) and 0.4295 (128x5) with the geometry compiled in, 0.4253
// with pairs as well (A: 0.438 and 0.413).  Pairs of right-hand sides with
// run-time strides (0.470), three and four per thread (0.539, 0.502) and a
// kernel that stages a domain's links and spinors in shared memory (0.467:
// one block per SM, latency) were slower.
constexpr int kRhs = 2;

template <int MU, int PM, bool FIRST, typename LP>
__device__ __forceinline__ void hop_mrhs(const Geom& g, const F32Spinor& in, const LP& U, int dom, int s,
                                         const int off[kRhs], const int nb[8], int tf, Spinor<float> acc[kRhs], bool fwd) {
  const int c = (s >> g.shift[MU]) & (g.d[MU] - 1);
  const int step = 1 << g.shift[MU];
  const int span = (g.d[MU] - 1) * step;
  const bool inside = fwd ? c < g.d[MU] - 1 : c > 0;
  const int k = 2 * MU + (fwd ? 0 : 1);
  const int nd = inside ? dom : nb[k];
  const int ns = inside ? (fwd ? s + step : s - step) : (fwd ? s - span : s + span);
  const float f = (MU == 3 && !inside && ((tf >> k) & 1)) ? (float)g.bc_t : 1.0f;
  SU3<float> u;
  if (fwd) U.load(g, dom, MU, s, u);
  else U.load(g, nd, MU, ns, u);
#pragma unroll
  for (int r = 0; r < kRhs; ++r) {
    Spinor<float> p;
    in.load(g, nd + off[r], ns, p);
    HalfSpinor<float> h, uh;
    project<MU, PM>(p, h);
    if (fwd) su3_mul(u, h, uh);
    else su3_dag_mul(u, h, uh);
    if (FIRST) rebuild<MU, PM>(acc[r], uh);
    else accumulate<MU, PM>(acc[r], uh, f);
  }
}

template <int MODE, int THREADS, int MINB, typename LP>
__global__ void __launch_bounds__(THREADS, MINB)
    dslash_mrhs_kernel(Geom g, F32Spinor out, F32Spinor in, LP U, CloverPtrF32 clov, float kappa, int nrhs,
                       int groups) {
  fix_geom<true>(g);
  constexpr int PMF = MODE == MODE_DDAG ? +1 : -1, PMB = -PMF;
  const int group = blockIdx.x % groups;  // fastest: the groups of a tile share its operator in L2
  const long long gid = (blockIdx.x / groups) * (long long)THREADS + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (gid >= g.vol || loop_idle(g)) return;
  const int dom = __ldg(g.lex2dom + (int)(gid >> g.logvd));
  const int s = (int)(gid & (g.vd - 1));
  int off[kRhs], nb[8];
#pragma unroll
  for (int r = 0; r < kRhs; ++r) off[r] = min(group * kRhs + r, nrhs - 1) * g.ndom;
  const int4 n0 = __ldg(reinterpret_cast<const int4*>(g.nbr) + 2 * dom);
  const int4 n1 = __ldg(reinterpret_cast<const int4*>(g.nbr) + 2 * dom + 1);
  nb[0] = n0.x; nb[1] = n0.y; nb[2] = n0.z; nb[3] = n0.w;
  nb[4] = n1.x; nb[5] = n1.y; nb[6] = n1.z; nb[7] = n1.w;
  const int tf = __ldg(g.tflag + dom);
  Spinor<float> acc[kRhs];
  hop_mrhs<0, PMF, true>(g, in, U, dom, s, off, nb, tf, acc, true);
  hop_mrhs<0, PMB, false>(g, in, U, dom, s, off, nb, tf, acc, false);
  hop_mrhs<1, PMF, false>(g, in, U, dom, s, off, nb, tf, acc, true);
  hop_mrhs<1, PMB, false>(g, in, U, dom, s, off, nb, tf, acc, false);
  hop_mrhs<2, PMF, false>(g, in, U, dom, s, off, nb, tf, acc, true);
  hop_mrhs<2, PMB, false>(g, in, U, dom, s, off, nb, tf, acc, false);
  hop_mrhs<3, PMF, false>(g, in, U, dom, s, off, nb, tf, acc, true);
  hop_mrhs<3, PMB, false>(g, in, U, dom, s, off, nb, tf, acc, false);
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    CloverBlockF32 blk;
    clov.load_block(g, dom, s, b, blk);
#pragma unroll
    for (int r = 0; r < kRhs; ++r) {
      cx<float> x[6], h[6], y[6];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 v = __ldg(in.p + in.idx(g, dom + off[r], 3 * b + k, s));
        x[2 * k] = make_cx(v.x, v.y);
        x[2 * k + 1] = make_cx(v.z, v.w);
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) h[i] = acc[r].v[2 * b + i / 3][i % 3];
      if (MODE == MODE_A) {
        herm6_mul<float>(blk, h, y);
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = make_cx(fma(-kappa, y[i].re, x[i].re), fma(-kappa, y[i].im, x[i].im));
      } else {
        herm6_mul<float>(blk, x, y);
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = make_cx(fma(-kappa, h[i].re, y[i].re), fma(-kappa, h[i].im, y[i].im));
      }
      if (group * kRhs + r < nrhs) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
          __stcs(out.p + out.idx(g, dom + off[r], 3 * b + k, s),
                 make_float4(y[2 * k].re, y[2 * k].im, y[2 * k + 1].re, y[2 * k + 1].im));
      }
    }
  }
}

template <int MODE, int THREADS, int MINB, typename LP>
static void launch_mrhs_shape(const Geom& g, void* out, const void* in, const void* U, const void* clov, float kappa,
                              int nrhs, cudaStream_t st, bool pdl) {
  const int groups = (nrhs + kRhs - 1) / kRhs;
  const long long blocks = (long long)grid_for(g.vol, THREADS) * groups;
  QCD_REQUIRE(blocks < (1LL << 31), QCD_ERR_ARG, "lattice too large for one launch");
  const F32Spinor o{(float4*)out}, i{(float4*)in};
  const LP u{(decltype(LP::p))U};
  const CloverPtrF32 c{(const float4*)clov};
  auto kernel = dslash_mrhs_kernel<MODE, THREADS, MINB, LP>;
  if (pdl) launch_pdl(kernel, dim3((unsigned)blocks), dim3(THREADS), 0, st, g, o, i, u, c, kappa, nrhs, groups);
  else kernel<<<(unsigned)blocks, THREADS, 0, st>>>(g, o, i, u, c, kappa, nrhs, groups);
}

// One right-hand side per thread, the right-hand sides of a tile in
// neighbouring blocks, or two per thread.
template <int MODE, typename LP>
static void launch_dslash_mrhs(int variant, const Geom& g, void* out, const void* in, const void* U, const void* clov,
                               float kappa, int nrhs, cudaStream_t st, bool pdl) {
  switch (variant) {
    case 0: launch_dslash_shape<float, MODE, 128, 4, false, LP, true>(g, out, in, U, clov, kappa, nrhs, st, pdl); break;
    case 1: launch_dslash_shape<float, MODE, 128, 5, false, LP, true>(g, out, in, U, clov, kappa, nrhs, st, pdl); break;
    case 2: launch_mrhs_shape<MODE, 128, 3, LP>(g, out, in, U, clov, kappa, nrhs, st, pdl); break;
    default: launch_mrhs_shape<MODE, 128, 4, LP>(g, out, in, U, clov, kappa, nrhs, st, pdl); break;
  }
}
static const char* kShapes[] = {"128x4", "128x5", "128x3r2", "128x4r2"};
static const char* kShapes12[] = {"128x4c", "128x5c", "128x3r2c", "128x4r2c"};  // links as 12 reals
constexpr int kNumShapes = 4, kDefaultPair = 3;

// The shape without tuning.  A pair per thread needs the launch's blocks to
// be several per slot (152 SMs x 4) and few idle halves: at 16^4 with 12
// right-hand sides (3072 blocks of pairs) A takes 0.0672 ms against 0.0684,
// but on 8^4 with 4 (64 blocks) 8.4 us against 5.0, and with 3 right-hand
// sides (a quarter of the pairs' work spare) 0.139 ms against 0.1215.  With an
// odd number of them the line lies between 11 and 13 (24^3 x 32, pairs against
// one per thread: D 0.4145 and 0.4095 ms with 11, 0.4840 and 0.4921 with 13,
// 0.5514 and 0.5501 with 15, 0.6188 and 0.6344 with 17; A 0.4052 and 0.4037
// with 11, 0.4728 and 0.4873 with 13).
static int default_shape(const Geom& g, int nrhs) {
  const int pairs = (nrhs + 1) / 2;
  const bool few_spare = nrhs % 2 == 0 || nrhs > 12;
  return few_spare && (long long)grid_for(g.vol, 128) * pairs >= 5 * 152 * 4 ? kDefaultPair : 0;
}

bool dslash_mrhs_fits(const Geom& g, int nrhs) {
  return nrhs > 1 && g.d[0] == 4 && g.d[1] == 4 && g.d[2] == 4 && g.d[3] == 4;
}

void dslash_mrhs_launch(qcd_ctx* ctx, void* out, const void* in, int mode, int nrhs, bool use12, cudaStream_t st,
                        bool pdl) {
  const Geom& g = ctx->geom;
  const float k = (float)ctx->kappa;
  const void* clov = mode == MODE_A ? (const void*)ctx->cinv32 : (const void*)ctx->clov32;
  const void* links = use12 ? (const void*)ctx->u32c : (const void*)ctx->u32;
  auto run = [&](int v) {
    auto by_mode = [&](auto lp) {
      using LP = decltype(lp);
      if (mode == MODE_A) launch_dslash_mrhs<MODE_A, LP>(v, g, out, in, links, clov, k, nrhs, st, pdl);
      else if (mode == MODE_D) launch_dslash_mrhs<MODE_D, LP>(v, g, out, in, links, clov, k, nrhs, st, pdl);
      else launch_dslash_mrhs<MODE_DDAG, LP>(v, g, out, in, links, clov, k, nrhs, st, pdl);
    };
    if (use12) by_mode(LinkPtr12{});
    else by_mode(LinkPtr<float>{});
    check_launch();
  };
  char key[64];
  std::snprintf(key, sizeof key, "dslash_f32_mode%d_nrhs%d%s", mode, nrhs, use12 ? "_links12" : "");
  const int v = tune_pick(ctx, key, kNumShapes, use12 ? kShapes12 : kShapes, run, st, default_shape(g, nrhs));
  LaunchScope ls(ctx, QCD_KC_DSLASH, st);
  run(v);
}

}  // namespace qcd
