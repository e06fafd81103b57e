// The operator kernel with one right-hand side per thread, shared by
// dslash.cu and dslash_mrhs.cu (several right-hand sides on 4^4 blocks).
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

template <typename R>
struct Prec;
template <>
struct Prec<float> {
  using SIO = F32Spinor;
  using LP = LinkPtr<float>;
  using CP = CloverPtrF32;
  using CB = CloverBlockF32;
};
template <>
struct Prec<double> {
  using SIO = F64Spinor;
  using LP = LinkPtr<double>;
  using CP = CloverPtrF64;
  using CB = CloverBlockF64;
};
template <>
struct Prec<df64> {
  using SIO = DF64Spinor;
  using LP = LinkPtr<df64>;
  using CP = CloverPtrDF64;
  using CB = CloverBlockDF64;
};

// The geometry of 4^4 storage blocks as constants of the compiled kernel
// (D4): every stride is then an immediate offset of a load.  Only the kernels
// for several right-hand sides use it, which issue binds; with one, HBM does,
// and the registers of the wider schedule cost more than they save (32^4: 0.1224 ms
// against 0.1204, 24^3 x 32: 54.9 us against 52.7).
template <bool D4>
__device__ __forceinline__ void fix_geom(Geom& g) {
  if constexpr (D4) {
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      g.d[mu] = 4;
      g.logd[mu] = 2;
      g.shift[mu] = 2 * mu;
    }
    g.vd = 256;
    g.logvd = 8;
  }
}

// Both hops of direction MU without branches: the neighbour (domain, site)
// and the boundary sign are selected, not branched on, so that the loads of
// all eight hops are independent straight-line code the compiler can issue
// early (the operator is bound by how many loads are in flight).  nb holds
// the eight neighbour domains of dom, tf its boundary-sign flags.
template <int MU, int PMF, int PMB, bool FIRST, typename R, typename SIO, typename LP>
__device__ __forceinline__ void hop_dir_bf(const Geom& g, const SIO& in, const LP& U, int dom, int s, int rhs_off,
                                           const int nb[8], int tf, Spinor<R>& acc) {
  static_assert(!FIRST || MU < 3, "the first hop must carry no boundary sign");
  const int c = (s >> g.shift[MU]) & (g.d[MU] - 1);
  const int step = 1 << g.shift[MU];
  const int span = (g.d[MU] - 1) * step;
  {
    const bool inside = c < g.d[MU] - 1;
    const int nd = inside ? dom : nb[2 * MU];
    const int ns = inside ? s + step : s - span;
    const R f = (!inside && ((tf >> (2 * MU)) & 1)) ? R(g.bc_t) : R(1.0f);
    Spinor<R> p;
    in.load(g, nd + rhs_off, ns, p);
    HalfSpinor<R> h, uh;
    project<MU, PMF>(p, h);
    SU3<R> u;
    U.load(g, dom, MU, s, u);
    su3_mul(u, h, uh);
    if (FIRST) rebuild<MU, PMF>(acc, uh);  // f = 1: the sign is for t hops only
    else accumulate<MU, PMF>(acc, uh, f);
  }
  {
    const bool inside = c > 0;
    const int nd = inside ? dom : nb[2 * MU + 1];
    const int ns = inside ? s - step : s + span;
    const R f = (!inside && ((tf >> (2 * MU + 1)) & 1)) ? R(g.bc_t) : R(1.0f);
    Spinor<R> p;
    in.load(g, nd + rhs_off, ns, p);
    HalfSpinor<R> h, uh;
    project<MU, PMB>(p, h);
    SU3<R> u;
    U.load(g, nd, MU, ns, u);
    su3_dag_mul(u, h, uh);
    accumulate<MU, PMB>(acc, uh, f);
  }
}

template <int PMF, int PMB, typename R, typename SIO, typename LP>
__device__ __forceinline__ void hopping_bf(const Geom& g, const SIO& in, const LP& U, int dom, int s, int rhs_off,
                                           Spinor<R>& acc) {
  int nb[8];
  const int4 n0 = __ldg(reinterpret_cast<const int4*>(g.nbr) + 2 * dom);
  const int4 n1 = __ldg(reinterpret_cast<const int4*>(g.nbr) + 2 * dom + 1);
  nb[0] = n0.x; nb[1] = n0.y; nb[2] = n0.z; nb[3] = n0.w;
  nb[4] = n1.x; nb[5] = n1.y; nb[6] = n1.z; nb[7] = n1.w;
  const int tf = __ldg(g.tflag + dom);
  hop_dir_bf<0, PMF, PMB, true>(g, in, U, dom, s, rhs_off, nb, tf, acc);  // starts the sum
  hop_dir_bf<1, PMF, PMB, false>(g, in, U, dom, s, rhs_off, nb, tf, acc);
  hop_dir_bf<2, PMF, PMB, false>(g, in, U, dom, s, rhs_off, nb, tf, acc);
  hop_dir_bf<3, PMF, PMB, false>(g, in, U, dom, s, rhs_off, nb, tf, acc);
}

// D:    out = (1 + C) x - kappa H x
// D^dag: out = (1 + C) x - kappa H^dag x   (gamma_5 H gamma_5 swaps the projectors)
// A:    out = x - kappa C_inv H x
//
// Launch shape: THREADS per block, at least MINB blocks per SM (a register
// budget); the autotuner picks among the instantiated shapes.  Blocks are
// numbered rhs-fastest, so the nrhs blocks that share a tile of sites (and
// its links and clover) run back to back and reuse them from L2.
// One site (lexicographic-domain index gid) of one right-hand side.
template <typename R, int MODE, bool HINT = false, typename LP = typename Prec<R>::LP>
__device__ __forceinline__ void dslash_site(const Geom& g, const typename Prec<R>::SIO& out,
                                            const typename Prec<R>::SIO& in, const LP& U,
                                            const typename Prec<R>::CP& clov, R kappa, long long gid, int rhs) {
  // domains are visited in lexicographic order, so that the neighbouring
  // domains whose surface spinors a domain reads are processed at about the
  // same time and their data is still in L2
  const int dom = __ldg(g.lex2dom + (int)(gid >> g.logvd));
  const int s = (int)(gid & (g.vd - 1));
  const int rhs_off = rhs * g.ndom;
  Spinor<R> acc;
  if (MODE == MODE_DDAG) hopping_bf<+1, -1>(g, in, U, dom, s, rhs_off, acc);
  else hopping_bf<-1, +1>(g, in, U, dom, s, rhs_off, acc);
  Spinor<R> x;
  in.load(g, dom + rhs_off, s, x);
  if constexpr (HINT) {
    const CloverPtrF32Stream cs{clov.p};
    clover_mul<R, CloverPtrF32Stream, typename Prec<R>::CB>(cs, g, dom, s, MODE == MODE_A ? acc : x);
  } else if (MODE == MODE_A) {
    clover_mul<R, typename Prec<R>::CP, typename Prec<R>::CB>(clov, g, dom, s, acc);
  } else {
    clover_mul<R, typename Prec<R>::CP, typename Prec<R>::CB>(clov, g, dom, s, x);
  }
#pragma unroll
  for (int sp = 0; sp < 4; ++sp)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x.v[sp][c].re = fma(-kappa, acc.v[sp][c].re, x.v[sp][c].re);
      x.v[sp][c].im = fma(-kappa, acc.v[sp][c].im, x.v[sp][c].im);
    }
  if constexpr (HINT) out.store_stream(g, dom + rhs_off, s, x);
  else out.store(g, dom + rhs_off, s, x);
}

// HINT: the clover rows and the output, touched once per application, are
// read and written with the streaming (evict-first) cache operators, so
// that L2 keeps the spinor and link lines that neighbouring sites read
// again.  float32 only.  LP: the links' storage (LinkPtr12: the first two
// rows of SU(3) links, float32 only).
template <typename R, int MODE, int THREADS, int MINB, bool HINT, typename LP, bool D4>
__global__ void __launch_bounds__(THREADS, MINB)
    dslash_kernel(Geom g, typename Prec<R>::SIO out, typename Prec<R>::SIO in, LP U, typename Prec<R>::CP clov,
                  R kappa, int nrhs) {
  fix_geom<D4>(g);
  const int rhs = blockIdx.x % nrhs;
  const long long gid = (blockIdx.x / nrhs) * (long long)THREADS + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (gid >= g.vol || loop_idle(g)) return;
  dslash_site<R, MODE, HINT, LP>(g, out, in, U, clov, kappa, gid, rhs);
}

template <typename R, int MODE, int THREADS, int MINB, bool HINT = false, typename LP = typename Prec<R>::LP,
          bool D4 = false>
void launch_dslash_shape(const Geom& g, void* out, const void* in, const void* U, const void* clov, R kappa,
                         int nrhs, cudaStream_t st, bool pdl) {
  using P = Prec<R>;
  const long long blocks = (long long)grid_for(g.vol, THREADS) * nrhs;
  QCD_REQUIRE(blocks < (1LL << 31), QCD_ERR_ARG, "lattice too large for one launch");
  const typename P::SIO o{(decltype(P::SIO::p))out}, i{(decltype(P::SIO::p))in};
  const LP u{(decltype(LP::p))U};
  const typename P::CP c{(decltype(P::CP::p))clov};
  auto kernel = dslash_kernel<R, MODE, THREADS, MINB, HINT, LP, D4>;
  if (pdl) launch_pdl(kernel, dim3((unsigned)blocks), dim3(THREADS), 0, st, g, o, i, u, c, kappa, nrhs);
  else kernel<<<(unsigned)blocks, THREADS, 0, st>>>(g, o, i, u, c, kappa, nrhs);
}

}  // namespace qcd
