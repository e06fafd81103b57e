// SAP half-sweep on storage-block domains of any shape but 4^4 (Sec. 3 of
// arXiv:2109.10687, Algorithms 1 and 2): one thread per site, several domains
// per block.
//
// Per launch, for the domains of one colour c: the surface term
// s <- s + kappa C_inv H_cc' x_c', n_jac Jacobi sweeps
// x <- s + kappa C_inv H_cc x, the residual update
// s <- s + b - x + kappa C_inv H_cc x (not in the closing sweep), and x_c to
// memory.
//
// What bounds it: with a thread per site these lattices leave about two warps
// per scheduler, so the time is that of one warp's chain of instructions.
// The operator of the block's sites (consecutive in memory) is therefore
// copied to shared memory first, asynchronously and ahead of the wait for the
// previous launch, and a direction in which a domain is two sites wide has
// one hop body instead of two: each site has exactly one neighbour inside and
// one outside, forward or backward by its coordinate, and the projector's
// sign and the adjoint of the link are taken per lane (the adjoint by reading
// the transposed entry).  Blocks have as few sites as a domain allows (64 at
// least): they share an SM in larger numbers and the last wave costs less.
// One half-sweep of 12x20x12x28 on 2^4 domains, float32, n_jac 4: 47.7 us with
// operator reads through L1 and branches, 40 us with four threads per site,
// 21.4 us here.

#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "qcd_internal.cuh"

namespace qcd {

template <bool HALF, typename SIO>
struct BlockArgs {
  Geom g;
  int colour, n_jac, do_surface, do_update;
  float kappa;
  SIO s_in, s_out;      // s, float16 or float32 storage
  F32Spinor s_in32;     // if set: the source of this half-sweep, instead of s_in
  F32Spinor x, b;
  const void* links;    // float2 or __half2 [dom][mu][9][vd]
  const void* cinv;     // float4 [dom][18][vd] or __half2 [dom][36][vd]
};

template <bool HALF>
struct BlockOp {
  using Link = typename std::conditional<HALF, __half2, float2>::type;
  static constexpr int LINK_BYTES = 36 * sizeof(Link);  // per site
  static constexpr int CINV_BYTES = HALF ? 144 : 288;
  __device__ static cx<float> entry(const Link* p) {
    if constexpr (HALF) {
      const float2 v = __half22float2(*p);
      return make_cx(v.x, v.y);
    } else {
      const float2 v = *p;
      return make_cx(v.x, v.y);
    }
  }
};

constexpr int SB_GHOST = 8;  // zero sites, one per 16-byte bank group
template <bool HALF, int NT>
constexpr size_t sb_smem() {
  return (size_t)6 * (NT + SB_GHOST) * 16 + (size_t)NT * (BlockOp<HALF>::LINK_BYTES + BlockOp<HALF>::CINV_BYTES);
}

__device__ __forceinline__ void sb_copy(void* dst, const void* src, int bytes, int tid, int nt) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  for (int i = tid * 16; i < bytes; i += nt * 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i),
                 "l"(static_cast<const unsigned char*>(src) + i)
                 : "memory");
}

// T of the projection h = u + sg T (sg = +1: 1 + gamma_MU, -1: 1 - gamma_MU)
template <int MU>
__device__ __forceinline__ void sb_project(const Spinor<float>& p, float sg, HalfSpinor<float>& h) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cx<float> l0 = p.v[2][c], l1 = p.v[3][c];
    const cx<float> t0 = MU == 0 ? times_mi(l1) : (MU == 1 ? -l1 : (MU == 2 ? times_mi(l0) : l0));
    const cx<float> t1 = MU == 0 ? times_mi(l0) : (MU == 1 ? l0 : (MU == 2 ? times_i(l1) : l1));
    h.h[0][c] = cfma(sg, t0, p.v[0][c]);
    h.h[1][c] = cfma(sg, t1, p.v[1][c]);
  }
}
template <int MU>
__device__ __forceinline__ void sb_accumulate(Spinor<float>& acc, const HalfSpinor<float>& h, float sg) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cx<float> h0 = h.h[0][c], h1 = h.h[1][c];
    const cx<float> t2 = MU == 0 ? times_i(h1) : (MU == 1 ? h1 : (MU == 2 ? times_i(h0) : h0));
    const cx<float> t3 = MU == 0 ? times_i(h0) : (MU == 1 ? -h0 : (MU == 2 ? times_mi(h1) : h1));
    acc.v[0][c] = acc.v[0][c] + h0;
    acc.v[1][c] = acc.v[1][c] + h1;
    acc.v[2][c] = cfma(sg, t2, acc.v[2][c]);
    acc.v[3][c] = cfma(sg, t3, acc.v[3][c]);
  }
}

// U (fwd) or U^dag from entries at p, e vd apart
template <bool HALF>
__device__ __forceinline__ void sb_link(const typename BlockOp<HALF>::Link* p, int logvd, bool fwd, SU3<float>& u) {
  const int rs = (fwd ? 3 : 1) << logvd, cs = (fwd ? 1 : 3) << logvd;
  const float sg = fwd ? 1.f : -1.f;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cx<float> v = BlockOp<HALF>::entry(p + a * rs + c * cs);
      u.m[a][c] = make_cx(v.re, sg * v.im);
    }
}

template <int NT>
__device__ __forceinline__ void sb_load_x(const float4* sx, int site, Spinor<float>& p) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = sx[k * (NT + SB_GHOST) + site];
    p.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    p.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
template <int NT>
__device__ __forceinline__ void sb_store_x(float4* sx, int site, const Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const cx<float> a0 = a.v[(2 * k) / 3][(2 * k) % 3], a1 = a.v[(2 * k + 1) / 3][(2 * k + 1) % 3];
    sx[k * (NT + SB_GHOST) + site] = make_float4(a0.re, a0.im, a1.re, a1.im);
  }
}

// acc += the hops of direction MU inside the domain.  l: site in the block,
// s: site in the domain; the domain's links start at sl + (l - s) 36.
template <int MU, bool HALF, int NT>
__device__ __forceinline__ void sb_intra(const Geom& g, const float4* sx, const typename BlockOp<HALF>::Link* sl,
                                         int l, int s, Spinor<float>& acc) {
  const int step = 1 << g.shift[MU], c = (s >> g.shift[MU]) & (g.d[MU] - 1);
  const typename BlockOp<HALF>::Link* links = sl + (l - s) * 36 + ((MU * 9) << g.logvd);
  Spinor<float> p;
  HalfSpinor<float> h, uh;
  SU3<float> u;
  if (g.logd[MU] == 1) {
    const bool fwd = c == 0;
    const int n = fwd ? step : -step;
    const float sg = fwd ? -1.f : 1.f;
    sb_load_x<NT>(sx, l + n, p);
    sb_link<HALF>(links + (fwd ? s : s - step), g.logvd, fwd, u);
    sb_project<MU>(p, sg, h);
    su3_mul(u, h, uh);
    sb_accumulate<MU>(acc, uh, sg);
  } else if (g.logd[MU] > 1) {
    const bool fin = c < g.d[MU] - 1, bin = c > 0;
    sb_load_x<NT>(sx, fin ? l + step : NT + (l & 7), p);
    sb_link<HALF>(links + s, g.logvd, true, u);
    project<MU, -1>(p, h);
    su3_mul(u, h, uh);
    accumulate<MU, -1>(acc, uh);
    sb_load_x<NT>(sx, bin ? l - step : NT + (l & 7), p);
    sb_link<HALF>(links + (bin ? s - step : s), g.logvd, false, u);
    project<MU, +1>(p, h);
    su3_mul(u, h, uh);
    accumulate<MU, +1>(acc, uh);
  }
}

// acc += the hop (fwd or not, per lane) of direction MU that leaves the
// domain, if `out`; x and the link from memory (x past L1: the previous
// launch wrote it)
template <int MU, bool HALF>
__device__ __forceinline__ void sb_outer(const Geom& g, const F32Spinor& x, const typename BlockOp<HALF>::Link* links,
                                         int dom, int s, int rhs_off, bool fwd, bool out, Spinor<float>& acc) {
  int nd = dom, ns = s;
  float f = 0.f;
  if (out) f = (float)nbr_site(g, dom, s, MU, fwd, nd, ns);
  Spinor<float> p;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (out) v = __ldcg(x.p + x.idx(g, nd + rhs_off, k, ns));
    p.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    p.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
  HalfSpinor<float> h, uh;
  SU3<float> u;
  sb_link<HALF>(links + (((size_t)(((fwd ? dom : nd) * 4 + MU) * 9)) << g.logvd) + (fwd ? s : ns), g.logvd, fwd, u);
  const float sg = fwd ? -1.f : 1.f;
  sb_project<MU>(p, sg, h);
  su3_mul(u, h, uh);
  scale_half(uh, f);
  sb_accumulate<MU>(acc, uh, sg);
}
template <int MU, bool HALF>
__device__ __forceinline__ void sb_surface(const Geom& g, const F32Spinor& x, const typename BlockOp<HALF>::Link* links,
                                           int dom, int s, int rhs_off, Spinor<float>& acc) {
  const int c = (s >> g.shift[MU]) & (g.d[MU] - 1);
  if (g.logd[MU] == 0) {  // both hops leave
    sb_outer<MU, HALF>(g, x, links, dom, s, rhs_off, true, true, acc);
    sb_outer<MU, HALF>(g, x, links, dom, s, rhs_off, false, true, acc);
  } else {
    const bool fwd = c == g.d[MU] - 1;
    sb_outer<MU, HALF>(g, x, links, dom, s, rhs_off, fwd, fwd || c == 0, acc);
  }
}

template <bool HALF>
__device__ __forceinline__ void sb_clover(const void* sc, int vd, int logvd, int l, int s, Spinor<float>& psi) {
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    CloverBlockF32 blk;
    if constexpr (HALF) {
      const __half2* p = static_cast<const __half2*>(sc) + (l - s) * 36 + ((18 * b) << logvd) + s;
#pragma unroll
      for (int k = 0; k < 18; ++k) {
        const float2 v = __half22float2(p[k << logvd]);
        blk.r[2 * k] = v.x;
        blk.r[2 * k + 1] = v.y;
      }
    } else {
      const float4* p = static_cast<const float4*>(sc) + (l - s) * 18 + ((9 * b) << logvd) + s;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const float4 v = p[k << logvd];
        blk.r[4 * k] = v.x; blk.r[4 * k + 1] = v.y; blk.r[4 * k + 2] = v.z; blk.r[4 * k + 3] = v.w;
      }
    }
    cx<float> x[6], y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) x[i] = psi.v[2 * b + i / 3][i % 3];
    herm6_mul<float>(blk, x, y);
#pragma unroll
    for (int i = 0; i < 6; ++i) psi.v[2 * b + i / 3][i % 3] = y[i];
  }
}

template <bool HALF, typename SIO, int NT>
__global__ void __launch_bounds__(NT, HALF ? 512 / NT : (NT == 64 ? 5 : 256 / NT))
    sap_block_kernel(BlockArgs<HALF, SIO> a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  using Link = typename BlockOp<HALF>::Link;
  float4* sx = reinterpret_cast<float4*>(bsm);
  Link* sl = reinterpret_cast<Link*>(sx + 6 * (NT + SB_GHOST));
  unsigned char* sc = reinterpret_cast<unsigned char*>(sl) + (size_t)NT * BlockOp<HALF>::LINK_BYTES;
  const Geom& g = a.g;
  if (pdl_enter(g, !a.do_surface)) return;
  const int l = threadIdx.x;
  const int total = g.nhalf << g.logvd, first = blockIdx.x * NT;
  const int nsites = min(NT, total - first);  // whole domains
  const int dom0 = a.colour * g.nhalf + (first >> g.logvd);
  // links and C_inv are constant: before the wait for the previous launch
  sb_copy(sl, static_cast<const unsigned char*>(a.links) + ((size_t)dom0 << g.logvd) * BlockOp<HALF>::LINK_BYTES,
          nsites * BlockOp<HALF>::LINK_BYTES, l, NT);
  sb_copy(sc, static_cast<const unsigned char*>(a.cinv) + ((size_t)dom0 << g.logvd) * BlockOp<HALF>::CINV_BYTES,
          nsites * BlockOp<HALF>::CINV_BYTES, l, NT);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int i = l; i < 6 * SB_GHOST; i += NT)
    sx[(i >> 3) * (NT + SB_GHOST) + NT + (i & 7)] = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool live = l < nsites;
  // threads past the last domain repeat the block's first site and store nothing
  const int li = live ? l : 0;
  const int dom = dom0 + (li >> g.logvd), s = li & (g.vd - 1);
  const int rhs_off = blockIdx.y * g.ndom, domr = dom + rhs_off;

  asm volatile("griddepcontrol.wait;" ::: "memory");
  Spinor<float> src;
  auto load32 = [&](const F32Spinor& f, Spinor<float>& v) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float4 q = __ldcg(f.p + f.idx(g, domr, k, s));
      v.v[(2 * k) / 3][(2 * k) % 3] = make_cx(q.x, q.y);
      v.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(q.z, q.w);
    }
  };
  if (a.s_in32.p) load32(a.s_in32, src);
  else if constexpr (std::is_same<SIO, F32Spinor>::value) load32(a.s_in, src);
  else {
    const float n = __ldcg(a.s_in.nrm + ((size_t)domr << g.logvd) + s);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint4 q = __ldcg(a.s_in.p + a.s_in.idx(g, domr, k, s));
      const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
        src.v[(4 * k + j) / 3][(4 * k + j) % 3] = make_cx(v.x * n, v.y * n);
      }
    }
  }
  Spinor<float> acc;
  if (a.do_surface) {
    zero(acc);
    const Link* links = static_cast<const Link*>(a.links);
    sb_surface<0, HALF>(g, a.x, links, dom, s, rhs_off, acc);
    sb_surface<1, HALF>(g, a.x, links, dom, s, rhs_off, acc);
    sb_surface<2, HALF>(g, a.x, links, dom, s, rhs_off, acc);
    sb_surface<3, HALF>(g, a.x, links, dom, s, rhs_off, acc);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // every thread's copies have landed
  auto axpy = [&](const Spinor<float>& base, Spinor<float>& out) {  // base + kappa acc
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c) out.v[sp][c] = cfma(a.kappa, acc.v[sp][c], base.v[sp][c]);
  };
  if (a.do_surface) {
    sb_clover<HALF>(sc, g.vd, g.logvd, li, s, acc);
    axpy(src, src);
  }
  if (live) sb_store_x<NT>(sx, l, src);
  __syncthreads();

  Spinor<float> xk = src;
  const int napp = a.n_jac + (a.do_update ? 1 : 0);
  for (int it = 0; it < napp; ++it) {
    zero(acc);
    sb_intra<0, HALF, NT>(g, sx, sl, li, s, acc);
    sb_intra<1, HALF, NT>(g, sx, sl, li, s, acc);
    sb_intra<2, HALF, NT>(g, sx, sl, li, s, acc);
    sb_intra<3, HALF, NT>(g, sx, sl, li, s, acc);
    sb_clover<HALF>(sc, g.vd, g.logvd, li, s, acc);
    if (it < a.n_jac) {
      axpy(src, xk);
      __syncthreads();
      if (live) sb_store_x<NT>(sx, l, xk);
      __syncthreads();
    } else {
      Spinor<float> v;
      load32(a.b, v);
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          v.v[sp][c] = make_cx(src.v[sp][c].re + v.v[sp][c].re - xk.v[sp][c].re,
                               src.v[sp][c].im + v.v[sp][c].im - xk.v[sp][c].im);
      axpy(v, v);
      if (live) a.s_out.store(g, domr, s, v);
    }
  }
  if (live) a.x.store(g, domr, s, xk);
}

// Shared memory of a launch: what its blocks use, or, if that is more, so much
// that an SM holds no more of them than an even share.  With room for more, and
// the next launch's blocks arriving while this one's still run, they pair up on
// some SMs and leave others idle.  M_SAP (n_sap 4, n_jac 4), float16 links, us
// without and with: 16^4 on 8x4x4x2 domains 280 and 182, on 2^4 239 and 156;
// 12x20x12x28 on 2^4 257 and 186; float32, 8^2 16 24 on 2^4, 154 and 104.
template <bool HALF, int NT>
static int sb_launch_smem(const qcd_ctx* ctx, long long blocks) {
  constexpr int SM_BYTES = 228 * 1024, BLOCK_RESERVED = 1024, BLOCK_MAX = 227 * 1024;
  const long long share = (blocks + ctx->sms - 1) / ctx->sms;
  const long long pad = SM_BYTES / (share + 1) - BLOCK_RESERVED + 16;  // share + 1 do not fit
  return (int)std::min<long long>(BLOCK_MAX, std::max<long long>((long long)sb_smem<HALF, NT>(), pad));
}

// Algorithm 1 as 2 (n_sap + 1) launches, every right-hand side in each.
// b: the source, also the first sweep's input; x: the result, which holds the
// iterates of both colours on the way.
template <bool HALF, typename SIO, int NT>
static void block_launches(qcd_ctx* ctx, SIO s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                           cudaStream_t st) {
  const long long sites = (long long)ctx->geom.nhalf << ctx->geom.logvd;
  QCD_REQUIRE(sites + NT < (1LL << 31), QCD_ERR_ARG, "SAP: lattice too large");
  const int blocks = (int)((sites + NT - 1) / NT), smem = sb_launch_smem<HALF, NT>(ctx, (long long)blocks * nrhs);
  // the limit is the current device's, and a process may use several
  QCD_CUDA_CHECK(cudaFuncSetAttribute(sap_block_kernel<HALF, SIO, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem));
  BlockArgs<HALF, SIO> a;
  a.g = ctx->geom;
  a.n_jac = n_jac;
  a.kappa = (float)ctx->kappa;
  a.s_in = s;
  a.s_out = s;
  a.x = x;
  a.b = b;
  a.links = HALF ? (const void*)ctx->u16 : (const void*)ctx->u32;
  a.cinv = HALF ? (const void*)ctx->cinv16 : (const void*)ctx->cinv32;
  for (int sweep = 0; sweep <= n_sap; ++sweep) {
    a.s_in32 = sweep == 0 ? b : F32Spinor{nullptr};
    a.do_update = sweep == n_sap ? 0 : 1;
    for (int colour = 0; colour < 2; ++colour) {
      a.colour = colour;
      a.do_surface = (sweep == 0 && colour == 0) ? 0 : 1;
      LaunchScope ls(ctx, QCD_KC_SAP_BLOCK, st);
      launch_pdl(sap_block_kernel<HALF, SIO, NT>, dim3((unsigned)blocks, nrhs), dim3(NT), smem, st, a);
      check_launch();
    }
  }
}
template <bool HALF, typename SIO>
static void block_sequence(qcd_ctx* ctx, SIO s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                           cudaStream_t st) {
  const int vd = ctx->geom.vd;
  if (vd <= 64) block_launches<HALF, SIO, 64>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
  else if (vd == 128) block_launches<HALF, SIO, 128>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
  else block_launches<HALF, SIO, 256>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}

void sap_block_f32(qcd_ctx* ctx, F32Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                   cudaStream_t st) {
  block_sequence<false, F32Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}
void sap_block_f16(qcd_ctx* ctx, F16Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                   cudaStream_t st) {
  block_sequence<true, F16Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}
void sap_block_h16g(qcd_ctx* ctx, F32Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                    cudaStream_t st) {
  block_sequence<true, F32Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}

}  // namespace qcd
