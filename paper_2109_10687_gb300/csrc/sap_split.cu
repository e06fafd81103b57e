// SAP half-sweep on 4^4 domains with four threads per site (Sec. 3 of
// arXiv:2109.10687, Algorithms 1 and 2), for lattices with too few domains to
// fill the GPU.
//
// Per launch, for the domains of one colour c: the surface term
// s <- s + kappa C_inv H_cc' x_c', n_jac Jacobi sweeps
// x <- s + kappa C_inv H_cc x, the residual update
// s <- s + b - x + kappa C_inv H_cc x (not in the closing sweep), and x_c to
// memory.
//
// What bounds it: a small lattice leaves a thread per site with two warps per
// scheduler, each waiting on its own chain of loads and multiply-adds.  So a
// site gets four threads, a block 64 sites (a time slice of the domain) and a
// domain a cluster of four blocks.
//   Hops: thread (site, direction) keeps U_mu(n) and U_mu(n - mu) in
//     registers for the whole launch, already converted to float32, reads the
//     two neighbours' spinors (the neighbouring block's through distributed
//     shared memory; zeros for a hop that leaves the domain) and leaves the
//     two products U P x in shared memory as half spinors.  The direction is
//     the same for a whole warp.
//   Sites: thread (site, spin), the spin also the same for a whole warp, adds
//     the spin's rows of the eight half spinors, swaps sums with the other
//     spin of its chirality through shared memory and multiplies by its three
//     rows of C_inv, which it also keeps in registers.
// Sums and products are in the order of the one-thread-per-site kernel
// (sap_staged.cu), so both give the same M_SAP bit for bit.
// M_SAP (n_sap 4, n_jac 4): 8^4 on 4^4 domains, float32, 0.134 ms with a thread
// per site (8 blocks a colour) and 0.105 ms here (32 blocks); 16 8^3 0.134 and
// 0.116; from 16^2 8^2 on (32 domains a colour) the block kernel is the faster.
// It is bound by shared memory (2.2 KB per site and sweep) in turn with the FMA
// pipe, between barriers.

#include <cooperative_groups.h>

#include <cstdio>
#include <type_traits>

#include "qcd_internal.cuh"

namespace cg = cooperative_groups;

namespace qcd {

constexpr int SP_SITES = 64;
constexpr int SP_THREADS = 4 * SP_SITES;
constexpr int SP_BLOCKS = 4;                 // blocks per domain (cluster size)
constexpr int SP_XF4 = 6 * SP_SITES;         // float4 of one buffer of x
constexpr int SP_HF2 = 8 * 6 * SP_SITES;     // float2 of the half spinors [hop 8][row 2][colour 3][site]

template <bool HALF, typename SIO>
struct SplitArgs {
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
__device__ __forceinline__ void sp_link(const void* base, const Geom& g, int dom, int mu, int s, SU3<float>& u) {
  if (HALF) LinkPtrHalf{static_cast<const __half2*>(base)}.load(g, dom, mu, s, u);
  else LinkPtr<float>{static_cast<const float2*>(base)}.load(g, dom, mu, s, u);
}

// rows 3 r .. 3 r + 2 of one chiral block (spin q = 2 b + r): the diagonal, the
// entries 01, 02, 12 of the own spin's block and the nine to the other spin
struct CinvRows {
  float d[3];
  cx<float> in[3], out[3][3];
};
template <bool HALF, int Q>
__device__ __forceinline__ void sp_cinv(const void* base, const Geom& g, int dom, int s, CinvRows& m) {
  constexpr int r = Q & 1;
  CloverBlockF32 k;
  if (HALF) CloverPtrF16{static_cast<const __half2*>(base)}.load_block(g, dom, s, Q >> 1, k);
  else CloverPtrF32{static_cast<const float4*>(base)}.load_block(g, dom, s, Q >> 1, k);
#pragma unroll
  for (int a = 0; a < 3; ++a) m.d[a] = k.r[3 * r + a];
  int o = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i + 1; j < 3; ++j, ++o) m.in[o] = k.off(herm_off(3 * r + i, 3 * r + j));
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) m.out[a][c] = r ? conjg(k.off(herm_off(c, 3 + a))) : k.off(herm_off(a, 3 + c));
}

// own three rows of C_inv times (own spin's sums, the other spin's sums), each
// row in ascending order of the column after the diagonal (herm6_mul's order)
template <int R>
__device__ __forceinline__ void sp_cinv_mul(const CinvRows& m, const cx<float> own[3], const cx<float> oth[3],
                                            cx<float> y[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cx<float> v = m.d[a] * own[a];
    if (R == 1)
#pragma unroll
      for (int c = 0; c < 3; ++c) v = cmac(v, m.out[a][c], oth[c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (c == a) continue;
      const cx<float> e = m.in[c + a - 1];
      v = c > a ? cmac(v, e, own[c]) : cmacc(v, e, own[c]);
    }
    if (R == 0)
#pragma unroll
      for (int c = 0; c < 3; ++c) v = cmac(v, m.out[a][c], oth[c]);
    y[a] = v;
  }
}

// the half spinor of hop (2 MU + side) of a site
__device__ __forceinline__ void sp_put(float2* hs, int hop, int site, const HalfSpinor<float>& h) {
#pragma unroll
  for (int row = 0; row < 2; ++row)
#pragma unroll
    for (int c = 0; c < 3; ++c) hs[((hop * 2 + row) * 3 + c) * SP_SITES + site] = make_float2(h.h[row][c].re, h.h[row][c].im);
}

// both products of direction MU, from the neighbours' spinors
template <int MU>
__device__ __forceinline__ void sp_hop_fwd(const SU3<float>& u, const Spinor<float>& p, float sign, float2* hs, int site) {
  HalfSpinor<float> h, uh;
  project<MU, -1>(p, h);
  su3_mul(u, h, uh);
  scale_half(uh, sign);
  sp_put(hs, 2 * MU, site, uh);
}
template <int MU>
__device__ __forceinline__ void sp_hop_bwd(const SU3<float>& u, const Spinor<float>& p, float sign, float2* hs, int site) {
  HalfSpinor<float> h, uh;
  project<MU, +1>(p, h);
  su3_dag_mul(u, h, uh);
  scale_half(uh, sign);
  sp_put(hs, 2 * MU + 1, site, uh);
}

// spinor from six float4, stride apart (stride 0: all the same float4 of zeros)
__device__ __forceinline__ void sp_read(const float4* p, int stride, Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = p[k * stride];
    a.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    a.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
// the same from memory, past L1: the previous launch wrote it
__device__ __forceinline__ void sp_read_global(const Geom& g, const F32Spinor& x, int dom, int s, Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = __ldcg(x.p + x.idx(g, dom, k, s));
    a.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    a.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}

// acc += spin Q of the spinor rebuilt from a hop's half spinor (the rules of
// accumulate1)
template <int MU, int PM, int Q, bool FIRST>
__device__ __forceinline__ void sp_take(const float2* hs, int site, cx<float> acc[3]) {
  constexpr int hop = 2 * MU + (PM < 0 ? 0 : 1), r = Q & 1;
  constexpr bool lower = Q >= 2;
  constexpr int row = lower && MU < 2 ? 1 - r : r;  // x and y: the lower spins come from the other row,
  constexpr bool imag = lower && (MU == 0 || MU == 2);  // x and z: times +-i,
  // with the sign of the projector, the opposite one on spin 3 for y and z
  constexpr bool neg = lower && ((PM < 0) != ((MU == 1 || MU == 2) && r == 1));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float2 v = hs[((hop * 2 + row) * 3 + c) * SP_SITES + site];
    cx<float> h = imag ? make_cx(-v.y, v.x) : make_cx(v.x, v.y);
    if (neg) h = -h;
    acc[c] = FIRST ? h : acc[c] + h;
  }
}
// all eight, in the order of the sweeps (x, t, y, z) or of the surface term (x, y, z, t)
template <bool SURFACE, int Q>
__device__ __forceinline__ void sp_gather(const float2* hs, int site, cx<float> acc[3]) {
  sp_take<0, -1, Q, true>(hs, site, acc);
  sp_take<0, +1, Q, false>(hs, site, acc);
  if (!SURFACE) {
    sp_take<3, -1, Q, false>(hs, site, acc);
    sp_take<3, +1, Q, false>(hs, site, acc);
  }
  sp_take<1, -1, Q, false>(hs, site, acc);
  sp_take<1, +1, Q, false>(hs, site, acc);
  sp_take<2, -1, Q, false>(hs, site, acc);
  sp_take<2, +1, Q, false>(hs, site, acc);
  if (SURFACE) {
    sp_take<3, -1, Q, false>(hs, site, acc);
    sp_take<3, +1, Q, false>(hs, site, acc);
  }
}
// f(k) for the warp-uniform k = 0..3 as a compile-time constant
template <typename F>
__device__ __forceinline__ void sp_switch(int k, F f) {
  if (k == 0) f(std::integral_constant<int, 0>{});
  else if (k == 1) f(std::integral_constant<int, 1>{});
  else if (k == 2) f(std::integral_constant<int, 2>{});
  else f(std::integral_constant<int, 3>{});
}

// y = spin q of C_inv (the sum of the hops).  One barrier, outside the
// switches: q differs between the warps of a block.
template <bool SURFACE>
__device__ __forceinline__ void sp_site_sum(const float2* hs, float2* ex, const CinvRows& m, int q, int site,
                                            cx<float> y[3]) {
  cx<float> acc[3], oth[3];
  sp_switch(q, [&](auto k) { sp_gather<SURFACE, decltype(k)::value>(hs, site, acc); });
#pragma unroll
  for (int c = 0; c < 3; ++c) ex[(q * 3 + c) * SP_SITES + site] = make_float2(acc[c].re, acc[c].im);
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float2 v = ex[((q ^ 1) * 3 + c) * SP_SITES + site];
    oth[c] = make_cx(v.x, v.y);
  }
  if (q & 1) sp_cinv_mul<1>(m, acc, oth, y);
  else sp_cinv_mul<0>(m, acc, oth, y);
}

// component comp = spin * 3 + colour of a float32 field
__device__ __forceinline__ float2* sp_comp(const F32Spinor& f, const Geom& g, int dom, int comp, int s) {
  return reinterpret_cast<float2*>(f.p + f.idx(g, dom, comp >> 1, s)) + (comp & 1);
}

template <bool HALF, typename SIO>
__global__ void __launch_bounds__(SP_THREADS, 2) sap_split_kernel(SplitArgs<HALF, SIO> a) {
  __shared__ float4 xs[2 * SP_XF4];
  __shared__ float2 hs[SP_HF2];
  __shared__ float2 ex[4 * 3 * SP_SITES];
  __shared__ float4 zero4;
  __shared__ float nrm[4 * SP_SITES];
  const Geom& g = a.g;
  if (pdl_enter(g, !a.do_surface)) return;  // the same decision in every block of the cluster
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // direction in the hops, spin in the site sums
  const int q = w >> 1, site = (w & 1) * 32 + lane;
  const cg::cluster_group cl = cg::this_cluster();
  const int dom = a.colour * g.nhalf + blockIdx.x / SP_BLOCKS;
  const int loc = (int)cl.block_rank() * SP_SITES + site;  // site of the domain
  const int rhs_off = blockIdx.y * g.ndom;
  const int domr = dom + rhs_off;

  SU3<float> uf, ub;
  int fd, fs, bd, bs;
  const float fsign = (float)nbr_site(g, dom, loc, q, true, fd, fs);
  const float bsign = (float)nbr_site(g, dom, loc, q, false, bd, bs);
  sp_link<HALF>(a.links, g, dom, q, loc, uf);
  sp_link<HALF>(a.links, g, bd, q, bs, ub);
  const bool fin = hop_is_intra(g, loc, q, true), bin = hop_is_intra(g, loc, q, false);
  const float4 *pf = &zero4, *pb = &zero4;
  if (fin) pf = cl.map_shared_rank(xs, fs / SP_SITES) + fs % SP_SITES;
  if (bin) pb = cl.map_shared_rank(xs, bs / SP_SITES) + bs % SP_SITES;
  const int sf = fin ? SP_SITES : 0, sb = bin ? SP_SITES : 0;
  CinvRows m;
  sp_switch(q, [&](auto k) { sp_cinv<HALF, decltype(k)::value>(a.cinv, g, dom, loc, m); });
  if (threadIdx.x == 0) zero4 = make_float4(0.f, 0.f, 0.f, 0.f);

  asm volatile("griddepcontrol.wait;" ::: "memory");  // links and C_inv are constant; everything below is not
  cx<float> src[3], y[3];
  if (std::is_same<SIO, F32Spinor>::value || a.s_in32.p) {
    F32Spinor in = a.s_in32;
    if constexpr (std::is_same<SIO, F32Spinor>::value)
      if (!in.p) in = a.s_in;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2 v = __ldcg(sp_comp(in, g, domr, 3 * q + c, loc));
      src[c] = make_cx(v.x, v.y);
    }
  } else if constexpr (std::is_same<SIO, F16Spinor>::value) {
    const float n = __ldcg(a.s_in.nrm + ((size_t)domr << g.logvd) + loc);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int k = 3 * q + c;
      const unsigned word = __ldcg(reinterpret_cast<const unsigned*>(a.s_in.p + a.s_in.idx(g, domr, k >> 2, loc)) + (k & 3));
      const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&word));
      src[c] = make_cx(v.x * n, v.y * n);
    }
  }
  auto put_x = [&](const cx<float> v[3], int buf) {
    float4* p = xs + buf * SP_XF4 + site;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int k = 3 * q + c;
      reinterpret_cast<float2*>(p + (k >> 1) * SP_SITES)[k & 1] = make_float2(v[c].re, v[c].im);
    }
  };
  if (a.do_surface) {
    sp_switch(q, [&](auto k) {
      constexpr int MU = decltype(k)::value;
      Spinor<float> p;
      zero(p);
      if (!fin) sp_read_global(g, a.x, fd + rhs_off, fs, p);
      sp_hop_fwd<MU>(uf, p, fsign, hs, site);
      zero(p);
      if (!bin) sp_read_global(g, a.x, bd + rhs_off, bs, p);
      sp_hop_bwd<MU>(ub, p, bsign, hs, site);
    });
    __syncthreads();
    sp_site_sum<true>(hs, ex, m, q, site, y);
#pragma unroll
    for (int c = 0; c < 3; ++c) src[c] = cfma(a.kappa, y[c], src[c]);
  }
  put_x(src, 0);
  cl.sync();

  cx<float> xk[3] = {src[0], src[1], src[2]};
  const int napp = a.n_jac + (a.do_update ? 1 : 0);
  int cur = 0;
  for (int it = 0; it < napp; ++it) {
    sp_switch(q, [&](auto k) {
      constexpr int MU = decltype(k)::value;
      const int off = cur * SP_XF4;
      Spinor<float> p;
      sp_read(pf + (fin ? off : 0), sf, p);
      sp_hop_fwd<MU>(uf, p, 1.f, hs, site);
      sp_read(pb + (bin ? off : 0), sb, p);
      sp_hop_bwd<MU>(ub, p, 1.f, hs, site);
    });
    __syncthreads();
    sp_site_sum<false>(hs, ex, m, q, site, y);
    if (it < a.n_jac) {
#pragma unroll
      for (int c = 0; c < 3; ++c) xk[c] = cfma(a.kappa, y[c], src[c]);
      cur ^= 1;  // the other blocks may still read this one's x
      put_x(xk, cur);
      cl.sync();
    } else {
      cx<float> v[3];
      float mx = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 bv = __ldcg(sp_comp(a.b, g, domr, 3 * q + c, loc));
        v[c] = cfma(a.kappa, y[c], make_cx(src[c].re + bv.x - xk[c].re, src[c].im + bv.y - xk[c].im));
        mx = fmaxf(mx, fmaxf(fabsf(v[c].re), fabsf(v[c].im)));
      }
      if constexpr (std::is_same<SIO, F32Spinor>::value) {
#pragma unroll
        for (int c = 0; c < 3; ++c) *sp_comp(a.s_out, g, domr, 3 * q + c, loc) = make_float2(v[c].re, v[c].im);
      } else {
        // the site's norm is the largest component of all four spins
        nrm[q * SP_SITES + site] = mx;
        __syncthreads();
        mx = fmaxf(fmaxf(nrm[site], nrm[SP_SITES + site]), fmaxf(nrm[2 * SP_SITES + site], nrm[3 * SP_SITES + site]));
        const float inv = mx > 0.f ? 1.0f / mx : 0.f;
        if (q == 0) a.s_out.nrm[((size_t)domr << g.logvd) + loc] = mx;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int k = 3 * q + c;
          const __half2 h = __floats2half2_rn(v[c].re * inv, v[c].im * inv);
          reinterpret_cast<__half2*>(a.s_out.p + a.s_out.idx(g, domr, k >> 2, loc))[k & 3] = h;
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) *sp_comp(a.x, g, domr, 3 * q + c, loc) = make_float2(xk[c].re, xk[c].im);
  cl.sync();  // the neighbours' last reads of this block's x are done
}

// Algorithm 1 as 2 (n_sap + 1) launches, every right-hand side in each.
// b: the source, also the first sweep's input; x: the result, which holds the
// iterates of both colours on the way.
template <bool HALF, typename SIO>
static void split_sequence(qcd_ctx* ctx, SIO s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                           cudaStream_t st) {
  const Geom& g = ctx->geom;
  SplitArgs<HALF, SIO> a;
  a.g = g;
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
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(g.nhalf * SP_BLOCKS, nrhs);
      cfg.blockDim = dim3(SP_THREADS);
      cfg.stream = st;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      attr[1].id = cudaLaunchAttributeClusterDimension;
      attr[1].val.clusterDim.x = SP_BLOCKS;
      attr[1].val.clusterDim.y = 1;
      attr[1].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      QCD_CUDA_CHECK(cudaLaunchKernelEx(&cfg, sap_split_kernel<HALF, SIO>, a));
      check_launch();
    }
  }
}

void sap_split_f32(qcd_ctx* ctx, F32Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                   cudaStream_t st) {
  split_sequence<false, F32Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}
void sap_split_f16(qcd_ctx* ctx, F16Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                   cudaStream_t st) {
  split_sequence<true, F16Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}
void sap_split_h16g(qcd_ctx* ctx, F32Spinor s, F32Spinor x, F32Spinor b, int nrhs, int n_sap, int n_jac,
                    cudaStream_t st) {
  split_sequence<true, F32Spinor>(ctx, s, x, b, nrhs, n_sap, n_jac, st);
}

}  // namespace qcd
