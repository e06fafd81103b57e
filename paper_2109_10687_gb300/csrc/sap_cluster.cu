// SAP half-sweep on large domains of any extents (the paper's 16x6x4x3 and
// 16x6x4x6, Sec. 4.3, Tables 2-3) with one thread-block cluster per domain
// (Sec. 3, Algorithms 1 and 2; float16 links and C_inv, float32 vectors).
//
// A domain d0 x d1 x d2 x d3 is cut into its d3 time slices; CTA t of the
// cluster (cluster rank t) holds slice t, d0 d1 d2 sites, one thread per
// site.  At entry a CTA brings its slice's links (float16, 40 B per link)
// and C_inv (float16, 144 B per site) into shared memory with two bulk
// copies on an mbarrier (bounded wait), from a staging layout built for this
// kernel.  Its shared memory also holds the slice's float32 iterate x and, for the hops in t, two half
// spinors per site that the neighbouring slices' CTAs write there through
// distributed shared memory: P- x(t + 1) from above and U^dag P+ x(t - 1),
// finished by the CTA that holds the link, from below.  Hops in x, y and z
// read x of the own slice, without branches: a hop that leaves the domain
// reads a site of zeros.
//
// Two cluster barriers per sweep: the first (arrive after the hops' reads,
// wait after the C_inv multiply) separates the reads of x and of the half
// spinors from the next writes, the second those writes from the next reads.
//
// The surface term (hops that leave the domain): at the end of a launch every
// site on a face leaves its half spinor for the neighbouring domain in a halo
// in memory (cs_slot), from registers and the staged link; the next launch
// reads one half spinor per face site, all of them in flight while the staging
// copies are under way.  Domains whose faces need more than the caller's 96
// bytes per site (extents of one) read the neighbours' x and links in place.
//
// The next launch may start early (programmatic dependent launch): its first
// clusters take the SMs that the last wave of clusters leaves idle and bring
// their operator in, then wait for this launch.  So whatever changes between
// launches is read past L1.
//
// What bounds it: one CTA of 12 warps per SM (16x6x4x3: 190 KB of shared
// memory), so each warp's chain of loads and multiply-adds, and whole waves
// of clusters.  32x24x16x24, 128 clusters in three waves, a half-sweep with
// n_jac 2: 96 us with the t neighbours' spinors and links read from the other
// CTAs in place and a branch per hop; 70 with half spinors pushed there; 67
// with the halo (before, the surface hops gathered x and links from memory);
// 59 with early starts.  Of those 35 are the three sweeps.
// M_SAP (n_sap 4, n_jac 2) 1000 -> 628 us.

#include <cooperative_groups.h>

#include <cstdio>

#include "qcd_internal.cuh"

namespace cg = cooperative_groups;

namespace qcd {

constexpr int CS_MAX_K = 8;            // slices (CTAs) per cluster, the portable maximum
constexpr int CS_MAX_SLICE = 448;      // sites per slice: 496 B of shared memory each
constexpr int CS_LINK_H2 = 10;         // half2 per staged link (9 + 1 pad)
constexpr int CS_CLOV_U4 = 9;          // uint4 per site of staged C_inv
constexpr int CS_BYTES_PER_SITE = 96 + 2 * 48 + 4 * CS_LINK_H2 * 4 + CS_CLOV_U4 * 16;  // 496
constexpr int CS_GHOST = 8;            // zero sites after x, one per 16-byte bank group
constexpr int CS_EXTRA_BYTES = 6 * CS_GHOST * 16 + 16;

struct ClusterSapArgs {
  Geom g;
  int sd[4];     // SAP domain extents; sd[3] slices per domain = cluster size
  int snd[4];    // SAP domains per direction
  int slice;     // sites per slice
  int colour, n_jac, do_surface, do_update;
  float kappa;
  F32Spinor s_in, s_out, x, b;
  LinkPtrHalf U16;             // links in the internal layout (backward hops that enter the domain, without halo)
  float4* halo;                // half spinors at the faces between domains, see cs_slot
  size_t halo_at[4];           // where direction mu's begin
  int face[4];                 // sites of a face of a domain
  int do_halo;                 // leave the neighbours' half spinors (0 in the last launch)
  const unsigned char* links;  // staging: [domain][slice][mu][site][10 half2]
  const unsigned char* clov;   // staging: [domain][slice][site][9 uint4]
  int* status;
  int extra_tx;                // testing: bytes the staging wait expects beyond its copies
};

__device__ __forceinline__ SU3<float> cs_link(const unsigned char* base, int slice, int mu, int site) {
  const uint2* p = reinterpret_cast<const uint2*>(base) + (mu * slice + site) * (CS_LINK_H2 / 2);
  SU3<float> u;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const uint2 w = p[k];
    const float2 v0 = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
    u.m[(2 * k) / 3][(2 * k) % 3] = make_cx(v0.x, v0.y);
    if (2 * k + 1 < 9) {
      const float2 v1 = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
      u.m[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v1.x, v1.y);
    }
  }
  return u;
}

// C_inv of a site: two blocks of 36 halves back to back in 9 uint4
__device__ __forceinline__ void cs_clover(const unsigned char* base, int site, Spinor<float>& psi) {
  const uint4* p = reinterpret_cast<const uint4*>(base) + site * CS_CLOV_U4;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    unsigned w[18];
    const uint2 mid = reinterpret_cast<const uint2*>(p + 4)[b];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint4 v = p[b == 0 ? k : 5 + k];
      const int o = b == 0 ? 4 * k : 2 + 4 * k;
      w[o] = v.x; w[o + 1] = v.y; w[o + 2] = v.z; w[o + 3] = v.w;
    }
    w[b == 0 ? 16 : 0] = mid.x;
    w[b == 0 ? 17 : 1] = mid.y;
    CloverBlockF32 blk;
#pragma unroll
    for (int k = 0; k < 18; ++k) {
      const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
      blk.r[2 * k] = v.x;
      blk.r[2 * k + 1] = v.y;
    }
    cx<float> xin[6], y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) xin[i] = psi.v[2 * b + i / 3][i % 3];
    herm6_mul<float>(blk, xin, y);
#pragma unroll
    for (int i = 0; i < 6; ++i) psi.v[2 * b + i / 3][i % 3] = y[i];
  }
}

// x: float4 [6][slice + CS_GHOST]
__device__ __forceinline__ void cs_load_x(const float4* buf, int stride, int s, Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = buf[k * stride + s];
    a.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    a.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
__device__ __forceinline__ void cs_store_x(float4* buf, int stride, int s, const Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const cx<float> a0 = a.v[(2 * k) / 3][(2 * k) % 3], a1 = a.v[(2 * k + 1) / 3][(2 * k + 1) % 3];
    buf[k * stride + s] = make_float4(a0.re, a0.im, a1.re, a1.im);
  }
}
// a field's site from memory, past L1 (an earlier launch wrote it)
__device__ __forceinline__ void cs_read_x(const Geom& g, const F32Spinor& f, int dom, int s, Spinor<float>& a) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = __ldcg(f.p + f.idx(g, dom, k, s));
    a.v[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    a.v[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
// half spinors: float4 [3][slice]
__device__ __forceinline__ void cs_load_half(const float4* buf, int slice, int s, HalfSpinor<float>& h) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 v = buf[k * slice + s];
    h.h[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    h.h[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
__device__ __forceinline__ void cs_store_half(float4* buf, int slice, int s, const HalfSpinor<float>& h) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cx<float> a0 = h.h[(2 * k) / 3][(2 * k) % 3], a1 = h.h[(2 * k + 1) / 3][(2 * k + 1) % 3];
    buf[k * slice + s] = make_float4(a0.re, a0.im, a1.re, a1.im);
  }
}

template <int MU, int PM>
__device__ __forceinline__ void cs_hop(const SU3<float>& u, const Spinor<float>& p, float sign, Spinor<float>& acc) {
  HalfSpinor<float> h, uh;
  project<MU, PM>(p, h);
  if (PM < 0) su3_mul(u, h, uh);
  else su3_dag_mul(u, h, uh);
  accumulate<MU, PM>(acc, uh, sign);
}

// both hops of direction MU (0..2): the neighbours' sites in the slice, or a
// zero site (and some valid link) for a hop that leaves the domain
template <int MU>
__device__ __forceinline__ void cs_intra_space(const float4* xb, const unsigned char* sl, int slice, int s, int stride,
                                               bool fin, bool bin, Spinor<float>& acc) {
  const int zero_site = slice + (s & (CS_GHOST - 1));
  Spinor<float> p;
  cs_load_x(xb, slice + CS_GHOST, fin ? s + stride : zero_site, p);
  cs_hop<MU, -1>(cs_link(sl, slice, MU, s), p, 1.f, acc);
  cs_load_x(xb, slice + CS_GHOST, bin ? s - stride : zero_site, p);
  cs_hop<MU, +1>(cs_link(sl, slice, MU, bin ? s - stride : s), p, 1.f, acc);
}

// this site's half spinors for the neighbouring slices' t hops, into their
// CTAs' shared memory (null: no such slice)
__device__ __forceinline__ void cs_push_t(float4* below, float4* above, const unsigned char* sl, int slice, int s,
                                          const Spinor<float>& x) {
  HalfSpinor<float> h, uh;
  if (below) {
    project<3, -1>(x, h);
    cs_store_half(below, slice, s, h);
  }
  if (above) {
    project<3, +1>(x, h);
    su3_dag_mul(cs_link(sl, slice, 3, s), h, uh);
    cs_store_half(above, slice, s, uh);
  }
}

__device__ __forceinline__ void cs_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cs_wait_all() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Half spinors between domains: float4 [direction][domain][3][face site], one
// slot per site of the face between a domain and the next one up.  The lower
// domain leaves U^dag P+ x there, the finished hop backward of the upper one,
// which in its own launch leaves P- x, to be multiplied by the lower one's
// link.  Either way the thread that reads a slot at the start of a launch is
// the one that writes it at the end, and no other touches it in that launch.
// At most 96 bytes per site as long as the extents' reciprocals sum to two.
__device__ __forceinline__ float4* cs_slot(const ClusterSapArgs& a, const int D[4], long long jd, const int lc[4],
                                           int mu, bool up) {
  long long step = 1;
  int f = 0, m = 1;
#pragma unroll
  for (int nu = 0; nu < 4; ++nu) {
    if (nu < mu) step *= a.snd[nu];
    if (nu == mu) continue;
    f += m * lc[nu];
    m *= a.sd[nu];
  }
  if (!up) jd += D[mu] == 0 ? (a.snd[mu] - 1) * step : -step;
  return a.halo + a.halo_at[mu] + (size_t)jd * 3 * a.face[mu] + f;
}
// a slot, past L1: the launch before wrote it
__device__ __forceinline__ void cs_read_slot(const float4* p, int face, HalfSpinor<float>& h) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 v = __ldcg(p + k * face);
    h.h[(2 * k) / 3][(2 * k) % 3] = make_cx(v.x, v.y);
    h.h[(2 * k + 1) / 3][(2 * k + 1) % 3] = make_cx(v.z, v.w);
  }
}
// the half spinor of direction mu that a site on either face (upper first)
// takes in; read long before it is used
__device__ __forceinline__ void cs_halo_read(const ClusterSapArgs& a, const int D[4], long long jd, const int lc[4],
                                             int mu, HalfSpinor<float>& h) {
  const bool up = lc[mu] == a.sd[mu] - 1;
  if (up || lc[mu] == 0) cs_read_slot(cs_slot(a, D, jd, lc, mu, up), a.face[mu], h);
}
template <int MU>
__device__ __forceinline__ void cs_halo_in(const ClusterSapArgs& a, const unsigned char* sl, const int D[4],
                                           long long jd, const int X[4], const int lc[4], int s,
                                           const HalfSpinor<float>& in, Spinor<float>& acc) {
  HalfSpinor<float> uh;
  const bool up = lc[MU] == a.sd[MU] - 1;
  if (up) {
    su3_mul(cs_link(sl, a.slice, MU, s), in, uh);
    accumulate<MU, -1>(acc, uh, (MU == 3 && X[3] + 1 == a.g.L[3]) ? (float)a.g.bc_t : 1.f);
  }
  if (lc[MU] == 0) {
    if (up) cs_read_slot(cs_slot(a, D, jd, lc, MU, false), a.face[MU], uh);  // an extent of one: both faces
    else uh = in;
    accumulate<MU, +1>(acc, uh, (MU == 3 && X[3] == 0) ? (float)a.g.bc_t : 1.f);
  }
}
template <int MU>
__device__ __forceinline__ void cs_halo_out(const ClusterSapArgs& a, const unsigned char* sl, const int D[4],
                                            long long jd, const int lc[4], int s, const Spinor<float>& x) {
  HalfSpinor<float> h, uh;
  if (lc[MU] == a.sd[MU] - 1) {
    project<MU, +1>(x, h);
    su3_dag_mul(cs_link(sl, a.slice, MU, s), h, uh);
    cs_store_half(cs_slot(a, D, jd, lc, MU, true), a.face[MU], 0, uh);
  }
  if (lc[MU] == 0) {
    project<MU, -1>(x, h);
    cs_store_half(cs_slot(a, D, jd, lc, MU, false), a.face[MU], 0, h);
  }
}
// L1 prefetch of what cs_inter reads for one hop: the spinor and, for a
// backward hop, the neighbouring domain's link
__device__ __forceinline__ void cs_prefetch(const ClusterSapArgs& a, const int Y[4], int mu, bool bwd) {
  const Geom& g = a.g;
  int nd, ns;
  coords_to_internal(g, Y, nd, ns);
#pragma unroll
  for (int k = 0; k < 6; ++k) asm volatile("prefetch.global.L1 [%0];" ::"l"(a.x.p + a.x.idx(g, nd, k, ns)));
  if (bwd) {
    const __half2* p = a.U16.p + (((size_t)((nd * 4 + mu) * 9)) << g.logvd) + ns;
#pragma unroll
    for (int e = 0; e < 9; ++e) asm volatile("prefetch.global.L1 [%0];" ::"l"(p + ((size_t)e << g.logvd)));
  }
}
__device__ __forceinline__ void cs_prefetch_surface(const ClusterSapArgs& a, const int X[4], const int lc[4]) {
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    int Y[4] = {X[0], X[1], X[2], X[3]};
    if (lc[mu] == a.sd[mu] - 1) {
      Y[mu] = X[mu] + 1 == a.g.L[mu] ? 0 : X[mu] + 1;
      cs_prefetch(a, Y, mu, false);
    }
    if (lc[mu] == 0) {
      Y[mu] = X[mu] == 0 ? a.g.L[mu] - 1 : X[mu] - 1;
      cs_prefetch(a, Y, mu, true);
    }
  }
}

// hops that leave the domain (surface term): x of the other colour and the
// neighbouring domain's links from memory
template <int MU>
__device__ __forceinline__ void cs_inter(const ClusterSapArgs& a, const unsigned char* sl, const int X[4],
                                         const int lc[4], int s, Spinor<float>& acc) {
  const Geom& g = a.g;
  int Y[4] = {X[0], X[1], X[2], X[3]};
  if (lc[MU] == a.sd[MU] - 1) {
    Y[MU] = X[MU] + 1 == g.L[MU] ? 0 : X[MU] + 1;
    const float sign = (MU == 3 && X[3] + 1 == g.L[3]) ? (float)g.bc_t : 1.f;
    int nd, ns;
    coords_to_internal(g, Y, nd, ns);
    Spinor<float> p;
    a.x.load(g, nd, ns, p);
    cs_hop<MU, -1>(cs_link(sl, a.slice, MU, s), p, sign, acc);
    Y[MU] = X[MU];
  }
  if (lc[MU] == 0) {
    Y[MU] = X[MU] == 0 ? g.L[MU] - 1 : X[MU] - 1;
    const float sign = (MU == 3 && X[3] == 0) ? (float)g.bc_t : 1.f;
    int nd, ns;
    coords_to_internal(g, Y, nd, ns);
    Spinor<float> p;
    a.x.load(g, nd, ns, p);
    SU3<float> u;
    a.U16.load(g, nd, MU, ns, u);
    cs_hop<MU, +1>(u, p, sign, acc);
  }
}

__device__ __forceinline__ bool cs_wait(uint64_t* bar) {
  unsigned ok = 0;
  const unsigned addr = static_cast<unsigned>(__cvta_generic_to_shared(bar));
  unsigned long long t0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (int i = 0; i < (1 << 24); ++i) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(addr)
        : "memory");
    if (ok) return true;
    if ((i & 255) == 255) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > 500000000ull) return false;
    }
  }
  return false;
}

template <bool HALO>
__global__ void __launch_bounds__(CS_MAX_SLICE, 1) sap_cluster_kernel(ClusterSapArgs a) {
  extern __shared__ __align__(128) unsigned char csm[];
  const Geom& g = a.g;
  cg::cluster_group cl = cg::this_cluster();
  const int K = a.sd[3];
  const int lt = (int)cl.block_rank();  // time slice of this CTA
  const int S = a.slice;
  float4* xb = reinterpret_cast<float4*>(csm);   // the iterate
  float4* t_up = xb + 6 * (S + CS_GHOST);        // P- x of the slice above
  float4* t_dn = t_up + 3 * S;                   // U^dag P+ x of the slice below
  unsigned char* sl = reinterpret_cast<unsigned char*>(t_dn + 3 * S);  // links
  unsigned char* sc = sl + 4 * CS_LINK_H2 * 4 * S;  // C_inv
  uint64_t* bar = reinterpret_cast<uint64_t*>(sc + CS_CLOV_U4 * 16 * S);
  int* bad = reinterpret_cast<int*>(bar + 1);
  // the same decision in every CTA of the cluster: the flag was written before
  // the first launch of the sequence, which is no early one
  if (loop_idle(g)) return;
  if (HALO) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x;
  const bool live = tid < S;
  const int s = live ? tid : 0;
  // this cluster's domain: the k-th domain of colour a.colour (see sap_general.cu)
  int D[4];
  {
    const int per = a.snd[0] / 2, k = (int)blockIdx.x / K;
    const int row = k / per, i = k - row * per;
    D[1] = row % a.snd[1];
    D[2] = (row / a.snd[1]) % a.snd[2];
    D[3] = row / (a.snd[1] * a.snd[2]);
    D[0] = 2 * i + ((a.colour + D[1] + D[2] + D[3]) & 1);
  }
  const long long jd = ((long long)(D[3] * a.snd[2] + D[2]) * a.snd[1] + D[1]) * a.snd[0] + D[0];
  const size_t slice_id = (size_t)jd * K + lt;
  if (tid == 0) {
    const unsigned addr = static_cast<unsigned>(__cvta_generic_to_shared(bar));
    const unsigned lbytes = 4 * CS_LINK_H2 * 4 * S, cbytes = CS_CLOV_U4 * 16 * S;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(addr) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr),
                 "r"(lbytes + cbytes + a.extra_tx)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(sl))),
                 "l"(a.links + slice_id * lbytes), "r"(lbytes), "r"(addr)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     static_cast<unsigned>(__cvta_generic_to_shared(sc))),
                 "l"(a.clov + slice_id * cbytes), "r"(cbytes), "r"(addr)
                 : "memory");
  }
  int lc[4], X[4];
  lc[0] = s % a.sd[0];
  lc[1] = (s / a.sd[0]) % a.sd[1];
  lc[2] = s / (a.sd[0] * a.sd[1]);
  lc[3] = lt;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) X[mu] = D[mu] * a.sd[mu] + lc[mu];
  int dom, st;
  coords_to_internal(g, X, dom, st);
  for (int i = tid; i < 6 * CS_GHOST; i += blockDim.x)
    xb[(i / CS_GHOST) * (S + CS_GHOST) + S + i % CS_GHOST] = make_float4(0.f, 0.f, 0.f, 0.f);
  // links and C_inv are constant; everything from here on is not
  if (HALO) asm volatile("griddepcontrol.wait;" ::: "memory");
  HalfSpinor<float> hin[4];
  Spinor<float> src;
  if (live) {
    if (a.do_surface) {
      if (HALO) {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) cs_halo_read(a, D, jd, lc, mu, hin[mu]);
      } else {
        cs_prefetch_surface(a, X, lc);
      }
    }
    cs_read_x(g, a.s_in, dom, st, src);
  }
  __syncthreads();  // barrier initialisation visible to every thread
  {
    // every CTA of the cluster takes the same decision on a wait that gave up
    const bool ok = cs_wait(bar);
    const int cta_bad = __syncthreads_or(!ok);
    if (tid == 0) *bad = cta_bad;
    cl.sync();
    int any = 0;
    for (int r = 0; r < K; ++r) any |= *cl.map_shared_rank(bad, r);
    if (any) {
      if (tid == 0) atomicExch(a.status, QCD_ERR_TIMEOUT);
      if (cta_bad) cs_wait(bar);
      cl.sync();
      return;
    }
  }
  Spinor<float> acc;
  if (a.do_surface && live) {
    zero(acc);
    if (HALO) {
      cs_halo_in<0>(a, sl, D, jd, X, lc, s, hin[0], acc);
      cs_halo_in<1>(a, sl, D, jd, X, lc, s, hin[1], acc);
      cs_halo_in<2>(a, sl, D, jd, X, lc, s, hin[2], acc);
      if (lt == K - 1 || lt == 0) cs_halo_in<3>(a, sl, D, jd, X, lc, s, hin[3], acc);
    } else {
      cs_inter<0>(a, sl, X, lc, s, acc);
      cs_inter<1>(a, sl, X, lc, s, acc);
      cs_inter<2>(a, sl, X, lc, s, acc);
      if (lt == K - 1 || lt == 0) cs_inter<3>(a, sl, X, lc, s, acc);
    }
    cs_clover(sc, s, acc);
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        src.v[sp][c].re = fmaf(a.kappa, acc.v[sp][c].re, src.v[sp][c].re);
        src.v[sp][c].im = fmaf(a.kappa, acc.v[sp][c].im, src.v[sp][c].im);
      }
  }
  float4* below = lt > 0 ? cl.map_shared_rank(t_up, lt - 1) : nullptr;
  float4* above = lt < K - 1 ? cl.map_shared_rank(t_dn, lt + 1) : nullptr;
  if (live) {
    cs_store_x(xb, S + CS_GHOST, s, src);
    cs_push_t(below, above, sl, S, s, src);
  }
  cs_arrive();
  cs_wait_all();  // every slice holds x_0 and its neighbours' half spinors
  const bool fx = lc[0] < a.sd[0] - 1, fy = lc[1] < a.sd[1] - 1, fz = lc[2] < a.sd[2] - 1;
  const bool bx = lc[0] > 0, by = lc[1] > 0, bz = lc[2] > 0;
  Spinor<float> xk = src;  // this site's current iterate
  const int napp = a.n_jac + (a.do_update ? 1 : 0);
  for (int it = 0; it < napp; ++it) {
    const bool more = it + 1 < napp;
    if (live) {
      zero(acc);
      // A direction one site wide has no hops inside: left out where several
      // are (no halo; 16x4x1x1 domains 645 -> 595 us), else the branches cost
      // more than they save (16x6x4x3 588 -> 596 us).
      if (HALO || a.sd[0] > 1) cs_intra_space<0>(xb, sl, S, s, 1, fx, bx, acc);
      if (HALO || a.sd[1] > 1) cs_intra_space<1>(xb, sl, S, s, a.sd[0], fy, by, acc);
      if (HALO || a.sd[2] > 1) cs_intra_space<2>(xb, sl, S, s, a.sd[0] * a.sd[1], fz, bz, acc);
      HalfSpinor<float> h, uh;
      if (above) {
        cs_load_half(t_up, S, s, h);
        su3_mul(cs_link(sl, S, 3, s), h, uh);
        accumulate<3, -1>(acc, uh);
      }
      if (below) {
        cs_load_half(t_dn, S, s, uh);
        accumulate<3, +1>(acc, uh);
      }
    }
    if (more) cs_arrive();  // this thread has read x and the half spinors
    if (live) {
      cs_clover(sc, s, acc);
      if (it < a.n_jac) {
        // x_k = s + kappa C_inv H_cc x_{k-1}
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            xk.v[sp][c].re = fmaf(a.kappa, acc.v[sp][c].re, src.v[sp][c].re);
            xk.v[sp][c].im = fmaf(a.kappa, acc.v[sp][c].im, src.v[sp][c].im);
          }
      } else {
        // s + b - x + kappa C_inv H_cc x
        Spinor<float> b;
        cs_read_x(g, a.b, dom, st, b);
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float re = src.v[sp][c].re + b.v[sp][c].re - xk.v[sp][c].re;
            const float im = src.v[sp][c].im + b.v[sp][c].im - xk.v[sp][c].im;
            acc.v[sp][c].re = fmaf(a.kappa, acc.v[sp][c].re, re);
            acc.v[sp][c].im = fmaf(a.kappa, acc.v[sp][c].im, im);
          }
        a.s_out.store(g, dom, st, acc);
      }
    }
    if (more) {
      cs_wait_all();  // every slice has read the old x and half spinors
      if (live) {
        cs_store_x(xb, S + CS_GHOST, s, xk);
        cs_push_t(below, above, sl, S, s, xk);
      }
      cs_arrive();
      cs_wait_all();  // and now holds the new ones
    }
  }
  if (!live) return;
  a.x.store(g, dom, st, xk);
  if (HALO && a.do_halo) {
    cs_halo_out<0>(a, sl, D, jd, lc, s, xk);
    cs_halo_out<1>(a, sl, D, jd, lc, s, xk);
    cs_halo_out<2>(a, sl, D, jd, lc, s, xk);
    if (lt == K - 1 || lt == 0) cs_halo_out<3>(a, sl, D, jd, lc, s, xk);
  }
}

// ---------------------------------------------------------------------------
// staging layout and launches
// ---------------------------------------------------------------------------
// one thread per site: its links and C_inv, float16, into the domain-slice
// staging layout [domain][slice][mu][site][10 half2] and [domain][slice][site][9 uint4]
__global__ void build_cluster_stage_kernel(Geom g, int sd0, int sd1, int sd2, int sd3, int snd0, int snd1,
                                           int snd2, const double2* u64, const double2* cinv64, __half2* l16,
                                           __half2* c16) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= g.vol) return;
  int X[4];
  site_coords(g, n, X);
  int dom, s;
  coords_to_internal(g, X, dom, s);
  const int sd[4] = {sd0, sd1, sd2, sd3};
  int D[4], l[4];
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    D[mu] = X[mu] / sd[mu];
    l[mu] = X[mu] - D[mu] * sd[mu];
  }
  const int S = sd0 * sd1 * sd2;
  const long long jd = ((long long)(D[3] * snd2 + D[2]) * snd1 + D[1]) * snd0 + D[0];
  const size_t slice_id = (size_t)jd * sd3 + l[3];
  const int site = l[0] + sd0 * (l[1] + sd1 * l[2]);
  for (int mu = 0; mu < 4; ++mu) {
    __half2* dst = l16 + slice_id * 4 * S * CS_LINK_H2 + ((size_t)mu * S + site) * CS_LINK_H2;
    for (int e = 0; e < 9; ++e) {
      const double2 v = u64[(((size_t)((dom * 4 + mu) * 9 + e)) << g.logvd) + s];
      dst[e] = __floats2half2_rn((float)v.x, (float)v.y);
    }
    dst[9] = __floats2half2_rn(0.f, 0.f);
  }
  __half2* h = c16 + (slice_id * S + site) * (CS_CLOV_U4 * 4);
  for (int b = 0; b < 2; ++b)
    for (int k = 0; k < 18; ++k) {
      const double2 v = cinv64[(((size_t)(dom * 36 + 18 * b + k)) << g.logvd) + s];
      h[18 * b + k] = __floats2half2_rn((float)v.x, (float)v.y);
    }
}

// a domain whose time slices fit the cluster kernel: at most CS_MAX_K
// slices of at most CS_MAX_SLICE sites
bool sap_cluster_fits(const int d[4]) {
  const long long S = (long long)d[0] * d[1] * d[2];
  return d[3] >= 1 && d[3] <= CS_MAX_K && S >= 1 && S <= CS_MAX_SLICE;
}

bool sap_cluster_eligible(const qcd_ctx* ctx, int sap_prec) {
  if (!ctx->sap_general || sap_prec != QCD_PREC_HALF_GAUGE) return false;
  return sap_cluster_fits(ctx->sap_dom);
}

// build (or rebuild after a new clover term or domain) the staging copy
static void cluster_staging(qcd_ctx* ctx, cudaStream_t st) {
  const int* d = ctx->sap_dom;
  bool same = ctx->cl_gen == ctx->clover_gen && ctx->cl_link && ctx->cl_clov;
  for (int mu = 0; mu < 4; ++mu) same = same && ctx->cl_dom[mu] == d[mu];
  if (same) return;
  const Geom& g = ctx->geom;
  if (!ctx->cl_link) {
    QCD_CUDA_CHECK(cudaMalloc(&ctx->cl_link, (size_t)g.vol * 4 * CS_LINK_H2 * sizeof(__half2)));
    QCD_CUDA_CHECK(cudaMalloc(&ctx->cl_clov, (size_t)g.vol * CS_CLOV_U4 * 16));
  }
  LaunchScope ls(ctx, QCD_KC_OTHER, st);
  build_cluster_stage_kernel<<<grid_for(g.vol, 128), 128, 0, st>>>(
      g, d[0], d[1], d[2], d[3], g.L[0] / d[0], g.L[1] / d[1], g.L[2] / d[2], ctx->u64, ctx->cinv64,
      (__half2*)ctx->cl_link, (__half2*)ctx->cl_clov);
  check_launch();
  for (int mu = 0; mu < 4; ++mu) ctx->cl_dom[mu] = d[mu];
  ctx->cl_gen = ctx->clover_gen;
}

// M_SAP with one cluster per domain, nrhs stacked float32 fields
void sap_cluster_apply(qcd_ctx* ctx, float4* x, const float4* b, int nrhs, int n_sap, int n_jac, void* ws_s,
                       void* halo, cudaStream_t st) {
  cluster_staging(ctx, st);
  ClusterSapArgs a;
  a.g = ctx->geom;
  long long nsd = 1;
  for (int mu = 0; mu < 4; ++mu) {
    a.sd[mu] = ctx->sap_dom[mu];
    a.snd[mu] = a.g.L[mu] / a.sd[mu];
    nsd *= a.snd[mu];
  }
  a.slice = a.sd[0] * a.sd[1] * a.sd[2];
  a.n_jac = n_jac;
  a.halo = (float4*)halo;
  size_t halo_f4 = 0;
  for (int mu = 0; mu < 4; ++mu) {
    a.face[mu] = a.slice * a.sd[3] / a.sd[mu];
    a.halo_at[mu] = halo_f4;
    halo_f4 += (size_t)3 * nsd * a.face[mu];
  }
  a.kappa = (float)ctx->kappa;
  a.U16 = LinkPtrHalf{ctx->u16};
  a.links = (const unsigned char*)ctx->cl_link;
  a.clov = (const unsigned char*)ctx->cl_clov;
  a.status = ctx->d_status;
  // test hook: wait for 16 bytes that no copy brings, so that the bounded
  // wait gives up (in every CTA of every cluster) and reports QCD_ERR_TIMEOUT
  a.extra_tx = ctx->inject == QCD_INJECT_STAGING_WAIT ? 16 : 0;
  const int K = a.sd[3];
  const int threads = (a.slice + 31) / 32 * 32;
  const size_t smem = (size_t)CS_BYTES_PER_SITE * a.slice + CS_EXTRA_BYTES;
  const size_t v4 = (size_t)a.g.vol * 6;
  // the caller's buffer holds 96 bytes per site; domains with several extents
  // of one, whose faces need more, read the other colour's x in place
  const bool with_halo = halo_f4 <= v4;
  auto kernel = with_halo ? sap_cluster_kernel<true> : sap_cluster_kernel<false>;
  QCD_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((size_t)CS_BYTES_PER_SITE * CS_MAX_SLICE + CS_EXTRA_BYTES)));
  for (int r = 0; r < nrhs; ++r) {
    a.b = F32Spinor{(float4*)b + r * v4};
    a.x = F32Spinor{x + r * v4};
    a.s_out = F32Spinor{(float4*)ws_s + r * v4};
    for (int sweep = 0; sweep <= n_sap; ++sweep) {
      a.s_in = sweep == 0 ? a.b : a.s_out;
      a.do_update = sweep == n_sap ? 0 : 1;
      for (int colour = 0; colour < 2; ++colour) {
        a.colour = colour;
        a.do_surface = (sweep == 0 && colour == 0) ? 0 : 1;
        a.do_halo = (sweep == n_sap && colour == 1) ? 0 : 1;
        LaunchScope ls(ctx, QCD_KC_SAP_BLOCK, st);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(nsd / 2 * K));
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = K;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        // early start: not the first launch (what ran before may have built the
        // staging copy), nor the kernel that reads x through L1
        cfg.numAttrs = with_halo && (r > 0 || sweep > 0 || colour > 0) ? 2 : 1;
        QCD_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kernel, a));
        check_launch();
      }
    }
  }
}

}  // namespace qcd
