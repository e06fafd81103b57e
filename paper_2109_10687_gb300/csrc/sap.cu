// SAP preconditioner with Jacobi domain inverses (Sec. 3 of
// arXiv:2109.10687: Eq. Msap, Algorithms 1-3): the choice of kernel.
//
// One kernel launch performs one half-sweep of Algorithm 1 on every domain
// of one colour c (E = 0, O = 1):
//
//   1. surface term (skipped in the first E half-sweep, where x_O = 0):
//        s_c <- s_c - A_{c,c'} x_{c'} = s_c + kappa C_inv H_{c c'} x_{c'};
//   2. Jacobi domain inverse (Algorithm 2):
//        x_0 = s_c,  x_k = s_c + kappa C_inv H_cc x_{k-1}, k = 1..n_jac.
//      This is Algorithm 2 written without the cancelling terms
//      (x + b - (x - kappa C_inv H x) = b + kappa C_inv H x), so
//      x_{n_jac} = sum_{j=0}^{n_jac} (I - A_cc)^j s_c;
//   3. residual update of Algorithm 1 (skipped in the closing sweep):
//        s_c <- s_c + b_c - A_cc x_c = s_c + b_c - x_c + kappa C_inv H_cc x_c.
//
// The whole preconditioner is 2 (n_sap + 1) such launches; A M_SAP adds one
// application of A to the result (Algorithm 3 as A (M_SAP b)).

#include "qcd_internal.cuh"

namespace qcd {

// x = M_SAP b for nrhs stacked float32 fields.  ws_s holds s (float32 or
// float16), halo the block and cluster kernels' face halo (96 bytes per site);
// both are sized for nrhs right-hand sides, which go through every launch
// together.
// Domains set apart from the storage blocks have kernels of their own; 4^4
// storage blocks take the block kernel (which on small lattices may hand over
// to the split one), all others the kernel of sap_block.cu.
void sap_apply_launch(qcd_ctx* ctx, float4* x, const float4* b, int nrhs, int n_sap, int n_jac, int sap_prec,
                      void* ws_s, void* halo, cudaStream_t st) {
  if (ctx->sap_general) {
    sap_general_apply(ctx, x, b, nrhs, n_sap, n_jac, sap_prec, ws_s, halo, st);
    return;
  }
  const bool staged = sap_staged_available(ctx);
  const F32Spinor xs{x}, bs{(float4*)b}, s32{(float4*)ws_s};
  const size_t nv = (size_t)ctx->geom.vol * nrhs;
  const F16Spinor s16{(uint4*)ws_s, (float*)((uint4*)ws_s + 3 * nv)};
  float4* h = (float4*)halo;
  if (sap_prec == QCD_PREC_HALF) {  // float16 links, C_inv and s
    if (staged) sap_staged_sequence_f16(ctx, bs, s16, bs, xs, h, nrhs, n_sap, n_jac, st);
    else sap_block_f16(ctx, s16, xs, bs, nrhs, n_sap, n_jac, st);
  } else if (sap_prec == QCD_PREC_HALF_GAUGE) {  // float16 links and C_inv, float32 vectors
    if (staged) sap_staged_sequence_h16g(ctx, bs, s32, xs, bs, h, nrhs, n_sap, n_jac, st);
    else sap_block_h16g(ctx, s32, xs, bs, nrhs, n_sap, n_jac, st);
  } else {
    if (staged) sap_staged_sequence_f32(ctx, bs, s32, xs, bs, h, nrhs, n_sap, n_jac, st);
    else sap_block_f32(ctx, s32, xs, bs, nrhs, n_sap, n_jac, st);
  }
}

}  // namespace qcd
