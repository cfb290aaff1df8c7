// FP64 conjugate gradient on M^dag M (Sec. 1 after Eq. 3; Sec. 3): one
// iteration is three fused passes over the lattice,
//   k1  t = M p,                         tt = |t|^2, alpha = rr / tt
//   k2  r -= alpha M^dag t, x += alpha p, rr = |r|^2, beta
//   k3  p = r + beta p
// and the FP64 true residual r = phi - M^dag (M x) used to stop the solve
// and, for mixed-precision solves, as the reliable update.  The operator is
// the fixed-point one of lq_fix64.cuh.
#include "lq_internal.h"
#include "lq_fix64.cuh"

namespace lq {

void cg64_step(lq_ctx* c, int which, double kappa, cudaStream_t stream) {
  const FixGauge U = fix_gauge_of(c);
  if (which == 1) {
    FixEpiCG1 e1{{c->t64.ref(), c->state}};
    launch_dslash_fix<false>(c->geo, U, c->p64.ref(), kappa, e1, c->rs, stream);
  } else {
    FixEpiCG2 e2{{c->r64.ref(), c->x64.ref(), c->p64.ref(), c->state}};
    launch_dslash_fix<true>(c->geo, U, c->t64.ref(), kappa, e2, c->rs, stream);
  }
}

void cg64_iteration(lq_ctx* c, double kappa, cudaStream_t stream) {
  cg64_step(c, 1, kappa, stream);
  cg64_step(c, 2, kappa, stream);
  launch_xpay_p(c->geo, SStore::F64, c->r64.ref(), c->p64.ref(), c->state, false, stream);
}

template <SStore SLO, bool STORE_LO>
static void residual(lq_ctx* c, double kappa, SpinorRef rlo, cudaStream_t stream) {
  FixEpiResidual<SLO, STORE_LO> e{c->phi64.ref(), c->r64.ref(), rlo, FinSolver{c->state}};
  launch_dslash_fix<true>(c->geo, fix_gauge_of(c), c->tmp64.ref(), kappa, e, c->rs, stream);
}

void cg64_true_residual(lq_ctx* c, double kappa, int store_lo_prec, cudaStream_t stream) {
  FixEpiStore e0{c->tmp64.ref()};
  launch_dslash_fix<false>(c->geo, fix_gauge_of(c), c->x64.ref(), kappa, e0, c->rs, stream);
  if (store_lo_prec == LQ_F64) {
    residual<SStore::F64, false>(c, kappa, SpinorRef{nullptr, nullptr}, stream);
    return;
  }
  const SStore slo = spinor_store_of(store_lo_prec);
  SpinorRef rlo = c->r_lo[(int)slo].ref();
  switch (slo) {
    case SStore::F32: residual<SStore::F32, true>(c, kappa, rlo, stream); break;
    case SStore::F16: residual<SStore::F16, true>(c, kappa, rlo, stream); break;
    case SStore::BF16: residual<SStore::BF16, true>(c, kappa, rlo, stream); break;
    case SStore::I16: residual<SStore::I16, true>(c, kappa, rlo, stream); break;
    default: break;
  }
}

}  // namespace lq
