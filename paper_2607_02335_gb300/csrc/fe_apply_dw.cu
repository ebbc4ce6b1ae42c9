// fe_apply_dw.cu -- FP64-accurate apply in double-word arithmetic on the FP32 pipe.
#include "fe_apply_launch.cuh"

fe_status fe_launch_apply_f64dw(const ApplyLaunch& L) {
  return launch_apply_v<dw2>(L, L.m->geodw, L.m->xyzdw, static_cast<float*>(L.m->rc_scratch));
}

// The fused kernel saves the launches and passes of the p update and of <q,p>, and pays for them with a
// slower apply and a block reduction per CTA.  FP32 (iterations of the mixed solve, fused against
// separate): Q5 12^3 39 against 44 us, Q3 24^3 47 against 54, Q5 20^3 67 against 73, equal from 6 million
// entries on.  FP64: Q4 12^3 44.6 against 47.0 us where single cells are taken, slower above (Q3 32^3 141
// against 134).
bool fe_apply_fuses_cg(const fe_mesh* m, int prec) {
  if (m->d.geom_mode == FE_GEOM_RECOMPUTE || m->packed) return false;
  if (prec == FE_F32) return m->ncw <= 4ll << 20;
  return pair_single(m->ncells, m->n, fe_sm_count());
}
