// Device-side scalars of one CG run (cg.cu) and the two formulas that other
// kernels evaluate for it.
#pragma once

#include "common.cuh"

namespace ax {

struct CgScalars {
  double rz, rz_new, rr, rr0, pap, alpha, beta;
  int status;     // 0 ok, 1 breakdown (p.Ap <= 0 or non-finite)
  int use_corr;   // flexible CG: 1 if the learned correction is in z
  int fallbacks;  // flexible CG: steps that fell back to Jacobi
  unsigned ticket;  // blocks done of the reduction in flight (finish_sums)
};

// alpha = rz / <p, Ap>
AX_D void cg_set_alpha(CgScalars *s, double pap) {
  const double rz = __ldcg(&s->rz);
  s->pap = pap;
  if (!(pap > 0.0) || !isfinite(pap) || !isfinite(rz)) {
    s->status = 1;
    s->alpha = 0.0;
  } else {
    s->alpha = rz / pap;
  }
}

// The apply's partials of <p, Ap>, summed by one extra block of the
// gather-scatter that follows the apply, which then sets alpha.
struct AlphaJob {
  const double *partials = nullptr;
  int n = 0;
  CgScalars *s = nullptr;
};

}  // namespace ax
