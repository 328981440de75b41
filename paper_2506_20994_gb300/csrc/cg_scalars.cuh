// Device-side scalars of one CG run (cg.cu) and the two formulas that other
// kernels evaluate for it.
#pragma once

#include "common.cuh"

namespace ax {

struct CgScalars {
  double rz, rr, rr0, pap, alpha, beta;
  int status;     // 0 ok, 1 breakdown (p.Ap <= 0 or non-finite)
  int use_corr;   // flexible CG: 1 if the learned correction is in z
  int fallbacks;  // flexible CG: steps that fell back to Jacobi
  unsigned ticket;  // blocks done of the reduction in flight (finish_sums)
};

// What the host tests for convergence, in pinned host memory: the reduction
// that forms rr writes it there itself, seq last, and the host polls seq.  (A
// copy of the scalars and a stream synchronisation cost some 15 us per test,
// through which the GPU stood idle.)
struct CgMail {
  double rr;
  int status, fallbacks;
  unsigned seq;
};
struct CgMailTo {
  CgMail *mail = nullptr;  // null: none
  unsigned seq = 0;
};
AX_D void cg_post(const CgMailTo &to, const CgScalars *s, double rr, int status) {
  if (!to.mail) return;
  volatile CgMail *m = to.mail;
  m->rr = rr;
  m->status = status;
  m->fallbacks = __ldcg(&s->fallbacks);
  __threadfence_system();
  m->seq = to.seq;
}

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
// gather-scatter that follows the apply, which then sets alpha.  chained: the
// gather-scatter may begin while the apply ends.
struct AlphaJob {
  const double *partials = nullptr;
  int n = 0;
  CgScalars *s = nullptr;
  bool chained = true;
};

}  // namespace ax
