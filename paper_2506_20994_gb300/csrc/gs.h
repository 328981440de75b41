// Library-internal entry points of the gather-scatter (gs.cu).
#pragma once

#include "cg_scalars.cuh"

struct ax_gs;

namespace ax {
// The gather-scatter of the solvers' loops: also sets alpha from the apply's
// partials (one extra block).
int gs_sum_alpha(ax_gs *g, double *v, const AlphaJob &job, cudaStream_t st);
int gs_sum_alpha(ax_gs *g, float *v, const AlphaJob &job, cudaStream_t st);
}  // namespace ax
