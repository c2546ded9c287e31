// adacad.cuh -- dynamic contrast strength from materialised log-probabilities.
#pragma once
#include "common.cuh"

namespace pced {

// beta[b][k-1] = Jensen-Shannon divergence in bits between rows b*(N+1)+k and
// b*(N+1) of lp [B*(N+1)][V].  pdl: launched as a programmatic dependent of the
// stream's previous kernel.
cudaError_t adacad_beta_launch(const float* lp, int32_t B, int32_t N, int32_t V, float* beta, bool pdl,
                               cudaStream_t stream);

}  // namespace pced
