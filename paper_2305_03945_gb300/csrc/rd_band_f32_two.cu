// k_primal in float for the two-species equations.
#include "rd_band.cuh"

namespace rd {
RD_PRIMAL_KIND(float, KK_GS)
RD_PRIMAL_KIND(float, KK_SCHNAK)
}  // namespace rd
