// k_primal in double for the two-species equations.
#include "rd_band.cuh"

namespace rd {
RD_PRIMAL_KIND(double, KK_GS)
RD_PRIMAL_KIND(double, KK_SCHNAK)
}  // namespace rd
