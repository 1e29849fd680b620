// k_primal in float for the second-order equations (five-point Laplacian).
#include "rd_band.cuh"

namespace rd {
RD_PRIMAL_KIND(float, KK_NONE_LAP)
RD_PRIMAL_KIND(float, KK_AC)
}  // namespace rd
