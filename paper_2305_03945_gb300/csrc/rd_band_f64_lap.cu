// k_primal in double for the second-order equations (five-point Laplacian).
#include "rd_band.cuh"

namespace rd {
RD_PRIMAL_KIND(double, KK_NONE_LAP)
RD_PRIMAL_KIND(double, KK_AC)
}  // namespace rd
