// k_primal in float for the fourth-order equations (thirteen-point biharmonic).
#include "rd_band.cuh"

namespace rd {
RD_PRIMAL_KIND(float, KK_CH_IMPL)
RD_PRIMAL_KIND(float, KK_CH_SPLIT)
RD_PRIMAL_KIND(float, KK_NONE_BIH)
}  // namespace rd
