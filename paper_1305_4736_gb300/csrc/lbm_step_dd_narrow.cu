// lbm_step_dd_narrow.cu -- the double-float kernels on DdNarrowShape tiles.
#include "lbm_step_dd.cuh"

template struct lbm::DdOps<lbm::DdNarrowShape>;
