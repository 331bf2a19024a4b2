// lbm_step_dd_wide.cu -- the double-float kernels on DdWideShape tiles.
#include "lbm_step_dd.cuh"

template struct lbm::DdOps<lbm::DdWideShape>;
