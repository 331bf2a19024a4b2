// lbm_step_dd_mid.cu -- the double-float kernels on DdMidShape tiles.
#include "lbm_step_dd.cuh"

template struct lbm::DdOps<lbm::DdMidShape>;
