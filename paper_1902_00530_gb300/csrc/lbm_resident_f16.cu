// lbm_resident_f16.cu -- on-chip resident steps of small lattices, f16 population storage.
#include "lbm_internal.h"
#include "lbm_step_staged.cuh"
#include "lbm_step_resident.cuh"

LBM_INSTANTIATE_RESIDENT(lbm::ST_F16, f16)
