// lbm_resident_bf16.cu -- on-chip resident steps of small lattices, bf16 population storage.
#include "lbm_internal.h"
#include "lbm_step_staged.cuh"
#include "lbm_step_resident.cuh"

LBM_INSTANTIATE_RESIDENT(lbm::ST_BF16, bf16)
