// One part of the products' instantiations (-DBITCOS_PART=n; the parts are listed in gemv_inst.cuh).
#include "gemv.cuh"
#define BITCOS_INST template
#include "gemv_inst.cuh"
