// tma_map.h -- tensor maps for the TMA-fed kernels.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

namespace tsm {

// cuTensorMapEncodeTiled from the driver (no link-time dependency on libcuda);
// null when the driver does not have it
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();

// 1: operand copies are withheld (tsm_umma_inject_timeout)
int copies_withheld();

}  // namespace tsm
