// x rows with products, float (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_x_rows<float>(cudaStream_t, const XDesc&);
}  // namespace spectau
