// x rows with products, double (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_x_rows<double>(cudaStream_t, const XDesc&);
}  // namespace spectau
