// y transforms of the right-hand side, float (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_y_cols<float>(cudaStream_t, const YDesc&, int);
}  // namespace spectau
