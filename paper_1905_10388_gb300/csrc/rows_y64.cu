// y transforms of the right-hand side, double (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_y_cols<double>(cudaStream_t, const YDesc&, int);
}  // namespace spectau
