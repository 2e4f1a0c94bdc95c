// z transforms of the right-hand side, float (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_z_cols<float>(cudaStream_t, const ZDesc&, int, bool);
}  // namespace spectau
