// z transforms of the right-hand side, double (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_z_cols<double>(cudaStream_t, const ZDesc&, int, bool);
}  // namespace spectau
