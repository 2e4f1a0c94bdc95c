// batched x rows and z transforms, double (rows.cuh)
#include "rows.cuh"

namespace spectau {
template cudaError_t launch_x_rows_batched<double>(cudaStream_t, const XDesc*, const int4*, int, size_t, int*);
template cudaError_t launch_z_cols_batched<double>(cudaStream_t, bool, const ZDesc*, const int4*, int, size_t, int*);
}  // namespace spectau
