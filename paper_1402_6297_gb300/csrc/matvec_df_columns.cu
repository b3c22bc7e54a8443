// Column kernels of the A_r product in double-single arithmetic (matvec_df.cu),
// a translation unit of their own because they take longest to compile.
#include "dfloat.cuh"
#include "matvec_impl.cuh"

namespace nfs {
NFS_INSTANTIATE_COLUMNS(df)
}  // namespace nfs
