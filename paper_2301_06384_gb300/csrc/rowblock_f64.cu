// Instances of the tall-skinny block kernels (rowblock.cuh), one translation unit per stored
// type so that they compile in parallel.
#include "rowblock.cuh"

namespace kb {
namespace rb {
template int launch_w<double, 16>(int, const RowArgs<double> &, cudaStream_t, int *);
template int launch_w<double, 32>(int, const RowArgs<double> &, cudaStream_t, int *);
template int launch_w<double, 64>(int, const RowArgs<double> &, cudaStream_t, int *);
}  // namespace rb
}  // namespace kb
