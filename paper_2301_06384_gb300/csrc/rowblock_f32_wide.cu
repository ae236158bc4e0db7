// Instances of the tall-skinny block kernels (rowblock.cuh), one translation unit per stored
// type so that they compile in parallel.
#include "rowblock.cuh"

namespace kb {
namespace rb {
template int launch_w<float, 64>(int, const RowArgs<float> &, cudaStream_t, int *);
template int launch_w<float, 128>(int, const RowArgs<float> &, cudaStream_t, int *);
}  // namespace rb
}  // namespace kb
