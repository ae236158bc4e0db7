// Instances of the tall-skinny block kernels (rowblock.cuh), one translation unit per stored
// type so that they compile in parallel.
#include "rowblock.cuh"

namespace kb {
namespace rb {
template int launch_w<__nv_bfloat16, 16>(int, const RowArgs<__nv_bfloat16> &, cudaStream_t, int *);
template int launch_w<__nv_bfloat16, 32>(int, const RowArgs<__nv_bfloat16> &, cudaStream_t, int *);
template int launch_w<__nv_bfloat16, 64>(int, const RowArgs<__nv_bfloat16> &, cudaStream_t, int *);
template int launch_w<__nv_bfloat16, 128>(int, const RowArgs<__nv_bfloat16> &, cudaStream_t, int *);
}  // namespace rb
}  // namespace kb
