// Ordered instances of the tall-skinny block kernels (rowblock.cuh).
#include "rowblock.cuh"

namespace kb {
namespace rb {
template int launch_ordered<16>(int, const RowArgs<float> &, cudaStream_t, int *);
template int launch_ordered<32>(int, const RowArgs<float> &, cudaStream_t, int *);
template int launch_ordered<64>(int, const RowArgs<float> &, cudaStream_t, int *);
template int launch_ordered<128>(int, const RowArgs<float> &, cudaStream_t, int *);
}  // namespace rb
}  // namespace kb
