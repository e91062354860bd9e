// Instantiations of the decode kernel (see sa_decode_mma.cuh): uniform INT8 keys.
#include "sa_decode_mma.cuh"

namespace sa {
template <int D, int FMT, int CODE, int KB>
static void launch(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = mma_shape(D, KB);
    launch_mma<D, FMT, CODE, sh.warps, sh.blocks_per_sm, sh.stages>(a, grid, s);
}
void launch_mma_int8(int d, const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    if (d == 64) launch<64, FMT_INT8, 32, 8>(a, grid, s);
    else launch<128, FMT_INT8, 32, 8>(a, grid, s);
}
}  // namespace sa
