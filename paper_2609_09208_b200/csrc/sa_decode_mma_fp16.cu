// Instantiations of the decode kernel (see sa_decode_mma.cuh): the unquantised binary16 cache, textbook
// softmax(Q K^T / sqrt(d)) V of eq. (1) with FP32 accumulation.
#include "sa_decode_mma.cuh"

namespace sa {
template <int D>
static void launch(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = fp16_shape(D);
    launch_mma<D, FMT_FP16, 16, sh.warps, sh.blocks_per_sm, sh.stages>(a, grid, s);
}
void launch_mma_fp16(int d, const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    if (d == 64) launch<64>(a, grid, s);
    else launch<128>(a, grid, s);
}
}  // namespace sa
