// Instantiations of the decode kernel (see sa_decode_mma.cuh): byte container, any number of mantissa bits.
#include "sa_decode_mma.cuh"

namespace sa {
template <int D, int FMT, int CODE, int KB>
static void launch(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = mma_shape(D, KB);
    launch_mma<D, FMT, CODE, sh.warps, sh.blocks_per_sm, sh.stages>(a, grid, s);
}
void launch_mma_byte(int d, int k, const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    if (d == 128) {
        if (k == 4) launch<128, FMT_BYTE, 7, 4>(a, grid, s);
        else launch<128, FMT_BYTE3, 7, 2>(a, grid, s);
    } else if (k == 4) launch<64, FMT_BYTE, 7, 4>(a, grid, s);
    else if (k == 0) launch<64, FMT_BYTE3, 7, 0>(a, grid, s);
    else launch<64, FMT_BYTE3, 7, 2>(a, grid, s);
}
void launch_mma_lost_copy(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = mma_shape(64, 4);
    if (a.whole) launch_mma_as<64, FMT_BYTE, 7, sh.warps, sh.blocks_per_sm, sh.stages, true, true>(a, grid, s);
    else launch_mma_as<64, FMT_BYTE, 7, sh.warps, sh.blocks_per_sm, sh.stages, true, false>(a, grid, s);
}
}  // namespace sa
