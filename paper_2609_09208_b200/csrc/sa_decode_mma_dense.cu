// Instantiations of the decode kernel (see sa_decode_mma.cuh): sub-byte containers.
#include "sa_decode_mma.cuh"

namespace sa {
template <int D, int FMT, int CODE, int KB>
static void launch(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = mma_shape(D, KB);
    launch_mma<D, FMT, CODE, sh.warps, sh.blocks_per_sm, sh.stages>(a, grid, s);
}
void launch_mma_dense(int d, int k, const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    if (d == 64) {
        if (k == 0) launch<64, FMT_NIBBLE, 8, 0>(a, grid, s);
        else if (k == 1) launch<64, FMT_PLANAR1, 9, 1>(a, grid, s);
        else launch<64, FMT_PLANAR2, 10, 2>(a, grid, s);
    } else {
        if (k == 0) launch<128, FMT_NIBBLE, 8, 0>(a, grid, s);
        else if (k == 1) launch<128, FMT_PLANAR1, 9, 1>(a, grid, s);
        else launch<128, FMT_PLANAR2, 10, 2>(a, grid, s);
    }
}
}  // namespace sa
