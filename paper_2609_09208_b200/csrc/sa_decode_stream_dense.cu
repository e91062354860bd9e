// Instantiations of the decode kernel of one block per SM (see sa_decode_stream.cuh): sub-byte containers.
#include "sa_decode_stream.cuh"

namespace sa {
template <int D>
static void launch(int k, const DecodeArgs& a, cudaStream_t s) {
    if (k == 0) launch_stream<D, FMT_NIBBLE, 8>(a, s);
    else if (k == 1) launch_stream<D, FMT_PLANAR1, 9>(a, s);
    else launch_stream<D, FMT_PLANAR2, 10>(a, s);
}
void launch_stream_dense(int d, int k, const DecodeArgs& a, cudaStream_t s) { d == 64 ? launch<64>(k, a, s) : launch<128>(k, a, s); }
}  // namespace sa
