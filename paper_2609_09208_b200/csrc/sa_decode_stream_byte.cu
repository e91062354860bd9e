// Instantiations of the decode kernel of one block per SM (see sa_decode_stream.cuh): byte container, any number of mantissa bits.
#include "sa_decode_stream.cuh"

namespace sa {
void launch_stream_byte(int d, int k, const DecodeArgs& a, cudaStream_t s) {
    if (d == 128) k == 4 ? launch_stream<128, FMT_BYTE, 7>(a, s) : launch_stream<128, FMT_BYTE3, 7>(a, s);
    else k == 4 ? launch_stream<64, FMT_BYTE, 7>(a, s) : launch_stream<64, FMT_BYTE3, 7>(a, s);
}
void launch_stream_lost_copy(const DecodeArgs& a, cudaStream_t s) { launch_stream<64, FMT_BYTE, 7, true>(a, s); }
}  // namespace sa
