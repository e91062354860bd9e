// Instantiations of the decode kernel of one block per SM (see sa_decode_stream.cuh): uniform INT8 keys and the binary16 cache.
#include "sa_decode_stream.cuh"

namespace sa {
void launch_stream_int8(int d, const DecodeArgs& a, cudaStream_t s) { d == 64 ? launch_stream<64, FMT_INT8, 32>(a, s) : launch_stream<128, FMT_INT8, 32>(a, s); }
void launch_stream_fp16(int d, const DecodeArgs& a, cudaStream_t s) { d == 64 ? launch_stream<64, FMT_FP16, 16>(a, s) : launch_stream<128, FMT_FP16, 16>(a, s); }
}  // namespace sa
