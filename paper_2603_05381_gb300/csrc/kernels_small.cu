// Instantiations of the kernel that decodes several small shots per warp (decode_small.cuh):
// 8, 16, 24 and 32 rows, FP32 and 16-bit messages.
#include "decode_small.cuh"
#include "device.cuh"

namespace bp4m {
namespace {

template <typename MS>
cudaError_t dispatch_small(int list, const DecodeArgs& a, int num_sms, cudaStream_t st, bool prep) {
    switch (list) {
        case 0: return run_small<8, 8, MS>(a, num_sms, st, prep);
        case 1: return run_small<16, 16, MS>(a, num_sms, st, prep);
        case 2: return run_small<32, 24, MS>(a, num_sms, st, prep);
        case 3: return run_small<32, 32, MS>(a, num_sms, st, prep);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_decode_small(int precision, int list, const DecodeArgs& a, int num_sms, cudaStream_t st,
                                bool prepare_only) {
    if (precision == 1) return dispatch_small<float>(list, a, num_sms, st, prepare_only);
    if (precision == 2) return dispatch_small<__half>(list, a, num_sms, st, prepare_only);
    if (precision == 3) return dispatch_small<__nv_bfloat16>(list, a, num_sms, st, prepare_only);
    return cudaErrorInvalidValue;
}

}  // namespace bp4m
