// Decoding with 16-bit message storage (IEEE half or bfloat16): the shared-memory kernel and
// the streaming kernel with MS = __half / __nv_bfloat16 and FP32 priors and arithmetic.
// Same tiers as FP32; shots above the widest streaming variant (1024 columns) use the FP32
// general global-memory kernel.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "decode_smem.cuh"
#include "decode_wide.cuh"
#include "device.cuh"

namespace bp4m {
namespace {

template <typename MS>
cudaError_t dispatch_half(int list, const DecodeArgs& a, int num_sms, cudaStream_t st, bool prep) {
    switch (list) {
        case 4: return run_tier2<float, 24, 2, MS>(a, num_sms, st, prep);
        case 5: return run_tier2<float, 32, 2, MS>(a, num_sms, st, prep);
        case 6: return run_tier2<float, 20, 4, MS>(a, num_sms, st, prep);
        case 7: return run_tier2<float, 24, 4, MS>(a, num_sms, st, prep);
        case 8: return run_tier2<float, 28, 4, MS>(a, num_sms, st, prep);
        // 128 rows: two blocks per SM
        case 9: return run_tier2<float, 32, 4, MS>(a, num_sms, st, prep);
        case 10: return run_tier2<float, 36, 4, MS>(a, num_sms, st, prep);
        case 11: return run_tier2<float, 40, 4, MS>(a, num_sms, st, prep);
        default: return cudaErrorInvalidValue;
    }
}

template <typename MS>
cudaError_t dispatch_stream_half(int ch, const DecodeArgs& a, int slots, int num_sms, cudaStream_t st) {
    switch (ch) {
        case 6: return run_wide<6, MS>(a, slots, num_sms, st);
        case 8: return run_wide<8, MS>(a, slots, num_sms, st);
        case 10: return run_wide<10, MS>(a, slots, num_sms, st);
        case 12: return run_wide<12, MS>(a, slots, num_sms, st);
        case 14: return run_wide<14, MS>(a, slots, num_sms, st);
        case 16: return run_wide<16, MS>(a, slots, num_sms, st);
        case 20: return run_wide<20, MS>(a, slots, num_sms, st);
        case 24: return run_wide<24, MS>(a, slots, num_sms, st);
        case 28: return run_wide<28, MS>(a, slots, num_sms, st);
        case 32: return run_wide<32, MS>(a, slots, num_sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_stream_half(int precision, int ch, const DecodeArgs& a, int slots, int num_sms, cudaStream_t st) {
    if (precision == 2) return dispatch_stream_half<__half>(ch, a, slots, num_sms, st);
    if (precision == 3) return dispatch_stream_half<__nv_bfloat16>(ch, a, slots, num_sms, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_decode_list_half(int precision, int list, const DecodeArgs& a, int num_sms, cudaStream_t st,
                                    bool prepare_only) {
    if (list < kSmallLists) return launch_decode_small(precision, list, a, num_sms, st, prepare_only);
    if (precision == 2) return dispatch_half<__half>(list, a, num_sms, st, prepare_only);
    if (precision == 3) return dispatch_half<__nv_bfloat16>(list, a, num_sms, st, prepare_only);
    return cudaErrorInvalidValue;
}

}  // namespace bp4m
