// Instantiation of the CUDA-core encode and decode for f32 inputs.
#include "simt_kernels.cuh"

namespace flarepp {

cudaError_t simt_encode_f32(const Plan& p, int call, const void* k, const void* v,
                          const void* seeds, float scale, char* ws, cudaStream_t st) {
    return simt::encode_f32(p, call, (const float*)k, (const float*)v, (const float*)seeds, scale, ws,
                            st);
}

cudaError_t simt_decode_f32(const Plan& p, const void* K, float scale, void* Y, char* ws,
                          cudaStream_t st, float* lse, const float* Qh) {
    return simt::decode_f32(p, (const float*)K, scale, (float*)Y, ws, st, lse, Qh);
}

}  // namespace flarepp
