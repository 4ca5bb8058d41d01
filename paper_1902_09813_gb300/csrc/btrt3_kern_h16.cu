// btrt3_kern_h16.cu -- D3Q19 sweep, FP32 compute with FP16 or BF16 storage (both shifts).
#include "../../include/btrt.h"
#include "btrt_launch3.cuh"

namespace btrt {

// Two nodes per thread for constant coefficients (256^3 hill, FP16 local shift, 20 steps:
// 5.36 ms against 6.56 with a node per thread).  Per-node coefficients were slower that
// way (250 x 131 x 200: 7.14 ms at three blocks per SM against 6.56).  Below 2^17 nodes
// both take the same time, set by the launches (48^3, 50 steps: 334 us).
constexpr long long kPairNodes = 1 << 17;

cudaError_t launch_sweep3_f32_h16(const Sweep3Params<float> &p, int storage, int shift, int mode, cudaStream_t s) {
    const bool vec = !p.first && mode != kGeneral && (long long)p.nx * p.ny * p.nz >= kPairNodes;
    if (storage == BTRT_F16)
        return vec ? launch3_vec<__half>(p, shift, mode, s) : launch3_f32_storage<__half>(p, shift, mode, s);
    return vec ? launch3_vec<__nv_bfloat16>(p, shift, mode, s) : launch3_f32_storage<__nv_bfloat16>(p, shift, mode, s);
}

}  // namespace btrt
