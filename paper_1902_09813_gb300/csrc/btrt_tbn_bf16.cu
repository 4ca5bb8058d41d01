// btrt_tbn_bf16.cu -- several steps per launch, FP32 compute with bf16 storage.
#include "btrt_internal.h"
#include "btrt_tbn.cuh"

namespace btrt {

cudaError_t launch_sweep_tbn_bf16(const SweepParams<float> &p, TbnSteps<float> &st, int shift, int mode, int *rounds,
                                 cudaStream_t s) {
    return launch_tbn_storage<__nv_bfloat16>(p, st, shift, mode, rounds, s);
}

}  // namespace btrt
