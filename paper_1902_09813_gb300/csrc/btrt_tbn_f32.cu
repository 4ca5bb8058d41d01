// btrt_tbn_f32.cu -- several steps per launch, FP32 compute with f32 storage.
#include "btrt_internal.h"
#include "btrt_tbn.cuh"

namespace btrt {

cudaError_t launch_sweep_tbn_f32(const SweepParams<float> &p, TbnSteps<float> &st, int shift, int mode, int *rounds,
                                 cudaStream_t s) {
    return launch_tbn_storage<float>(p, st, shift, mode, rounds, s);
}

}  // namespace btrt
