// btrt_tbn_f16.cu -- several steps per launch, FP32 compute with f16 storage.
#include "btrt_internal.h"
#include "btrt_tbn.cuh"

namespace btrt {

cudaError_t launch_sweep_tbn_f16(const SweepParams<float> &p, TbnSteps<float> &st, int shift, int mode, int *rounds,
                                 cudaStream_t s) {
    return launch_tbn_storage<__half>(p, st, shift, mode, rounds, s);
}

}  // namespace btrt
