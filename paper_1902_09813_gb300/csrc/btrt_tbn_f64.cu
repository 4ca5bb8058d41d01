// btrt_tbn_f64.cu -- several steps per launch, FP64 and double-word.
#include "btrt_internal.h"
#include "btrt_tbn.cuh"

namespace btrt {

cudaError_t launch_sweep_tbn_f64(const SweepParams<double> &p, TbnSteps<double> &st, int mode, int *rounds, cudaStream_t s) {
    return launch_tbn_sh<double, double, kShiftNone>(p, st, mode, rounds, s);
}
cudaError_t launch_sweep_tbn_dw(const SweepParams<dw> &p, TbnSteps<dw> &st, int mode, int *rounds, cudaStream_t s) {
    return launch_tbn_sh<dw, dw, kShiftNone>(p, st, mode, rounds, s);
}

}  // namespace btrt
