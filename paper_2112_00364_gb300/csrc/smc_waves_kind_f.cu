// smc_waves_kind_f.cu -- the wave kernels of the linear-Gaussian and CRBD models, FP32 (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_LG, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);
template cudaError_t launch_kind<SMC_MODEL_CRBD, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
