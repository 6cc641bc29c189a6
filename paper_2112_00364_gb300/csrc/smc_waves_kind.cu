// smc_waves_kind.cu -- the wave kernels of the linear-Gaussian and CRBD models (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_LG>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);
template cudaError_t launch_kind<SMC_MODEL_CRBD>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);

}  // namespace smc
