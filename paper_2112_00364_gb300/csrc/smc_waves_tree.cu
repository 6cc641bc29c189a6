// smc_waves_tree.cu -- the wave kernels of the rate-shift model and the geometric program (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_RATESHIFT>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);
template cudaError_t launch_kind<SMC_MODEL_GEOMETRIC>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);

}  // namespace smc
