// smc_waves_tree_f.cu -- the wave kernels of the rate-shift model, FP32 (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_RATESHIFT, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
