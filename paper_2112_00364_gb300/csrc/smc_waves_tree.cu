// smc_waves_tree.cu -- the wave kernels of the rate-shift model, FP64, and the geometric program (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_RATESHIFT, double>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);
template cudaError_t launch_kind<SMC_MODEL_GEOMETRIC, double>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);
template cudaError_t launch_kind<SMC_MODEL_GEOMETRIC, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
