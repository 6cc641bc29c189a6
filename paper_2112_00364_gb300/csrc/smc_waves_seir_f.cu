// smc_waves_seir_f.cu -- the wave kernels of the SEIR model, FP32 (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_SEIR, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
