// smc_waves_ds_f.cu -- the wave kernels of the delayed-sampling CRBD, FP32 (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_CRBD_DS, float>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
