// smc_waves_ds.cu -- the wave kernels of the delayed-sampling CRBD, FP64 (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_CRBD_DS, double>(const WaveChain&, int, const RunDev*, cudaStream_t, unsigned,
    bool, bool);

}  // namespace smc
