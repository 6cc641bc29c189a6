// smc_waves_ds.cu -- the wave kernels of the delayed-sampling CRBD (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_CRBD_DS>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);

}  // namespace smc
