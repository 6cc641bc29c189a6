// smc_waves_seir.cu -- the wave kernels of the SEIR model (smc_waves.cuh).
#include "smc_waves.cuh"

namespace smc {

template cudaError_t launch_kind<SMC_MODEL_SEIR>(const WaveChain&, const RunDev*, int, cudaStream_t, unsigned,
                                              bool);

}  // namespace smc
