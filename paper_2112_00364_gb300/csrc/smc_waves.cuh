// smc_waves.cuh -- launching the wave kernels of one model.  A wave of a set of
// runs is one launch per model and CTA size among them (a chain of such launches,
// wave after wave): each kernel holds one model's block table only, so its code
// and registers (one kernel dispatching on each run's model spilled 250 bytes a
// thread at the 64 registers of FP32 particles: 150 us instead of 143 a rate-shift
// wave of 2^20).  Models and precisions have translation units of their own.
#pragma once
#include <cuda_runtime.h>

#include "smc_engine.h"
#include "smc_step.cuh"

namespace smc {

template <int KIND, typename R>
cudaError_t launch_kind(const WaveChain& c, int n_ctas, const RunDev* runs, cudaStream_t st,
                        unsigned wave, bool alone, bool dense) {
  return dense ? launch_bucket<R, KIND, true>(c.bucket, runs, c.map, n_ctas, st, wave, alone)
               : launch_bucket<R, KIND, false>(c.bucket, runs, c.map, n_ctas, st, wave, alone);
}

}  // namespace smc
