// sk_step_gauss_mcmcmc_direct_sum32.cu -- step-kernel instantiation for Gaussian (float) couplings, the MCMCMC rule, row a read through L1, 16 lanes with two
// Philox blocks each and the weights added in the whole-warp order (compiled as
// its own translation unit so that the variants build in parallel).
#include "sk_step.cuh"

namespace sk {

cudaError_t launch_step_gauss_mcmcmc_direct_sum32(int nb, int G, const JobDev* jobs, const WorkItem* items,
                           uint32_t n_items, uint32_t* queue, uint32_t nsteps, uint32_t W, uint32_t per_chain,
                           uint32_t grid, cudaStream_t st) {
    if (nb != 2 || G != 16) return cudaErrorInvalidValue;
    return step::launch_g<float, 0, 2, 16, 3>(jobs, items, n_items, queue, nsteps, W, per_chain, grid, st);
}

int occupancy_gauss_mcmcmc_direct_sum32(int nb, int G, uint32_t W, uint32_t per_chain) {
    return nb == 2 && G == 16 ? step::occupancy_g<float, 0, 2, 16, 3>(W, per_chain) : 0;
}

}  // namespace sk
