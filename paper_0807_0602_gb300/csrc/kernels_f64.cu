// FP64 instantiation of the step (standard species) and its reductions.  Built with
// --fmad=false: every product and sum of the canonical order is rounded on
// its own, so the results equal a plain FP64 evaluation of the same order.
#include "lbm_launch.cuh"

namespace sc {

__global__ void __launch_bounds__(kMassThreads) k_mass_final(const RunDesc* __restrict__ runs,
                                                             const double* __restrict__ partials,
                                                             double* __restrict__ mass, uint32_t* __restrict__ err) {
    double M[2];
    mass_total(runs[blockIdx.x], partials, err, M);
    if (threadIdx.x == 0) {
        mass[2 * blockIdx.x + 0] = M[0];
        mass[2 * blockIdx.x + 1] = M[1];
    }
}

template struct Launch<double>;
template struct Step<double, false>;

}  // namespace sc
