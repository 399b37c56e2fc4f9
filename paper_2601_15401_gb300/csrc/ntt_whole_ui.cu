// Instantiations of the inverse one-phase NTT kernels of uniform launches
// (N <= 2^12; ntt_kernel.cuh).
#include "ntt_kernel.cuh"

namespace ckks {

cudaError_t ntt_whole_ui(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                         const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    if (logn <= 8) return dispatch_tiny<false>(logn, P, J, L, S, G);
    return dispatch_whole<false, false>(logn, P, J, jobs, n_jobs, L, S, G);
}

}  // namespace ckks
