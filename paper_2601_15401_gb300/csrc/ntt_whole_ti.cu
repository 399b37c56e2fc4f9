// Instantiations of the inverse one-phase NTT kernels of table-driven launches
// (N <= 2^12; ntt_kernel.cuh).
#include "ntt_kernel.cuh"

namespace ckks {

cudaError_t ntt_whole_ti(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                         const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    return dispatch_whole<false, true>(logn, P, J, jobs, n_jobs, L, S, G);
}

}  // namespace ckks
