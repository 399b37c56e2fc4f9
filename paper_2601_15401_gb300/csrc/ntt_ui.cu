// Instantiations of the inverse two-phase NTT kernels of uniform launches
// (general products; ntt_kernel.cuh); a translation unit of its own so that
// they compile in parallel.
#include "ntt_kernel.cuh"

namespace ckks {

cudaError_t ntt_two_ui(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                       const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    return dispatch_two<false, false, false>(logn, P, J, jobs, n_jobs, L, S, G);
}

}  // namespace ckks
