// acct_fp32.cu -- the account-resident ADMM (acct_admm.cuh) with the rows of B in FP32.
#include "acct_admm.cuh"

namespace prism {

cudaError_t launch_acct_fp32(const AcctArgs<float>& A, const AcctShape& sh, int n, cudaStream_t st) {
    return launch_acct_float<float>(A, sh, n, st);
}

}  // namespace prism
