// acct_bf16.cu -- the account-resident ADMM (acct_admm.cuh) with the rows of B in BF16.
#include "acct_admm.cuh"

namespace prism {

cudaError_t launch_acct_bf16(const AcctArgs<float>& A, const AcctShape& sh, int n, cudaStream_t st) {
    return launch_acct_float<__nv_bfloat16>(A, sh, n, st);
}

}  // namespace prism
