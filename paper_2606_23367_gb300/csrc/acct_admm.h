// acct_admm.h -- the account-resident ADMM kernel (acct_admm.cuh): every iteration of an account in
// one launch, its rows of B in shared memory and its entries in registers, one CTA per account
// or a cluster of up to eight that split the account's entries.
#pragma once

#include "internal.h"

namespace prism {

constexpr int ACCT_THREADS = 512;       // largest block
constexpr int ACCT_CLUSTER = 8;         // largest cluster
constexpr size_t ACCT_SMEM = 227 * 1024;   // shared memory of a CTA at most

// T: the arithmetic; the rows of B are kept as BF16 (bf16 mode), FP32 or FP64 (T = double)
template <typename T>
struct AcctArgs {
    int M = 0, N = 0, Npad = 0, K = 0, S = 0;
    // universe, sorted positions
    const __nv_bfloat16* B16p = nullptr;   // Npad x 64: set in the BF16 mode
    const float* B32p = nullptr;           // Npad x 64 (FP32 modes)
    const double* B64 = nullptr;           // Npad x K (T = double)
    const T* f = nullptr;                  // K
    const T* d = nullptr;                  // Npad
    const T* mu = nullptr;                 // Npad
    const float* Cinv = nullptr;           // NRHO x K x K capacitance inverses (T = float; in FP64 the
                                           // kernel forms them itself, for each penalty)
    const float* G = nullptr;              // NRHO x K x K Gram matrices beside it (factor bounds)
    const int* sec_start = nullptr;        // S + 1
    // per entry, dense M x Npad (sorted positions)
    const T *w0 = nullptr, *lo = nullptr, *up = nullptr, *c = nullptr;
    const T* tilt = nullptr;               // shift of mu per entry, or null
    const int* pw_idx = nullptr;           // -1 = plain L1 entry, else its row of the tables; or null
    const T* pw_bp = nullptr;              // MAXBP per row
    const T* pw_sl = nullptr;              // MAXBP - 1 per row
    const int* pw_nbp = nullptr;
    const T *band_lo = nullptr, *band_hi = nullptr;   // M x S
    const T* tau = nullptr;                // M (+inf = no cap)
    const T *flo = nullptr, *fhi = nullptr;           // M x K factor-exposure bounds, or null
    const int* order = nullptr;            // the accounts of this launch, or null: 0, 1, ...
    // state, M x Npad (also the start of a second pass) and per account
    T *z = nullptr, *y = nullptr;
    float* zf = nullptr;                   // what the polish reads (the same array when T = float)
    float *nu = nullptr, *eta_hi = nullptr, *eta_lo = nullptr, *theta = nullptr;
    int *rho_idx = nullptr, *iters = nullptr, *active = nullptr, *status = nullptr, *sflag = nullptr;
    T *s = nullptr, *ys = nullptr;         // M x K (factor-exposure block)
    T *rho_state = nullptr, *theta_state = nullptr;   // FP64: the penalty and the cap's multiplier (M)
    T rho0 = T(3);                         // FP64: the first penalty
    const unsigned long long* t0 = nullptr;   // device clock at the start of the solve
    unsigned long long budget_ns = 0;      // time budget from t0 (0: none)
    T alpha = T(1.5), eps = T(5e-4);
    int max_iter = 4000, min_iter = 20, adapt_every = 25;
    int settle = 0, settle_max = 60;       // iterations without a change of place to wait for once the target
                                           // is met, and for how many iterations to wait
    int resume = 0;                        // 1: z, y, s, ys and the multipliers continue from the state
    int pw_rows = 0;                       // rows of the cost tables that a CTA can keep in shared memory
};

// How one launch is cut: entries per thread, threads and CTAs per account.
struct AcctShape {
    int E = 0, threads = 0, cluster = 0;   // E = 0: the account does not fit
    int pw_rows = 0;
    size_t smem = 0;
};

// The shape for accounts of at most n entries (E = 0: they do not fit). bytes_b: size of an element
// of B, 8 in FP64; fac: factor bounds; pw: some accounts have piecewise-linear cost rows.
AcctShape acct_shape(int n, int K, int bytes_b, bool fac, bool pw);
template <typename T>
cudaError_t launch_acct_admm(const AcctArgs<T>& A, const AcctShape& sh, int n_accounts, cudaStream_t st);
cudaError_t launch_acct_bf16(const AcctArgs<float>& A, const AcctShape& sh, int n_accounts, cudaStream_t st);
cudaError_t launch_acct_fp32(const AcctArgs<float>& A, const AcctShape& sh, int n_accounts, cudaStream_t st);

}  // namespace prism
