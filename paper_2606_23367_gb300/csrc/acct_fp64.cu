// acct_fp64.cu -- the account-resident ADMM (acct_admm.cuh) in FP64, and the launch shapes.
#include "acct_admm.cuh"

namespace prism {

// ---------------------------------------------------------------------------
// launch shapes
// ---------------------------------------------------------------------------
static size_t acct_fixed(size_t t_bytes) {
    const size_t s = t_bytes == 8 ? sizeof(AcctShared<double>) : sizeof(AcctShared<float>);
    return (s + 15) / 16 * 16;
}

AcctShape acct_shape(int n, int K, int bytes_b, bool fac, bool pw) {
    AcctShape r;
    const bool f64 = bytes_b == 8;
    const size_t t = f64 ? 8 : 4, row = (size_t)PWROW * t;
    const int ldc = (K + 31) / 32 * 32 + 8, ncs = row_stride(K, 16 / bytes_b);
    const size_t fixed = acct_fixed(t) + (size_t)(1 + (fac ? 1 : 0) + (f64 ? 1 : 0)) * K * ldc * t;
    for (int cs = 1; cs <= (f64 ? 1 : ACCT_CLUSTER); cs *= 2) {
        const int nl = std::max(1, cdiv(n, cs));
        if (nl > ACCT_THREADS * (f64 ? 2 : 4)) continue;
        // Few entries: one a thread, so that a small account still spreads over several warps; else
        // four (two in FP64, whose registers hold no more), which divides the cost of the reductions
        // per warp by the most entries.
        r.E = f64 ? (nl <= 256 ? 1 : 2) : ((nl <= 256 && cs == 1) ? 1 : 4);
        r.threads = std::max((cs > 1 || f64) ? 128 : 64, cdiv(cdiv(nl, r.E), 32) * 32);
        r.cluster = cs;
        const size_t slots = (size_t)r.threads * r.E;
        const size_t b = fixed + (f64 ? slots * t : 0) + slots * ncs * 16;
        if (b > ACCT_SMEM) { r.E = 0; continue; }
        // cost rows: for every entry where there is room, else as many as fit
        r.pw_rows = pw ? (int)std::min<size_t>((size_t)nl, (ACCT_SMEM - b) / row) : 0;
        r.smem = b + (size_t)r.pw_rows * row;
        return r;
    }
    return r;
}

template <>
cudaError_t launch_acct_admm<float>(const AcctArgs<float>& A, const AcctShape& sh, int n, cudaStream_t st) {
    return A.B16p ? launch_acct_bf16(A, sh, n, st) : launch_acct_fp32(A, sh, n, st);
}

template <>
cudaError_t launch_acct_admm<double>(const AcctArgs<double>& A, const AcctShape& sh, int n, cudaStream_t st) {
    const bool gen = A.pw_idx || A.flo || A.tau;
    if (sh.E == 1) {
        if (gen) return launch_one<double, double, 1, 256, true, false>(A, sh, n, st);
        return launch_one<double, double, 1, 256, false, false>(A, sh, n, st);
    }
    if (gen) return launch_one<double, double, 2, 512, true, false>(A, sh, n, st);
    return launch_one<double, double, 2, 512, false, false>(A, sh, n, st);
}

}  // namespace prism
