// solve.cu -- prism_solve_batch: packing, feasibility test, ADMM loop, polish, unpack.
//
// Call structure (one call = one book of accounts, Fig. 2 public solver call):
//   1. validate and pack the ragged FP64 inputs into a sector-sorted M x Npad
//      device layout (FP64 copies for the polish, FP32 copies for the iterations);
//      lot data become per-entry piecewise-linear cost tables (built on the device);
//   2. closed-form capacity test per account (budget, box and bands admit a point);
//      accounts that fail get NO_FEASIBLE_RETURN;
//   3. ADMM iterations: account-resident, all of an account's iterations in one launch
//      (acct_route chooses), or batched over the book, check_every at a time, captured once
//      in a CUDA graph and replayed until every account has converged or hit its cap, the
//      last few accounts account-resident (few_fit);
//   4. FP64 polish rounds and certification; accounts the polish cannot settle go
//      back to the iterations with a tighter target, then fall back to the
//      projected iterate (FEASIBLE_NONCERTIFIED when it passes the gates);
//   5. unpack weights, multipliers, status and diagnostics into the caller's layout.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "acct_admm.h"
#include "block_admm.h"
#include "polish.h"
#include "solver.h"

namespace prism {

// ---------------------------------------------------------------------------
// workspace: one device arena per universe handle, grown on demand
// ---------------------------------------------------------------------------
struct Arena {
    char* base = nullptr;
    size_t cap = 0, used = 0;
    int alloc_fail = 0;
    template <typename T>
    T* take(size_t n) {
        size_t bytes = (n * sizeof(T) + 255) / 256 * 256;
        if (used + bytes > cap) { alloc_fail = 1; return nullptr; }
        T* p = reinterpret_cast<T*>(base + used);
        used += bytes;
        return p;
    }
};

// Launch accounting and, in profile mode, CUDA events around every launch.
struct Prof {
    bool on = false;
    std::vector<cudaEvent_t> pool;
    size_t used = 0;
    struct Mark { int cls; cudaEvent_t a, b; };
    std::vector<Mark> marks;
    int64_t launches[PRISM_NKCLASS] = {};
    cudaEvent_t get() {
        if (used == pool.size()) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            pool.push_back(e);
        }
        return pool[used++];
    }
    void reset() {
        used = 0;
        marks.clear();
        for (auto& l : launches) l = 0;
    }
    template <class F>
    void run(int cls, int nkernels, cudaStream_t st, F f) {
        launches[cls] += nkernels;
        if (!on) { f(); return; }
        cudaEvent_t a = get(), b = get();
        cudaEventRecord(a, st);
        f();
        cudaEventRecord(b, st);
        marks.push_back({cls, a, b});
    }
};

struct SolveCache {
    Prof prof;
    char* arena = nullptr;
    size_t arena_bytes = 0;
    int* pinned = nullptr;          // host-pinned counter readback
    static constexpr size_t BOX = 256 * 1024;
    char* box = nullptr;            // pinned, 2 x BOX: small host inputs on their way in, small outputs back
    cudaGraphExec_t gexec = nullptr;
    Dev gdev;                       // Dev the graph was captured with
    bool have_graph = false;
    int g_iters = 0;
    int64_t g_launches[PRISM_NKCLASS] = {};
    cudaEvent_t ev[6] = {};
    cudaStream_t pst = nullptr;                   // polish of the accounts that stopped iterating
    cudaEvent_t ev_pol = nullptr;
    int* hact = nullptr;                          // pinned: activity flags after each chunk (M)
    int* hsel = nullptr;                          // pinned: polish batch of each account (M)
    int hcap = 0;
    static constexpr int MAXCH = 4;               // independent chains of the fused iterations
    cudaStream_t chst[MAXCH - 1] = {};            // streams of chains 1 .. MAXCH-1 (chain 0: the solve stream)
    cudaEvent_t ev_fork = nullptr, ev_join[MAXCH - 1] = {};
    bool chains_ok = false;
};

static SolveCache& cache_of(prism_universe* uh) {
    static_assert(sizeof(void*) == 8, "64-bit only");
    // one cache per universe handle, stored alongside it
    struct Holder { prism_universe* u; SolveCache c; };
    static std::vector<Holder*> all;
    for (Holder* h : all) if (h->u == uh) return h->c;
    Holder* h = new Holder{uh, SolveCache()};
    all.push_back(h);
    return h->c;
}

void release_cache(prism_universe* uh);

// ---------------------------------------------------------------------------
// pack / validate
// ---------------------------------------------------------------------------
enum : int { ERR_INDEX = 1, ERR_NONFINITE = 2, ERR_BOUNDS = 4, ERR_DUP = 8, ERR_COST = 16, ERR_LEN = 32,
              ERR_LOT_OFFSETS = 64, ERR_LOT_COUNT = 128, ERR_LOT_LOWER = 256, ERR_LOT_DATA = 512, ERR_LOT_SUM = 1024,
              ERR_BENCH = 2048, ERR_TILT = 4096, ERR_BAND = 8192, ERR_CAP = 16384 };

struct PackArgs {
    int M, N, Npad;
    const int64_t* offsets;      // device
    const int32_t* asset_idx;    // device or null
    const double *w0, *lo, *up, *tc;   // device ragged
    const int* inv_perm;
    double *W0, *LO, *UP, *C;
    float *W0f, *LOf, *UPf, *Cf;
    int* member;                 // ragged books: 1 at the account's positions; else null
    int* err;
    int64_t nnz;
};

__global__ void k_pack(PackArgs A) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.nnz) return;
    // account of entry e: last a with offsets[a] <= e (every account spans the universe
    // when there is no asset_idx: then a = e / N)
    int a;
    if (A.asset_idx) {
        int lo = 0, hi = A.M;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (A.offsets[mid] <= e) lo = mid; else hi = mid;
        }
        a = lo;
    } else {
        a = int(e / A.N);
    }
    int i = A.asset_idx ? A.asset_idx[e] : int(e - (int64_t)a * A.N);
    if (i < 0 || i >= A.N) { atomicOr(A.err, ERR_INDEX); return; }
    const double w0 = A.w0[e], l = A.lo[e], u = A.up[e], c = A.tc[e];
    if (!(isfinite(w0) && isfinite(l) && isfinite(u) && isfinite(c))) { atomicOr(A.err, ERR_NONFINITE); return; }
    if (l > u) { atomicOr(A.err, ERR_BOUNDS); return; }
    if (c < 0) { atomicOr(A.err, ERR_COST); return; }
    const size_t d = (size_t)a * A.Npad + A.inv_perm[i];
    if (A.asset_idx) {
        if (atomicExch(&A.member[d], 1) != 0) { atomicOr(A.err, ERR_DUP); return; }
    }                                      // (else position i of account a: no duplicate is possible)
    A.W0[d] = w0; A.LO[d] = l; A.UP[d] = u; A.C[d] = c;
    A.W0f[d] = float(w0); A.LOf[d] = float(l); A.UPf[d] = float(u); A.Cf[d] = float(c);
}

// Everything a solve starts from per account, in one launch, where some 35 memsets and small copies
// stood (each 2-3 us on the stream: 0.12 of the 0.5 ms of a one-account call): bands, caps and factor
// bounds checked and in FP32 too, and the state of the iterations and the polish.
struct SetupArgs {
    int M, S, K, rho_idx, n_ctr;
    const double *band_lo, *band_hi, *tau, *flo, *fhi;     // device; tau, flo and fhi may be null
    double *bd_lo, *bd_hi, *bd_tau, *bd_flo, *bd_fhi;
    float *bd_lof, *bd_hif, *bd_tauf, *bd_flof, *bd_fhif;
    Dev D;
    PolDev P;
    int* err;                                              // [0] flags, [2] some cap is finite
};

__global__ void k_setup(SetupArgs A) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const Dev& D = A.D;
    const PolDev& P = A.P;
    if (e < (int64_t)A.M * A.S) {
        const double lo = A.band_lo[e], hi = A.band_hi[e];
        if (isnan(lo) || isnan(hi) || lo > hi) atomicOr(A.err, ERR_BAND);
        A.bd_lo[e] = lo; A.bd_hi[e] = hi;
        A.bd_lof[e] = float(lo); A.bd_hif[e] = float(hi);
        D.eta_hi[e] = D.eta_lo[e] = __int_as_float(-1);    // NaN: no warm start yet
        P.lam[e] = 0.0;
    }
    if (e < (int64_t)A.M * A.K) {
        P.kappa[e] = 0.0;
        if (A.flo) {
            const double lo = A.flo[e], hi = A.fhi[e];
            A.bd_flo[e] = lo; A.bd_fhi[e] = hi;
            A.bd_flof[e] = float(lo); A.bd_fhif[e] = float(hi);
            D.s[e] = D.ys[e] = 0.f;                        // s = 0 clipped on the first update
            D.sflag[e] = 0;
        }
    }
    if (e < (int64_t)A.M * KMAX) D.Qhi[e] = D.Qlo[e] = __float2bfloat16_rn(0.f);
    if (e < (int64_t)A.M * PRISM_NDIAG) P.diag[e] = 0.0;
    if (e < A.M) {
        const double tau = A.tau ? A.tau[e] : INFINITY;
        if (isnan(tau) || tau < 0) atomicOr(A.err, ERR_CAP);
        if (isfinite(tau)) A.err[2] = 1;
        A.bd_tau[e] = tau;
        A.bd_tauf[e] = float(tau);
        D.rho_idx[e] = A.rho_idx;
        D.active[e] = 1;
        D.iters[e] = D.status[e] = 0;
        D.nu[e] = D.theta[e] = 0.f;
        D.dnu[e] = __int_as_float(0x7f7f7f7f);             // 3.4e38: no margin yet
        P.skip[e] = P.done[e] = 0;
        P.nu[e] = P.theta[e] = 0.0;
        if (A.flo) D.rps[e] = D.rds[e] = 0.f;
    }
    if (e == 0) {
        D.n_active[0] = D.n_active[1] = 0;
        if (D.pcount) D.pcount[0] = D.pcount[1] = 0;
        for (int q = 0; q < A.n_ctr; ++q) D.xq_ctr[q] = 0;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(*D.t0));
    }
}

// The accounts that iterate on (active) begin again: what a first pass of the iterations starts from.
__global__ void k_restart(int M, int S, Dev D, int rho_idx) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < (int64_t)M * S && D.active[e / S]) D.eta_hi[e] = D.eta_lo[e] = __int_as_float(-1);
    if (e < M && D.active[e]) {
        D.rho_idx[e] = rho_idx;
        D.iters[e] = 0;
        D.nu[e] = D.theta[e] = 0.f;
    }
}

// The number of accounts that the polish left for another pass of the iterations.
__global__ void k_unsettled(int M, const int* skip, const int* done, const int* status, int* n) {
    int c = 0;
    for (int a = threadIdx.x; a < M; a += blockDim.x)
        c += !(skip[a] || done[a] == 1 || status[a] == PRISM_NUMERICAL_FAILURE);
    c = __syncthreads_count(c > 0);                        // (threads with any: zero exactly when there is none)
    if (threadIdx.x == 0) *n = c;
}

struct UnpackArgs {
    int M, Npad;
    const int64_t* offsets;
    const int32_t* asset_idx;
    const int* inv_perm;
    const double* W;
    double* out;
    int64_t nnz;
};

__global__ void k_unpack(UnpackArgs A) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.nnz) return;
    int lo = 0, hi = A.M;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (A.offsets[mid] <= e) lo = mid; else hi = mid;
    }
    const int a = lo;
    int i = A.asset_idx ? A.asset_idx[e] : int(e - A.offsets[a]);
    A.out[e] = A.W[(size_t)a * A.Npad + A.inv_perm[i]];
}

// Closed-form feasibility of budget + box + bands (+ the least-turnover test for a
// cap): sum_s max(lo_s, sum_{i in s} l_i) <= 1 <= sum_s min(hi_s, sum_{i in s} u_i).
// Closed-form feasibility of one account (budget, box, bands, and the cap when w0 sums to 1).
// The per-sector sums are taken first in FP32 from the iteration copies, one contiguous chunk
// of positions per thread (float4 loads, one pass); relative to their exact values they are
// off by less than 1e-5. The account is decided there when every comparison clears its
// threshold by 1e-4 relative; otherwise, and whenever a turnover cap is set, the sums are
// taken again in FP64 and decided as before.
__global__ void k_capacity(int S, int N, int Npad, const int* sec_start, const double* LO, const double* UP,
                           const double* W0, const float* LOf, const float* UPf, const float* W0f,
                           const double* band_lo, const double* band_hi, const double* tau, int* status, int* skip,
                           int* active, double* W) {
    const int a = blockIdx.x;
    __shared__ double s_up[SMAX], s_lo[SMAX], s_kept[SMAX], s_forced[SMAX], s_w0[SMAX];
    __shared__ float f_up[SMAX], f_lo[SMAX];
    __shared__ int sec[SMAX + 1];
    __shared__ int decided, rejected;             // rejected: nothing later writes the account's weights
    auto no_weights = [&]() {
        if (rejected)
            for (int p = threadIdx.x; p < Npad; p += blockDim.x) W[(size_t)a * Npad + p] = 0.0;
    };
    if (threadIdx.x == 0) rejected = 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t base = (size_t)a * Npad;
    for (int s = threadIdx.x; s <= S; s += blockDim.x) sec[s] = sec_start[s];
    for (int s = threadIdx.x; s < S; s += blockDim.x) { f_up[s] = 0.f; f_lo[s] = 0.f; }
    __syncthreads();
    if (!isfinite(tau[a])) {
        // FP32 pass: Npad is a multiple of 64, so chunks of whole float4s cover it
        const int nq = Npad / 4, per = (nq + blockDim.x - 1) / blockDim.x;
        const int q0 = threadIdx.x * per, q1 = min(nq, q0 + per);
        int cs = 0;
        float su = 0.f, sl = 0.f;
        auto flush = [&](int s) {
            if (s < S) { atomicAdd(&f_up[s], su); atomicAdd(&f_lo[s], sl); }
            su = 0.f; sl = 0.f;
        };
        if (q0 < q1) {
            const int p0 = 4 * q0;
            while (cs < S && p0 >= sec[cs + 1]) ++cs;
            for (int q = q0; q < q1; ++q) {
                const float4 u4 = reinterpret_cast<const float4*>(UPf + base)[q];
                const float4 l4 = reinterpret_cast<const float4*>(LOf + base)[q];
                const float uu[4] = {u4.x, u4.y, u4.z, u4.w}, ll[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int p = 4 * q + k;
                    if (p >= N) break;
                    while (cs < S && p >= sec[cs + 1]) { flush(cs); ++cs; }
                    su += uu[k]; sl += ll[k];
                }
            }
            flush(cs);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // each comparison is decided only when it clears its threshold by 1e-4 relative
            bool ok = true, sure = true;
            double cap = 0, flo = 0, mag = 0;
            for (int s = 0; s < S; ++s) {
                const double hi = band_hi[a * S + s], lo = band_lo[a * S + s];
                const double u = f_up[s], l = f_lo[s];
                const double tol_u = 1e-4 * (u + fabs(lo)) + 1e-12, tol_l = 1e-4 * (l + fabs(hi)) + 1e-12;
                if (fabs(lo - u) <= tol_u && !(lo == 0.0 && u == 0.0)) sure = false;
                if (fabs(l - hi) <= tol_l && !(l == 0.0 && hi == 0.0)) sure = false;
                if (lo > u + 1e-12 || l > hi + 1e-12) ok = false;
                cap += fmin(hi, u);
                flo += fmax(lo, l);
                mag += fabs(fmin(hi, u)) + fabs(fmax(lo, l));
            }
            if (fabs(cap - 1.0) <= 1e-4 * fmax(mag, 1.0) || fabs(flo - 1.0) <= 1e-4 * fmax(mag, 1.0)) sure = false;
            if (!(cap >= 1.0 - 1e-12 && flo <= 1.0 + 1e-12)) ok = false;
            decided = sure;
            if (sure && !ok) {
                status[a] = PRISM_NO_FEASIBLE_RETURN;
                skip[a] = 1;
                active[a] = 0;
                rejected = 1;
            }
        }
        __syncthreads();
        if (decided) { no_weights(); return; }
    }
    for (int s = warp; s < S; s += nw) {
        double su = 0, sl = 0, sk = 0, sf = 0, sw = 0;
        for (int p = sec[s] + lane; p < sec[s + 1]; p += 32) {
            double u = UP[base + p], l = LO[base + p], w = W0[base + p];
            su += u; sl += l; sk += fmin(w, u); sf += fmax(w - u, 0.0); sw += w;
        }
        su = warp_sum(su); sl = warp_sum(sl); sk = warp_sum(sk); sf = warp_sum(sf); sw = warp_sum(sw);
        if (lane == 0) { s_up[s] = su; s_lo[s] = sl; s_kept[s] = sk; s_forced[s] = sf; s_w0[s] = sw; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double cap = 0, flo = 0, forced = 0, w0s = 0;
        bool ok = true, lo_zero = true;
        for (int s = 0; s < S; ++s) {
            const double hi = band_hi[a * S + s], lo = band_lo[a * S + s];
            if (lo > s_up[s] + 1e-12 || s_lo[s] > hi + 1e-12) ok = false;
            cap += fmin(hi, s_up[s]);
            flo += fmax(lo, s_lo[s]);
            forced += s_forced[s] + fmax(s_kept[s] - hi, 0.0);
            w0s += s_w0[s];
            if (lo > 0 || s_lo[s] > 0) lo_zero = false;
        }
        if (!(cap >= 1.0 - 1e-12 && flo <= 1.0 + 1e-12)) ok = false;
        const double t = tau[a];
        if (ok && isfinite(t) && lo_zero && fabs(w0s - 1.0) < 1e-9 && 2.0 * forced > t * (1.0 + 1e-12)) ok = false;
        if (!ok) {
            status[a] = PRISM_NO_FEASIBLE_RETURN;
            skip[a] = 1;
            active[a] = 0;
            rejected = 1;
        }
    }
    __syncthreads();
    no_weights();
}

// ---------------------------------------------------------------------------
// tax lots (convex piecewise-linear transition cost, the lot-LP's partial minimum) and tilts
//
// One thread per entry with lots builds its row of breakpoints and slopes. The rows used to be built on
// the host, entry by entry, and copied: 25 of the 52 ms of a 200 x 1,924 tax-lot book, and 5 of the
// 18 ms of a 64 x 2,000 book with a benchmark, whose tilt 2 Sigma w_b needs two passes over the factors.
// ---------------------------------------------------------------------------
struct CostArgs {
    int M, N, Npad, K;
    int64_t nnz, n_lots;
    const int64_t* offsets;
    const int32_t* asset_idx;
    const int* inv_perm;
    const double *w0, *lo, *up, *tc;    // ragged
    const int64_t* lot_off;             // nnz + 1, or null
    const double *lot_size, *lot_kappa;
    const double *mu_tilt, *w_bench;    // ragged, or null
    const double *B, *f, *d;            // sorted positions
    double* h;                          // M x K: F B' w_b
    double* tilt;                       // M x Npad, and its FP32 copy
    float* tiltf;
    int tilt_rows;                      // 1: entries with a tilt carry it in a row (row n_lots + e)
    int* pw_idx;                        // M x Npad, -1 beforehand; or null
    double *bp, *sl, *phi_lo;
    float *bpf, *slf;
    int* nbp;
    int* err;                           // [0] flags, [1] rows written
};

__device__ __forceinline__ int account_of(const int64_t* offsets, int M, int64_t e) {
    int lo = 0, hi = M;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (offsets[mid] <= e) lo = mid; else hi = mid;
    }
    return lo;
}

// phi(x) = c (x - w0) + G(max(S*, w0 - x)), G(S) = 2 c S + cheapest-first lot cost of S; lots sorted by kappa
__device__ double lot_phi(double x, double w0, double c, int L, const double* sz, const double* ka) {
    double sstar = 0.0;
    for (int j = 0; j < L; ++j) if (2.0 * c + ka[j] < 0.0) sstar += sz[j];
    const double S = fmax(sstar, w0 - x);
    double g = 2.0 * c * S, rem = S;
    for (int j = 0; j < L && rem > 0; ++j) {
        const double take = (j + 1 < L) ? fmin(rem, sz[j]) : rem;
        g += ka[j] * take;
        rem -= take;
    }
    return c * (x - w0) + g;
}

__global__ void k_costs(CostArgs A) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.nnz) return;
    const int a = A.asset_idx ? account_of(A.offsets, A.M, e) : int(e / A.N);
    const int i = A.asset_idx ? A.asset_idx[e] : int(e - (int64_t)a * A.N);
    if (i < 0 || i >= A.N) return;                          // (flagged by the pack)
    const size_t at = (size_t)a * A.Npad + A.inv_perm[i];
    double t = 0.0;
    if (A.mu_tilt) t = A.mu_tilt[e];
    if (A.w_bench) {
        const double wb = A.w_bench[e];
        if (!isfinite(wb)) { atomicOr(A.err, ERR_BENCH); return; }
        const double* Bi = A.B + (size_t)A.inv_perm[i] * A.K;
        double acc = A.d[A.inv_perm[i]] * wb;
        for (int k = 0; k < A.K; ++k) acc += Bi[k] * A.h[(size_t)a * A.K + k];
        t += 2.0 * acc;
    }
    if (!isfinite(t)) { atomicOr(A.err, ERR_TILT); return; }
    if (A.tilt) { A.tilt[at] = t; A.tiltf[at] = float(t); }
    const double shift = A.tilt_rows ? t : 0.0;
    int64_t l0 = 0, l1 = 0;
    if (A.lot_off) {
        l0 = A.lot_off[e]; l1 = A.lot_off[e + 1];
        if (l0 < 0 || l1 < l0 || l1 > A.n_lots) { atomicOr(A.err, ERR_LOT_OFFSETS); return; }
    }
    if (l1 == l0 && shift == 0.0) return;
    const double w0 = A.w0[e], lo = A.lo[e], up = A.up[e], c = A.tc[e];
    double bp[MAXBP], sl[MAXBP - 1], phi;
    int nb;
    int64_t row;
    if (l1 > l0) {
        row = l0;                                           // unique: its lots are its own
        const int L = int(l1 - l0 > MAXLOT ? MAXLOT + 1 : l1 - l0);
        if (L > MAXLOT) { atomicOr(A.err, ERR_LOT_COUNT); return; }
        if (lo < 0) { atomicOr(A.err, ERR_LOT_LOWER); return; }
        double sz[MAXLOT], ka[MAXLOT], hs = 0;
        for (int q = 0; q < L; ++q) {
            const double s = A.lot_size[l0 + q], k = A.lot_kappa[l0 + q];
            if (!(s >= 0) || !isfinite(k)) { atomicOr(A.err, ERR_LOT_DATA); return; }
            hs += s;
            int j = q;                                      // stable insertion by kappa
            for (; j > 0 && ka[j - 1] > k; --j) { ka[j] = ka[j - 1]; sz[j] = sz[j - 1]; }
            ka[j] = k; sz[j] = s;
        }
        if (fabs(hs - w0) > 1e-9 * fmax(1.0, fabs(w0))) { atomicOr(A.err, ERR_LOT_SUM); return; }
        // kinks in increasing order; slope j is that left of kink j, c right of the last
        int js = 0;
        while (js < L && 2.0 * c + ka[js] < 0.0) ++js;
        const int nk = L - js;
        double kink[MAXLOT];
        double H = 0.0;
        for (int j = 0; j < js; ++j) H += sz[j];
        for (int j = 0; j < nk; ++j) {
            kink[nk - 1 - j] = w0 - H;
            H += sz[js + j];
        }
        auto slope = [&](int q) { return q < nk ? -c - ka[L - 1 - q] : c; };
        phi = lot_phi(lo, w0, c, L, sz, ka);
        nb = 1;
        bp[0] = lo;
        if (up > lo) {
            // the kinks and w0 inside the box, sorted, each once
            bool held = w0 > lo && w0 < up;
            for (int j = 0; j <= nk; ++j) {
                if (held && (j == nk || w0 <= kink[j])) {
                    if (w0 > bp[nb - 1]) bp[nb++] = w0;
                    held = false;
                }
                if (j < nk && kink[j] > lo && kink[j] < up && kink[j] > bp[nb - 1]) bp[nb++] = kink[j];
            }
            bp[nb++] = up;
            for (int j = 0; j + 1 < nb; ++j) {
                const double mid = 0.5 * (bp[j] + bp[j + 1]);
                int q = 0;
                while (q < nk && kink[q] <= mid) ++q;
                sl[j] = slope(q);
            }
        }
    } else {
        // the plain L1 cost as a row: breakpoints l, w0 (inside the box), u
        row = A.n_lots + e;
        phi = c * fabs(lo - w0);
        if (!(up > lo)) {
            nb = 1; bp[0] = lo;
        } else if (w0 > lo && w0 < up) {
            nb = 3; bp[0] = lo; bp[1] = w0; bp[2] = up; sl[0] = -c; sl[1] = c;
        } else {
            nb = 2; bp[0] = lo; bp[1] = up; sl[0] = (w0 <= lo) ? c : -c;
        }
    }
    // a term -t w shifts every slope by -t
    for (int j = 0; j + 1 < nb; ++j) {
        const double s = sl[j] - shift;
        A.sl[row * (MAXBP - 1) + j] = s;
        A.slf[row * (MAXBP - 1) + j] = float(s);
    }
    for (int j = 0; j < nb; ++j) {
        A.bp[row * MAXBP + j] = bp[j];
        A.bpf[row * MAXBP + j] = float(bp[j]);
    }
    A.phi_lo[row] = phi - shift * bp[0];
    A.nbp[row] = nb;
    A.pw_idx[at] = (int)row;
    if (A.err[1] == 0) A.err[1] = 1;
}

// F B' w_b of each account, FP64: a block per account, its warps over the entries, a lane per factor
__global__ void __launch_bounds__(256) k_bench_factors(CostArgs A) {
    const int a = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
    __shared__ double part[8][KMAX];
    double a0 = 0.0, a1 = 0.0;
    for (int64_t e = A.offsets[a] + warp; e < A.offsets[a + 1]; e += NW) {
        const int i = A.asset_idx ? A.asset_idx[e] : int(e - A.offsets[a]);
        if (i < 0 || i >= A.N) continue;
        const double wb = A.w_bench[e];
        const double* Bi = A.B + (size_t)A.inv_perm[i] * A.K;
        if (lane < A.K) a0 += Bi[lane] * wb;
        if (lane + 32 < A.K) a1 += Bi[lane + 32] * wb;
    }
    part[warp][lane] = a0;
    part[warp][lane + 32] = a1;
    __syncthreads();
    for (int k = threadIdx.x; k < A.K; k += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < NW; ++w) s += part[w][k];
        A.h[(size_t)a * A.K + k] = A.f[k] * s;
    }
}

template <typename T>
static bool is_dev(const T* p) {
    if (!p) return false;
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

template <typename T>
static int to_host(const T* src, size_t n, std::vector<T>& dst) {
    dst.resize(n);
    if (!n) return PRISM_OK;
    PRISM_CUDA_TRY(cudaMemcpy(dst.data(), src, n * sizeof(T), cudaMemcpyDefault));
    return PRISM_OK;
}

static double ms_between(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, a, b);
    return ms;
}

// ---------------------------------------------------------------------------
// the account-resident iterations: which books take them, in which launches
// ---------------------------------------------------------------------------
static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, sms);
}

// Time of one iteration of the whole book, us, fitted to both routes' times over 741 books (300 to 10,000
// assets, 10 to 64 factors, 2 to 400 accounts; the L1 cost in BF16 and FP32, and in BF16 lots, tilts, caps,
// factor bounds and ragged accounts). Account-resident: 4.5 for the chain of reductions, 2.5 more when it
// crosses a cluster, and the products with the CTA's rows; times the book's share of the SMs.
// Batched: the latency of the launches (with the iterations that a chunk runs past the last account's)
// and the traffic; lots and tilts are priced by rows, a cap by repeated budget roots. Of the 741
// choices 8 take longer than the other route by 10 to 24% (400 ragged x 3,000 x 16 the most: batched 1.96
// against 1.57 ms of iterations). Lots keep the line that they had: two books of 2 million entries would be
// 2.2 and 2.6 times as fast account-resident.
static double acct_iteration_us(const AcctShape& s, int n, int M, int K, int sms) {
    const int regs = s.threads > 256 ? 128 : 232;
    const int per_sm = std::max(1, std::min((int)(228 * 1024 / (s.smem + 1024)), 65536 / (s.threads * regs)));
    const double waves = std::max(1.0, double(M) * s.cluster / (double(sms) * per_sm));
    return waves * (4.5 + (s.cluster > 1 ? 2.5 : 0.0) + 4e-5 * cdiv(n, s.cluster) * K) * (per_sm > 1 ? 1.3 : 1.0);
}
static double batched_iteration_us(int M, int N, bool bf16, bool lots, bool tilt, bool cap) {
    if (lots || tilt) return 60.0 + (lots ? 9e-6 : 5e-5) * M * N;
    return bf16 && !cap ? 33.0 + 7e-6 * M * N : 40.0 + 3e-5 * M * N;
}

// Whether the options leave the form of the iterations open: one that names a form of the batched
// kernels keeps the book on them, and so does the failure-path test of their tensor-core waits.
static bool open_form(const prism_solve_opts& o) {
    return !(o.fold_products || o.xupdate_form || o.chains || o.g2_sets || !o.fuse_prox || o.ragged_layout == 1) &&
           !std::getenv("PRISM_TEST_STALLED_WAIT_NS");
}

// A ragged book is iterated over all positions, as the batched kernels do (non-members stay pinned at 0): the
// packed layout, whose capacitance is that of an account's own names, is another splitting.
static bool acct_route(const prism_solve_opts& o, bool plain, bool packed, bool fp64, bool bf16, int M, int N, int K, bool pw,
                       bool tilt, bool fac, bool cap, AcctShape& shape) {
    if (packed || !open_form(o)) return false;
    const int bytes = fp64 ? 8 : (bf16 ? 2 : 4);
    shape = acct_shape(N, K, bytes, fac, pw);
    if (shape.E == 0) return false;
    if (plain) return true;                           // (no batched form is the faster for one account)
    return acct_iteration_us(shape, N, M, K, sm_count()) <= batched_iteration_us(M, N, bf16, pw, tilt, cap);
}

// ---------------------------------------------------------------------------
// one batched solve (all accounts share the launch sequence)
// ---------------------------------------------------------------------------
static int solve_core(prism_universe* uh, const prism_batch* b, const prism_solve_opts* o,
                      prism_result* res, bool batched_mode_bf16, bool plain, bool fp64 = false) {
    Universe& U = uh->u;
    SolveCache& SC = cache_of(uh);
    const auto t_call0 = std::chrono::steady_clock::now();
    PRISM_CUDA_TRY(cudaSetDevice(U.device));
    cudaStream_t st = o->cuda_stream ? (cudaStream_t)o->cuda_stream : U.stream;
    const int M = b->n_accounts, N = U.N, Npad = U.Npad, K = U.K, S = U.S;
    // ---- offsets
    std::vector<int64_t> offs;
    int rc = to_host(b->offsets, (size_t)M + 1, offs);
    if (rc) return rc;
    if (offs[0] != 0) { set_error("offsets[0] must be 0"); return PRISM_ERR_ARGUMENT; }
    for (int a = 0; a < M; ++a) {
        if (offs[a + 1] < offs[a]) { set_error("offsets must be nondecreasing"); return PRISM_ERR_ARGUMENT; }
        if (!b->asset_idx && offs[a + 1] - offs[a] != N) {
            set_error("without asset_idx every account must span the universe (N entries)");
            return PRISM_ERR_ARGUMENT;
        }
        if (offs[a + 1] - offs[a] > N) { set_error("account longer than the universe"); return PRISM_ERR_ARGUMENT; }
    }
    const int64_t nnz = offs[M];
    // ---- lots and tilts (see k_costs)
    const bool has_lots = b->lot_offsets != nullptr, has_tilt = b->mu_tilt || b->w_bench;
    int64_t n_lots = 0;
    if (has_lots) PRISM_CUDA_TRY(cudaMemcpy(&n_lots, b->lot_offsets + nnz, sizeof(int64_t), cudaMemcpyDefault));
    if (n_lots < 0) { set_error("lot_offsets must be nondecreasing"); return PRISM_ERR_ARGUMENT; }
    // factor-exposure bounds: validated on the host, any finite one turns the block on
    std::vector<double> flo_h, fhi_h;
    bool has_fac_in = false;
    if (b->factor_lo || b->factor_hi) {
        flo_h.assign((size_t)M * K, -INFINITY);
        fhi_h.assign((size_t)M * K, INFINITY);
        if (b->factor_lo && (rc = to_host(b->factor_lo, (size_t)M * K, flo_h))) return rc;
        if (b->factor_hi && (rc = to_host(b->factor_hi, (size_t)M * K, fhi_h))) return rc;
        for (size_t q = 0; q < flo_h.size(); ++q) {
            if (std::isnan(flo_h[q]) || std::isnan(fhi_h[q]) || flo_h[q] > fhi_h[q]) {
                set_error("factor_lo <= factor_hi required (no NaN)");
                return PRISM_ERR_ARGUMENT;
            }
            has_fac_in |= std::isfinite(flo_h[q]) || std::isfinite(fhi_h[q]);
        }
    }
    // ---- ragged books in the batched modes: dense-masked, or packed (each account's own names)
    bool packed = false;
    if (b->asset_idx && !plain) {
        packed = o->ragged_layout == 2;
    }
    // ---- which iterations: account-resident (acct_admm.cuh) where its accounts fit and it is the faster
    AcctShape shape;
    std::vector<int> order_h;
    auto route = [&](bool cap) {
        return acct_route(*o, plain, packed, fp64, batched_mode_bf16, M, N, K, has_lots, has_tilt, has_fac_in, cap, shape);
    };
    // (whether some cap is finite is known once the device has looked at them, see below; until then only
    // the layout of a tilt depends on the route, and with a tilt the caps do not change it)
    bool acct = route(false);
    // the account-resident kernel takes a tilt as a shift of mu, the batched ones as cost rows
    const bool tilt_rows = has_tilt && !acct;
    const bool has_pw = has_lots || tilt_rows;
    const int64_t n_pw64 = n_lots + (tilt_rows ? nnz : 0);
    if (n_pw64 > INT32_MAX) { set_error("too many tax lots"); return PRISM_ERR_UNSUPPORTED; }
    const int n_pw = (int)n_pw64;
    // ---- workspace layout
    const size_t MN = (size_t)M * Npad;
    int tc_chunk = 0;
    const int nsplit = batched_mode_bf16 ? tc_nsplit(M, N, &tc_chunk, o->g2_sets) : choose_nsplit(M, N);
    const int FMAX = std::min(N, 2048);
    int* dsel = nullptr;               // device copy of SC.hsel (polish batches)
    BlkArgs<double> P64;               // PLAIN_FP64: the FP64 per-account kernel's arguments
    BlkArgs<float> PK;                 // ragged books, packed layout: the FP32 per-account kernel's
    unsigned long long* t0_dev = nullptr;   // device clock at the start of the solve
    char* inbox = nullptr;             // small host inputs (see stage_in)
    auto layout = [&](Arena& A, Dev& D, PolDev& P, BatchDev& BD, void** stage, int** member, int** err,
                      int** pwidx_dev, double** ragged_out) {
        BD.w0 = A.take<double>(MN); BD.lo = A.take<double>(MN); BD.up = A.take<double>(MN); BD.c = A.take<double>(MN);
        BD.w0f = A.take<float>(MN); BD.lof = A.take<float>(MN); BD.upf = A.take<float>(MN); BD.cf = A.take<float>(MN);
        *member = A.take<int>(b->asset_idx ? MN : 0);
        *pwidx_dev = has_pw ? A.take<int>(MN) : nullptr;
        BD.band_lo = A.take<double>((size_t)M * S); BD.band_hi = A.take<double>((size_t)M * S);
        BD.band_lof = A.take<float>((size_t)M * S); BD.band_hif = A.take<float>((size_t)M * S);
        BD.tau = A.take<double>(M); BD.tauf = A.take<float>(M);
        {
            const size_t nf = has_fac_in ? (size_t)M * K : 0;
            BD.flo = A.take<double>(nf); BD.fhi = A.take<double>(nf);
            BD.flof = A.take<float>(nf); BD.fhif = A.take<float>(nf);
            D.s = A.take<float>(nf); D.ys = A.take<float>(nf); D.sflag = A.take<int>(nf);
            D.rps = A.take<float>(has_fac_in ? M : 0); D.rds = A.take<float>(has_fac_in ? M : 0);
            P.wfac = A.take<int>(nf);
        }
        P.kappa = A.take<double>((size_t)M * K);
        D.z = A.take<float>(MN); D.y = A.take<float>(MN); D.v = A.take<float>(MN);
        D.X = A.take<float>(MN);
        D.Xhi = A.take<__nv_bfloat16>(MN); D.Xlo = A.take<__nv_bfloat16>(MN);
        D.Ppart = A.take<float>((size_t)nsplit * M * KMAX);
        D.Q = A.take<float>((size_t)M * K);
        D.Qhi = A.take<__nv_bfloat16>((size_t)M * KMAX); D.Qlo = A.take<__nv_bfloat16>((size_t)M * KMAX);
        D.rho_idx = A.take<int>(M); D.iters = A.take<int>(M); D.active = A.take<int>(M); D.status = A.take<int>(M);
        D.nu = A.take<float>(M); D.dnu = A.take<float>(M); D.eta_hi = A.take<float>((size_t)M * S); D.eta_lo = A.take<float>((size_t)M * S);
        D.theta = A.take<float>(M); D.rp = A.take<float>(M); D.rd = A.take<float>(M); D.n_active = A.take<int>(2);
        D.stats = A.take<unsigned long long>(8);
        // partials of the fused pass (tensor-core mode)
        const int nt = cdiv(N, 128);
        D.SOp = A.take<float>((size_t)U.nseg * M);
        D.Rt = A.take<float>((size_t)5 * nt * M); D.Cm = A.take<unsigned>((size_t)U.nq * M);
        D.lo_u = A.take<float>(M); D.c_u = A.take<float>(M);
        D.crec = A.take<float>(MN * 8);
        D.Pxp = A.take<float>(batched_mode_bf16 ? (size_t)xp_sets_for(N) * M * KMAX : 0);
        D.needP = A.take<int>(M);
        D.pcount = A.take<unsigned long long>(2);
        D.xq_ctr = A.take<unsigned>(2 * SolveCache::MAXCH);
        P.st = A.take<int8_t>(MN); P.wband = A.take<int>((size_t)M * S); P.wcap = A.take<int>(M);
        P.done = A.take<int>(M); P.Flist = A.take<int>((size_t)M * FMAX); P.NZlist = A.take<int>((size_t)M * FMAX);
        P.Fsig = A.take<double>((size_t)M * FMAX);
        P.Y = A.take<double>((size_t)M * FMAX * (PMAXROWS + 1));
        P.Fdinv = A.take<double>((size_t)M * FMAX);
        P.fh64 = A.take<double>((size_t)M * KMAX); P.fh32 = A.take<float>((size_t)M * K);
        P.quad = A.take<double>(M); P.fhmax = A.take<double>(M);
        P.ndep = A.take<int>(M); P.pending = A.take<int>(1);
        P.W = A.take<double>(MN); P.nu = A.take<double>(M); P.lam = A.take<double>((size_t)M * S);
        P.theta = A.take<double>(M); P.diag = A.take<double>((size_t)M * PRISM_NDIAG);
        int* skip = A.take<int>(M);
        P.skip = skip;
        dsel = A.take<int>(M);
        *err = A.take<int>(4);
        // staging for host inputs / outputs (ragged FP64 x 4, offsets, asset_idx, out)
        stage[0] = A.take<double>((size_t)nnz); stage[1] = A.take<double>((size_t)nnz);
        stage[2] = A.take<double>((size_t)nnz); stage[3] = A.take<double>((size_t)nnz);
        stage[4] = A.take<int64_t>((size_t)M + 1);
        stage[5] = b->asset_idx ? (void*)A.take<int32_t>((size_t)nnz) : nullptr;
        *ragged_out = A.take<double>((size_t)nnz);
        BD.pw_bp = A.take<double>((size_t)std::max(n_pw, 1) * MAXBP);
        BD.pw_sl = A.take<double>((size_t)std::max(n_pw, 1) * (MAXBP - 1));
        BD.pw_bpf = A.take<float>((size_t)std::max(n_pw, 1) * MAXBP);
        BD.pw_slf = A.take<float>((size_t)std::max(n_pw, 1) * (MAXBP - 1));
        BD.pw_nbp = A.take<int>((size_t)std::max(n_pw, 1));
        stage[6] = A.take<double>((size_t)std::max(n_pw, 1));   // phi_lo
        stage[7] = A.take<int64_t>(has_lots ? (size_t)nnz + 1 : 0);
        stage[8] = A.take<double>((size_t)n_lots); stage[9] = A.take<double>((size_t)n_lots);
        stage[10] = A.take<double>(b->mu_tilt ? (size_t)nnz : 0); stage[11] = A.take<double>(b->w_bench ? (size_t)nnz : 0);
        stage[12] = A.take<double>(b->w_bench ? (size_t)M * K : 0);
        const size_t nt64 = (has_tilt && !tilt_rows) ? MN : 0;
        P.tilt = A.take<double>(nt64); P.tiltf = A.take<float>(nt64);
        // FP64 iteration state of PLAIN_FP64 (z, y, X/v per entry; penalty and cap multiplier)
        const size_t n64 = fp64 ? MN : 0;
        P64.z = A.take<double>(n64); P64.y = A.take<double>(n64); P64.X = A.take<double>(n64);
        P64.rho_state = A.take<double>(fp64 ? M : 0); P64.theta_state = A.take<double>(fp64 ? M : 0);
        P64.s_state = A.take<double>((fp64 && has_fac_in) ? (size_t)M * K : 0);
        P64.ys_state = A.take<double>((fp64 && has_fac_in) ? (size_t)M * K : 0);
        P64.queue = A.take<int>(4);
        // packed layout of a ragged book: position lists, sector ranges, processing order, FP32
        // state and input copies for accounts too large for shared memory
        const size_t np = packed ? (size_t)nnz : 0;
        PK.plist = A.take<int>(packed ? (size_t)nnz : 0); PK.psec = A.take<int>(packed ? (size_t)M * (S + 1) : 0);
        PK.order = A.take<int>(M); PK.queue = A.take<int>(4);
        t0_dev = A.take<unsigned long long>(1);
        inbox = A.take<char>(SolveCache::BOX);
        PK.z = A.take<float>(np); PK.y = A.take<float>(np); PK.X = A.take<float>(np);
        PK.w0p = A.take<float>(np); PK.lop = A.take<float>(np); PK.upp = A.take<float>(np); PK.cp = A.take<float>(np);
        PK.pwp = A.take<int>(np);
        PK.rho_state = A.take<float>(packed ? M : 0); PK.theta_state = A.take<float>(packed ? M : 0);
        PK.s_state = A.take<float>((packed && has_fac_in) ? (size_t)M * K : 0);
        PK.ys_state = A.take<float>((packed && has_fac_in) ? (size_t)M * K : 0);
    };
    Dev D;
    std::memset((void*)&D, 0, sizeof(Dev));   // padding bytes take part in the graph-reuse test
    PolDev P;
    BatchDev BD;
    void* stage[13];
    int *member, *err, *pwidx;
    double* ragged_out;
    {
        Arena probe;
        probe.base = nullptr; probe.cap = SIZE_MAX;
        layout(probe, D, P, BD, stage, &member, &err, &pwidx, &ragged_out);
        size_t need = probe.used + 4096;
        if (SC.arena_bytes < need) {
            if (SC.arena) { cudaFree(SC.arena); SC.arena = nullptr; SC.arena_bytes = 0; }
            if (SC.have_graph) { cudaGraphExecDestroy(SC.gexec); SC.have_graph = false; }
            if (SC.hact) { cudaFreeHost(SC.hact); cudaFreeHost(SC.hsel); SC.hact = SC.hsel = nullptr; SC.hcap = 0; }
            if (cudaMalloc(&SC.arena, need) != cudaSuccess) {
                cudaGetLastError();
                set_error("device workspace allocation failed");
                return PRISM_ERR_ALLOCATION;
            }
            SC.arena_bytes = need;
        }
        if (!SC.pinned) {
            if (cudaMallocHost(&SC.pinned, 64) != cudaSuccess) { set_error("pinned alloc failed"); return PRISM_ERR_ALLOCATION; }
            if (cudaMallocHost(&SC.box, 2 * SolveCache::BOX) != cudaSuccess) { cudaGetLastError(); SC.box = nullptr; }
            for (auto& e : SC.ev) cudaEventCreate(&e);
            if (cudaStreamCreateWithFlags(&SC.pst, cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&SC.ev_pol, cudaEventDisableTiming) != cudaSuccess) {
                cudaGetLastError();
                SC.pst = nullptr;                        // the polish waits for the iterations
            }
            SC.chains_ok = cudaEventCreateWithFlags(&SC.ev_fork, cudaEventDisableTiming) == cudaSuccess;
            for (int c = 0; c + 1 < SolveCache::MAXCH && SC.chains_ok; ++c)
                SC.chains_ok = cudaStreamCreateWithFlags(&SC.chst[c], cudaStreamNonBlocking) == cudaSuccess &&
                               cudaEventCreateWithFlags(&SC.ev_join[c], cudaEventDisableTiming) == cudaSuccess;
            if (!SC.chains_ok) cudaGetLastError();        // one chain only
        }
        if (SC.hcap < M) {
            if (SC.have_graph) { cudaGraphExecDestroy(SC.gexec); SC.have_graph = false; }
            if (SC.hact) { cudaFreeHost(SC.hact); cudaFreeHost(SC.hsel); SC.hact = SC.hsel = nullptr; SC.hcap = 0; }
            if (cudaMallocHost(&SC.hact, (size_t)M * 4) != cudaSuccess ||
                cudaMallocHost(&SC.hsel, (size_t)M * 4) != cudaSuccess) {
                cudaGetLastError();
                set_error("pinned alloc failed");
                return PRISM_ERR_ALLOCATION;
            }
            SC.hcap = M;
        }
        Arena A;
        A.base = SC.arena; A.cap = SC.arena_bytes;
        std::memset((void*)&D, 0, sizeof(Dev));
        P = PolDev(); BD = BatchDev(); P64 = BlkArgs<double>(); PK = BlkArgs<float>();
        layout(A, D, P, BD, stage, &member, &err, &pwidx, &ragged_out);
        if (A.alloc_fail) { set_error("workspace layout overflow"); return PRISM_ERR_ALLOCATION; }
    }
    SC.prof.reset();
    SC.prof.on = o->profile != 0;
    cudaEventRecord(SC.ev[0], st);
    // ---- stage inputs on the device
    // (small host arrays are gathered in pinned memory and go over in one copy per flush: each copy of
    // its own from pageable memory takes 5 us and more of the host's time)
    size_t box_used = 0, box_sent = 0;
    auto stage_in = [&](const void* src, void* dst, size_t bytes) -> const void* {
        if (is_dev(src)) return src;
        const size_t room = (bytes + 255) / 256 * 256;
        if (SC.box && room <= SolveCache::BOX / 4 && box_used + room <= SolveCache::BOX) {
            std::memcpy(SC.box + box_used, src, bytes);
            void* at = inbox + box_used;
            box_used += room;
            return at;
        }
        cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
        return dst;
    };
    auto flush = [&]() {
        if (box_used > box_sent)
            cudaMemcpyAsync(inbox + box_sent, SC.box + box_sent, box_used - box_sent, cudaMemcpyHostToDevice, st);
        box_sent = box_used;
    };
    PackArgs PA;
    PA.M = M; PA.N = N; PA.Npad = Npad; PA.nnz = nnz;
    PA.w0 = (const double*)stage_in(b->w0, stage[0], nnz * 8);
    PA.lo = (const double*)stage_in(b->lower, stage[1], nnz * 8);
    PA.up = (const double*)stage_in(b->upper, stage[2], nnz * 8);
    PA.tc = (const double*)stage_in(b->tc, stage[3], nnz * 8);
    PA.offsets = (const int64_t*)stage_in(offs.data(), stage[4], (M + 1) * sizeof(int64_t));
    PA.asset_idx = b->asset_idx ? (const int32_t*)stage_in(b->asset_idx, stage[5], nnz * 4) : nullptr;
    PA.inv_perm = U.d_inv_perm;
    PA.W0 = BD.w0; PA.LO = BD.lo; PA.UP = BD.up; PA.C = BD.c;
    PA.W0f = BD.w0f; PA.LOf = BD.lof; PA.UPf = BD.upf; PA.Cf = BD.cf;
    PA.member = member; PA.err = err;
    if (b->asset_idx) {
        // ragged accounts: every position the pack does not write is a non-member (zeros)
        cudaMemsetAsync(BD.w0, 0, MN * 8, st); cudaMemsetAsync(BD.lo, 0, MN * 8, st);
        cudaMemsetAsync(BD.up, 0, MN * 8, st); cudaMemsetAsync(BD.c, 0, MN * 8, st);
        cudaMemsetAsync(BD.w0f, 0, MN * 4, st); cudaMemsetAsync(BD.lof, 0, MN * 4, st);
        cudaMemsetAsync(BD.upf, 0, MN * 4, st); cudaMemsetAsync(BD.cf, 0, MN * 4, st);
        cudaMemsetAsync(member, 0, MN * 4, st);
    } else if (Npad > N) {
        // every account spans the universe, so the pack writes every position below N: only
        // the padding columns N .. Npad-1 are cleared
        auto pad = [&](void* p, size_t es) {
            cudaMemset2DAsync(static_cast<char*>(p) + (size_t)N * es, (size_t)Npad * es, 0, (size_t)(Npad - N) * es,
                              (size_t)M, st);
        };
        pad(BD.w0, 8); pad(BD.lo, 8); pad(BD.up, 8); pad(BD.c, 8);
        pad(BD.w0f, 4); pad(BD.lof, 4); pad(BD.upf, 4); pad(BD.cf, 4);
    }
    cudaMemsetAsync(err, 0, 16, st);
    flush();
    if (nnz > 0) SC.prof.run(PRISM_K_PACK, 1, st, [&] { k_pack<<<(unsigned)cdiv64(nnz, 256), 256, 0, st>>>(PA); });
    // bands, caps, factor bounds and the accounts' state
    const int j0 = (int)std::lround(RHO_PER_DECADE * std::log10(std::max(o->rho0, 1e-12) / RHO_MIN));
    const int rho_idx0 = std::max(0, std::min(NRHO - 1, j0));
    {
        SetupArgs SA = {};
        SA.M = M; SA.S = S; SA.K = K;
        SA.rho_idx = rho_idx0;
        SA.n_ctr = 2 * SolveCache::MAXCH;
        SA.band_lo = (const double*)stage_in(b->band_lo, BD.band_lo, (size_t)M * S * 8);
        SA.band_hi = (const double*)stage_in(b->band_hi, BD.band_hi, (size_t)M * S * 8);
        SA.tau = b->turnover_cap ? (const double*)stage_in(b->turnover_cap, BD.tau, (size_t)M * 8) : nullptr;
        SA.bd_lo = BD.band_lo; SA.bd_hi = BD.band_hi; SA.bd_tau = BD.tau;
        SA.bd_lof = BD.band_lof; SA.bd_hif = BD.band_hif; SA.bd_tauf = BD.tauf;
        if (has_fac_in) {
            SA.flo = (const double*)stage_in(flo_h.data(), BD.flo, flo_h.size() * 8);
            SA.fhi = (const double*)stage_in(fhi_h.data(), BD.fhi, fhi_h.size() * 8);
            SA.bd_flo = BD.flo; SA.bd_fhi = BD.fhi; SA.bd_flof = BD.flof; SA.bd_fhif = BD.fhif;
            BD.has_fac = true;
        }
        SA.D = D; SA.P = P; SA.err = err;
        SA.D.t0 = t0_dev;
        const int64_t n = (int64_t)M * std::max(std::max(S, K), KMAX);
        flush();
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { k_setup<<<(unsigned)cdiv64(n, 256), 256, 0, st>>>(SA); });
    }
    // lots and tilts
    if (has_lots || has_tilt) {
        CostArgs CA = {};
        CA.M = M; CA.N = N; CA.Npad = Npad; CA.K = K; CA.nnz = nnz; CA.n_lots = n_lots;
        CA.offsets = PA.offsets; CA.asset_idx = PA.asset_idx; CA.inv_perm = U.d_inv_perm;
        CA.w0 = PA.w0; CA.lo = PA.lo; CA.up = PA.up; CA.tc = PA.tc;
        if (has_lots) {
            CA.lot_off = (const int64_t*)stage_in(b->lot_offsets, stage[7], (nnz + 1) * sizeof(int64_t));
            CA.lot_size = (const double*)stage_in(b->lot_size, stage[8], n_lots * 8);
            CA.lot_kappa = (const double*)stage_in(b->lot_kappa, stage[9], n_lots * 8);
        }
        if (b->mu_tilt) CA.mu_tilt = (const double*)stage_in(b->mu_tilt, stage[10], nnz * 8);
        if (b->w_bench) CA.w_bench = (const double*)stage_in(b->w_bench, stage[11], nnz * 8);
        CA.B = U.d_B64; CA.f = U.d_f64; CA.d = U.d_d64; CA.h = (double*)stage[12];
        CA.tilt_rows = tilt_rows;
        if (has_tilt && !tilt_rows) {
            CA.tilt = P.tilt; CA.tiltf = P.tiltf;
            cudaMemsetAsync(P.tilt, 0, MN * 8, st);
            cudaMemsetAsync(P.tiltf, 0, MN * 4, st);
        }
        CA.pw_idx = pwidx; CA.bp = BD.pw_bp; CA.sl = BD.pw_sl; CA.phi_lo = (double*)stage[6];
        CA.bpf = BD.pw_bpf; CA.slf = BD.pw_slf; CA.nbp = BD.pw_nbp; CA.err = err;
        if (pwidx) cudaMemsetAsync(pwidx, 0xff, MN * 4, st);
        flush();
        SC.prof.run(PRISM_K_PACK, b->w_bench ? 2 : 1, st, [&] {
            if (b->w_bench) k_bench_factors<<<M, 256, 0, st>>>(CA);
            if (nnz > 0) k_costs<<<(unsigned)cdiv64(nnz, 128), 128, 0, st>>>(CA);
        });
    }
    {
        int* flags = SC.pinned + 4;
        PRISM_CUDA_TRY(cudaMemcpyAsync(flags, err, 12, cudaMemcpyDeviceToHost, st));
        PRISM_CUDA_TRY(cudaStreamSynchronize(st));
        const int herr = flags[0];
        BD.has_cap = flags[2] != 0;
        acct = route(BD.has_cap);
        if (!has_lots && !flags[1]) pwidx = nullptr;      // every tilt is zero: plain costs throughout
        struct { int bit, code; const char* text; } lot_errors[] = {
            {ERR_LOT_OFFSETS, PRISM_ERR_ARGUMENT, "lot_offsets must be nondecreasing"},
            {ERR_LOT_COUNT, PRISM_ERR_UNSUPPORTED, "more than 4 lots on one entry"},
            {ERR_LOT_LOWER, PRISM_ERR_ARGUMENT, "lots need lower >= 0"},
            {ERR_LOT_DATA, PRISM_ERR_ARGUMENT, "bad lot data"},
            {ERR_LOT_SUM, PRISM_ERR_ARGUMENT, "lot sizes of an entry must sum to its w0"},
            {ERR_BENCH, PRISM_ERR_ARGUMENT, "w_bench must be finite"},
            {ERR_TILT, PRISM_ERR_ARGUMENT, "mu_tilt must be finite"},
            {ERR_BAND, PRISM_ERR_ARGUMENT, "band_lo <= band_hi required (no NaN)"},
            {ERR_CAP, PRISM_ERR_ARGUMENT, "turnover_cap must be >= 0 or +inf"}};
        for (auto& q : lot_errors)
            if (herr & q.bit) { set_error(q.text); return q.code; }
        if (herr) {
            std::string m = "invalid batch input:";
            if (herr & ERR_INDEX) m += " asset index out of range;";
            if (herr & ERR_NONFINITE) m += " non-finite w0/lower/upper/tc;";
            if (herr & ERR_BOUNDS) m += " lower > upper;";
            if (herr & ERR_COST) m += " negative tc;";
            if (herr & ERR_DUP) m += " duplicate asset within an account;";
            set_error(m);
            return PRISM_ERR_ARGUMENT;
        }
    }
    // ---- device views
    D.M = M; D.N = N; D.Npad = Npad; D.K = K; D.S = S;
    D.B32 = U.d_B32; D.d32 = U.d_d32; D.mu32 = U.d_mu32; D.sec_start = U.d_sec_start; D.sector = U.d_sector;
    D.B16 = U.d_B16; D.Bt16 = U.d_Bt16; D.B16p = U.d_B16p; D.Bt16p = U.d_Bt16p;
    D.err = D.n_active + 1;
    if (!std::getenv("PRISM_DEBUG_STATS")) D.stats = nullptr;   // counters only when asked for
    if (const char* sw = std::getenv("PRISM_TEST_STALLED_WAIT_NS")) {
        // failure-path test: a bounded tensor-core wait on a barrier nothing completes (at most
        // 0.1 s, so that the test ends quickly and a stray setting cannot stall a real run long)
        const long long ns = std::atoll(sw);
        D.stall_ns = (unsigned long long)std::max(0LL, std::min(ns, 100000000LL));
    }
    if (!o->profile) D.pcount = nullptr;
    D.bf16 = batched_mode_bf16;
    D.Cinv = batched_mode_bf16 ? U.d_Cinv16 : U.d_Cinv32;
    D.w0 = BD.w0f; D.lo = BD.lof; D.up = BD.upf; D.c = BD.cf;
    D.pw_idx = pwidx; D.pw_bp = BD.pw_bpf; D.pw_sl = BD.pw_slf; D.pw_nbp = BD.pw_nbp;
    D.band_lo = BD.band_lof; D.band_hi = BD.band_hif; D.tau = BD.tauf;
    if (BD.has_fac) {
        // the factor-exposure block: its own capacitance inverses and the Gram matrices
        D.Cinv = batched_mode_bf16 ? U.d_CinvF16 : U.d_CinvF32;
        D.G = batched_mode_bf16 ? U.d_G16 : U.d_G32;
        D.flo = BD.flof; D.fhi = BD.fhif;
    } else {
        D.s = nullptr; D.ys = nullptr; D.sflag = nullptr; D.rps = nullptr; D.rds = nullptr;
    }
    D.stream_prox = (!acct && pwidx == nullptr && !BD.has_cap) ? 1 : 0;
    D.t0 = t0_dev;
    // the streaming pass runs inside the tensor-core x-update when the roots kernel can hold
    // the account's candidate masks
    D.fused = (D.stream_prox && batched_mode_bf16 && U.nq <= XP_NQMAX && o->fuse_prox) ? 1 : 0;
    D.nq = U.nq; D.nseg = U.nseg; D.nt = cdiv(N, 128); D.qseg = U.d_qseg; D.sseg = U.d_sseg;
    D.xp_sets = xp_sets_for(N);
    if (!D.fused || o->xupdate_form != 0) D.xq_ctr = nullptr;   // one CTA per tile
    int* const needP_buf = D.needP;            // set for the fused loop only (null: every account)
    D.needP = nullptr;
    D.nsplit = nsplit;
    D.g2_sets = batched_mode_bf16 ? o->g2_sets : 0;
    D.pstride = batched_mode_bf16 ? KMAX : K;
    D.alpha = (float)o->alpha; D.eps_admm = (float)o->eps_admm; D.min_iter = o->min_iter; D.max_iter = o->max_iter;
    D.adapt_every = o->adapt_every > 0 ? o->adapt_every : 25;
    P.M = M; P.N = N; P.Npad = Npad; P.K = K; P.S = S;
    P.B64 = U.d_B64; P.f64 = U.d_f64; P.d64 = U.d_d64; P.mu64 = U.d_mu64; P.sec_start = U.d_sec_start; P.sector = U.d_sector;
    P.B32 = U.d_B32; P.B32p = U.d_B32p; P.Bn1 = U.d_Bn1; P.Bn1f = U.d_Bn1f; P.mu32 = U.d_mu32;
    P.w0f = BD.w0f; P.lof = BD.lof; P.upf = BD.upf; P.cf = BD.cf;
    P.w0 = BD.w0; P.lo = BD.lo; P.up = BD.up; P.c = BD.c;
    if (!has_tilt || tilt_rows) { P.tilt = nullptr; P.tiltf = nullptr; }
    P.pw_idx = pwidx; P.pw_bp = BD.pw_bp; P.pw_sl = BD.pw_sl; P.pw_phi_lo = (const double*)stage[6]; P.pw_nbp = BD.pw_nbp;
    P.band_lo = BD.band_lo; P.band_hi = BD.band_hi; P.tau = BD.tau;
    if (BD.has_fac) { P.flo = BD.flo; P.fhi = BD.fhi; P.sflag = D.sflag; }
    else P.wfac = nullptr;
    P.z = D.z; P.nu_f = D.nu; P.eta_hi_f = D.eta_hi; P.eta_lo_f = D.eta_lo; P.theta_f = D.theta;
    P.FMAX = FMAX;
    P.status = D.status;
    P.tol_dual = 1e-11; P.tol_primal = 1e-12;
    P.dmin = U.dmin;
    if (fp64) {
        P64.M = M; P64.N = N; P64.Npad = Npad; P64.K = K; P64.S = S;
        P64.B = U.d_B64; P64.f = U.d_f64; P64.d = U.d_d64; P64.mu = U.d_mu64;
        P64.sec_start = U.d_sec_start; P64.sector = U.d_sector;
        P64.w0 = BD.w0; P64.lo = BD.lo; P64.up = BD.up; P64.c = BD.c;
        P64.pw_idx = pwidx; P64.pw_bp = BD.pw_bp; P64.pw_sl = BD.pw_sl; P64.pw_nbp = BD.pw_nbp;
        P64.band_lo = BD.band_lo; P64.band_hi = BD.band_hi; P64.tau = BD.tau; P64.skip = P.skip;
        if (BD.has_fac) { P64.flo = BD.flo; P64.fhi = BD.fhi; P64.sflag = D.sflag; }
        P64.zf = D.z; P64.nu_f = D.nu; P64.eta_hi_f = D.eta_hi; P64.eta_lo_f = D.eta_lo; P64.theta_f = D.theta;
        P64.iters = D.iters; P64.active = D.active; P64.status = D.status;
        P64.alpha = o->alpha; P64.eps = o->eps_admm; P64.rho0 = o->rho0;
        P64.max_iter = o->max_iter; P64.min_iter = o->min_iter; P64.adapt_every = D.adapt_every;
    }
    if (packed) {
        PK.M = M; PK.N = N; PK.Npad = Npad; PK.K = K; PK.S = S;
        PK.B = U.d_B32; PK.Bp = U.d_B32p; PK.f = U.d_f32; PK.d = U.d_d32; PK.mu = U.d_mu32;
        PK.sec_start = U.d_sec_start; PK.sector = U.d_sector;
        PK.w0 = BD.w0f; PK.lo = BD.lof; PK.up = BD.upf; PK.c = BD.cf;
        PK.pw_idx = pwidx; PK.pw_bp = BD.pw_bpf; PK.pw_sl = BD.pw_slf; PK.pw_nbp = BD.pw_nbp;
        PK.band_lo = BD.band_lof; PK.band_hi = BD.band_hif; PK.tau = BD.tauf; PK.skip = P.skip;
        if (BD.has_fac) { PK.flo = BD.flof; PK.fhi = BD.fhif; PK.sflag = D.sflag; }
        PK.poff = PA.offsets;
        PK.zf = D.z; PK.nu_f = D.nu; PK.eta_hi_f = D.eta_hi; PK.eta_lo_f = D.eta_lo; PK.theta_f = D.theta;
        PK.iters = D.iters; PK.active = D.active; PK.status = D.status;
        PK.alpha = o->alpha; PK.eps = o->eps_admm; PK.rho0 = o->rho0;
        PK.max_iter = o->max_iter; PK.min_iter = o->min_iter; PK.adapt_every = D.adapt_every;
        // accounts largest first (the persistent blocks take them in this order); accounts of at
        // most stage_cap names keep their entries in shared memory
        int64_t nmax = 0;
        order_h.resize(M);
        for (int a = 0; a < M; ++a) { order_h[a] = a; nmax = std::max(nmax, offs[a + 1] - offs[a]); }
        std::stable_sort(order_h.begin(), order_h.end(),
                         [&](int x, int y) { return offs[x + 1] - offs[x] > offs[y + 1] - offs[y]; });
        BlkArgs<float> probe = PK;
        probe.stage_cap = 0;
        const size_t fixed = blk_smem_bytes(probe), per = 7 * sizeof(float) + 2 * sizeof(int);
        const size_t room = 227 * 1024 - 1024 > fixed ? 227 * 1024 - 1024 - fixed : 0;
        PK.stage_cap = (int)std::min<int64_t>(nmax, (int64_t)(room / per));
        PRISM_CUDA_TRY(cudaMemcpyAsync(PK.order, order_h.data(), (size_t)M * 4, cudaMemcpyHostToDevice, st));
    }
    // ---- control init (see k_setup)
    if (!acct) cudaMemsetAsync(D.v, 0, MN * 4, st);
    if (D.stats) cudaMemsetAsync(D.stats, 0, 32, st);
    SC.prof.run(PRISM_K_OTHER, acct ? 1 : 2, st, [&] {
        k_capacity<<<M, 256, 0, st>>>(S, N, Npad, U.d_sec_start, BD.lo, BD.up, BD.w0, BD.lof, BD.upf, BD.w0f,
                                      BD.band_lo, BD.band_hi, BD.tau, D.status, P.skip, D.active, P.W);
        if (!acct) launch_init_state(D, st);
    });
    if (D.fused) {
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_uniform(D, (float*)D.lo_u, (float*)D.c_u, st); });
        // the fused kernel's variant: per-account l and c throughout, or per-entry where they differ
        std::vector<float> lu(M), cu(M);
        PRISM_CUDA_TRY(cudaMemcpyAsync(lu.data(), D.lo_u, M * 4, cudaMemcpyDeviceToHost, st));
        PRISM_CUDA_TRY(cudaMemcpyAsync(cu.data(), D.c_u, M * 4, cudaMemcpyDeviceToHost, st));
        PRISM_CUDA_TRY(cudaStreamSynchronize(st));
        D.uniform = 1;
        for (int a = 0; a < M; ++a)
            if (std::isnan(lu[a]) || std::isnan(cu[a])) D.uniform = 0;
    }
    cudaEventRecord(SC.ev[1], st);
    // ---- ADMM iterations
    const int check_every = std::max(1, o->check_every);
    // Chains: the accounts are cut into up to MAXCH ranges that iterate independently on their
    // own streams, so that one range's latency-bound kernels (the roots, the small products)
    // run beside another range's streaming x-update. Every cut is a multiple of 128 (a product
    // tile never straddles two ranges); a range holds at least 128 accounts.
    int nch = 1;
    // automatic: as many chains as fit for the one-CTA-per-tile x-update; one for the persistent
    // form, whose CTAs take every SM (measured: several chains then lose more than they overlap)
    if (D.fused && SC.chains_ok && !D.xq_ctr) nch = std::min(SolveCache::MAXCH, std::max(1, M / 128));
    if (D.fused && SC.chains_ok && o->chains > 0) nch = std::min(std::min(SolveCache::MAXCH, std::max(1, M / 128)), o->chains);
    auto run_chunk = [&](int n) {
        if (nch > 1 && !SC.prof.on) {
            Dev DC[SolveCache::MAXCH];
            cudaStream_t cs[SolveCache::MAXCH];
            for (int c = 0; c < nch; ++c) {
                DC[c] = D;
                DC[c].m0 = ((M * c / nch) + 64) / 128 * 128;
                DC[c].m1 = (c + 1 == nch) ? M : ((M * (c + 1) / nch) + 64) / 128 * 128;
                if (D.xq_ctr) { DC[c].xq_ctr = D.xq_ctr + 2 * c; DC[c].xq_share = nch; }   // own tile counter
                cs[c] = c == 0 ? st : SC.chst[c - 1];
            }
            cudaEventRecord(SC.ev_fork, st);
            for (int c = 1; c < nch; ++c) cudaStreamWaitEvent(cs[c], SC.ev_fork, 0);
            for (int it = 0; it < n; ++it) {
                SC.prof.run(PRISM_K_GEMM_P, nch, st, [&] { for (int c = 0; c < nch; ++c) launch_tc_gemm_P(DC[c], cs[c], true); });
                SC.prof.run(PRISM_K_SOLVE_K, nch, st, [&] { for (int c = 0; c < nch; ++c) launch_small_solve(DC[c], cs[c], true); });
                SC.prof.run(PRISM_K_XPROX, nch, st, [&] { for (int c = 0; c < nch; ++c) launch_tc_xprox(DC[c], cs[c], true); });
                SC.prof.run(PRISM_K_ROOTS, nch, st, [&] { for (int c = 0; c < nch; ++c) launch_prox_roots(DC[c], cs[c], true); });
            }
            for (int c = 1; c < nch; ++c) {
                cudaEventRecord(SC.ev_join[c - 1], cs[c]);
                cudaStreamWaitEvent(st, SC.ev_join[c - 1], 0);
            }
            SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_count_active(D, st); });
            cudaMemcpyAsync(SC.pinned, D.n_active, 8, cudaMemcpyDeviceToHost, st);
            cudaMemcpyAsync(SC.hact, D.active, (size_t)M * 4, cudaMemcpyDeviceToHost, st);
            return;
        }
        for (int it = 0; it < n; ++it) {
            if (D.fused) {
                // the four kernels of an iteration overlap their prologues with the kernel
                // before (programmatic dependent launch; see pdl_wait)
                const bool pdl = !SC.prof.on;
                SC.prof.run(PRISM_K_GEMM_P, 1, st, [&] { launch_tc_gemm_P(D, st, pdl); });
                SC.prof.run(PRISM_K_SOLVE_K, 1, st, [&] { launch_small_solve(D, st, pdl); });
                SC.prof.run(PRISM_K_XPROX, 1, st, [&] { launch_tc_xprox(D, st, pdl); });
                SC.prof.run(PRISM_K_ROOTS, 1, st, [&] { launch_prox_roots(D, st, pdl); });
                continue;
            }
            SC.prof.run(PRISM_K_GEMM_P, 1, st, [&] { if (D.bf16) launch_tc_gemm_P(D, st); else launch_gemm_P(D, st); });
            SC.prof.run(PRISM_K_SOLVE_K, 1, st, [&] { launch_small_solve(D, st); });
            SC.prof.run(PRISM_K_GEMM_X, 1, st, [&] { if (D.bf16) launch_tc_gemm_x(D, st); else launch_gemm_x(D, st); });
            SC.prof.run(PRISM_K_PROX, 1, st, [&] { launch_prox(D, st); });
        }
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_count_active(D, st); });
        cudaMemcpyAsync(SC.pinned, D.n_active, 8, cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(SC.hact, D.active, (size_t)M * 4, cudaMemcpyDeviceToHost, st);
    };
    int64_t chunk_launches[PRISM_NKCLASS] = {};
    // Accounts that stop iterating are polished on their own stream while the others iterate:
    // after each chunk, those that stopped since the last check form a batch (hsel[a] = its
    // number) and are classified and polished beside the next chunk. Only the accounts' own
    // rows are touched, which the iterations no longer read or write.
    const int rounds = std::max(1, o->polish_rounds);
    int pol_gen = 0;
    std::vector<char> was_active(M, 1);
    auto polish_batch = [&](int gen, cudaStream_t s) {
        PolDev PB2 = P;
        PB2.sel = dsel;
        PB2.gen = gen;
        SC.prof.run(PRISM_K_OTHER, 1, s, [&] { launch_classify(PB2, s); });
        SC.prof.run(PRISM_K_POLISH, 1, s, [&] { launch_polish(PB2, rounds, s); });
    };
    AcctArgs<float> AF;
    AcctArgs<double> AD;
    // the few accounts that a batched book sends back to the iterations go on account-resident
    const AcctShape again = (!acct && !fp64 && !packed && open_form(*o))
                                ? acct_shape(N, K, batched_mode_bf16 ? 2 : 4, BD.has_fac, has_pw) : AcctShape();
    if (acct || again.E) {
        auto fill = [&](auto& A) {
            A.M = M; A.N = N; A.Npad = Npad; A.K = K; A.S = S;
            A.sec_start = U.d_sec_start;
            A.pw_idx = pwidx; A.pw_nbp = BD.pw_nbp;
            A.nu = D.nu; A.eta_hi = D.eta_hi; A.eta_lo = D.eta_lo; A.theta = D.theta; A.zf = D.z;
            A.rho_idx = D.rho_idx; A.iters = D.iters; A.active = D.active; A.status = D.status;
            if (BD.has_fac) A.sflag = D.sflag;
            A.t0 = t0_dev;
            A.alpha = o->alpha; A.eps = o->eps_admm;
            A.max_iter = o->max_iter; A.min_iter = o->min_iter; A.adapt_every = D.adapt_every;
        };
        fill(AF);
        fill(AD);
        if (batched_mode_bf16) AF.B16p = U.d_B16p; else AF.B32p = U.d_B32p;
        AF.f = U.d_f32; AF.d = U.d_d32; AF.mu = U.d_mu32;
        AF.Cinv = D.Cinv; AF.G = D.G;                 // (of the split-off factor block when there is one)
        AF.w0 = BD.w0f; AF.lo = BD.lof; AF.up = BD.upf; AF.c = BD.cf;
        AF.pw_bp = BD.pw_bpf; AF.pw_sl = BD.pw_slf;
        AF.band_lo = BD.band_lof; AF.band_hi = BD.band_hif;
        AF.z = D.z; AF.y = D.y;
        AF.tilt = P.tiltf; AD.tilt = P.tilt;
        if (BD.has_cap) AF.tau = BD.tauf;
        if (BD.has_fac) { AF.flo = BD.flof; AF.fhi = BD.fhif; AF.s = D.s; AF.ys = D.ys; }
        AD.B64 = U.d_B64; AD.f = U.d_f64; AD.d = U.d_d64; AD.mu = U.d_mu64;
        AD.w0 = BD.w0; AD.lo = BD.lo; AD.up = BD.up; AD.c = BD.c;
        AD.pw_bp = BD.pw_bp; AD.pw_sl = BD.pw_sl;
        AD.band_lo = BD.band_lo; AD.band_hi = BD.band_hi;
        AD.z = P64.z; AD.y = P64.y;
        AD.rho_state = P64.rho_state; AD.theta_state = P64.theta_state; AD.rho0 = o->rho0;
        if (BD.has_cap) AD.tau = BD.tau;
        if (BD.has_fac) { AD.flo = BD.flo; AD.fhi = BD.fhi; AD.s = P64.s_state; AD.ys = P64.ys_state; }
    }
    auto set_budget = [&]() {                         // (from t0, which the device took a little after the call began)
        if (o->time_budget_s > 0)                     // (FP64 iterations run through: checked between accounts)
            AF.budget_ns = (unsigned long long)(std::min(o->time_budget_s, 1e9) * 1e9) + 1;
    };
    // With lots or a cap the polish can lose its way from a start a few places off, and one such account
    // costs it eight rounds on hundreds of free entries: 8-11 ms of a 200 x 1,924 book against 0.6 when every
    // account first keeps its places for 12 iterations (ADMM 1.6 -> 2.2 ms). Books without them gain
    // nothing (100 x 5,000 x 48: 1.3 -> 2.3 against 0.67 -> 0.47). The few accounts that the polish leaves
    // all the same begin again and take the batched kernels' passes, without that wait: which accounts
    // certify is theirs (3 of 50,000 certify from there and not from the places that they kept).
    const int settle = (acct && (has_lots || BD.has_cap)) ? 12 : 0;
    // the accounts' iterations in one launch (refused: the call fails before the polish is queued)
    cudaError_t acct_err = cudaSuccess;
    auto run_acct = [&](int resume, double eps, int max_iter, int wait) {
        set_budget();
        AF.settle = AD.settle = wait;
        AF.resume = AD.resume = resume;
        AF.eps = (float)eps; AD.eps = eps;
        AF.max_iter = AD.max_iter = max_iter;
        SC.prof.run(PRISM_K_BLOCK, 1, st, [&] {
            acct_err = fp64 ? launch_acct_admm(AD, shape, M, st) : launch_acct_admm(AF, shape, M, st);
        });
    };
    // A batched book with only a few accounts left to iterate goes on account-resident once their CTAs
    // fit on the SMs side by side: the chain of the batched kernels costs 21-25 us an iteration however
    // few accounts are left and runs on to the end of its chunk. One to three accounts of 500 x 10,000 x
    // 64 that the polish sends back: 2.3-3.1 ms on the chain, 0.9-1.6 so (of calls of 6.0 ms without).
    auto few_fit = [&](int n) { return again.E && n > 0 && n * again.cluster <= sm_count(); };
    auto run_few = [&](const int* act, double eps, int max_iter) {
        order_h.clear();
        for (int a = 0; a < M; ++a) if (act[a]) order_h.push_back(a);
        cudaMemcpyAsync(PK.order, order_h.data(), order_h.size() * 4, cudaMemcpyHostToDevice, st);
        AF.resume = 1;
        AF.eps = (float)eps;
        AF.max_iter = max_iter;
        AF.order = PK.order;
        set_budget();
        SC.prof.run(PRISM_K_BLOCK, 1, st, [&] { acct_err = launch_acct_admm(AF, again, (int)order_h.size(), st); });
    };
    auto admm_loop = [&](int iter_budget, bool overlap) -> int {
        int done_iters = 0;
        if (D.needP) {
            // the folded iteration keeps no X of the entries it pins and leaves P, Q only for the
            // accounts that iterate on: on entry every active account gets X from its z, y, and
            // its first P and Q from the product kernels
            SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_refresh_X(D, st); });
            cudaMemsetAsync(D.needP, 0x01, (size_t)M * 4, st);
        }
        overlap = overlap && SC.pst && !SC.prof.on && o->polish_overlap > 0;
        bool use_graph = o->use_graph != 0 && !SC.prof.on;
        if (use_graph) {
            bool same = SC.have_graph && SC.g_iters == check_every && std::memcmp(&SC.gdev, &D, sizeof(Dev)) == 0;
            if (!same) {
                if (SC.have_graph) { cudaGraphExecDestroy(SC.gexec); SC.have_graph = false; }
                cudaGraph_t g;
                if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { cudaGetLastError(); use_graph = false; }
                else {
                    int64_t before[PRISM_NKCLASS];
                    std::memcpy(before, SC.prof.launches, sizeof(before));
                    run_chunk(check_every);
                    for (int q = 0; q < PRISM_NKCLASS; ++q) {
                        chunk_launches[q] = SC.prof.launches[q] - before[q];
                        SC.prof.launches[q] = before[q];
                    }
                    if (cudaStreamEndCapture(st, &g) != cudaSuccess ||
                        cudaGraphInstantiate(&SC.gexec, g, 0) != cudaSuccess) {
                        cudaGetLastError();
                        use_graph = false;
                    } else {
                        SC.have_graph = true;
                        SC.gdev = D;
                        SC.g_iters = check_every;
                        std::memcpy(SC.g_launches, chunk_launches, sizeof(chunk_launches));
                    }
                    cudaGraphDestroy(g);
                }
            }
        }
        while (done_iters < iter_budget) {
            if (use_graph) {
                cudaGraphLaunch(SC.gexec, st);
                for (int q = 0; q < PRISM_NKCLASS; ++q) SC.prof.launches[q] += SC.g_launches[q];
            } else {
                run_chunk(check_every);
            }
            done_iters += check_every;
            if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
            if (SC.pinned[1] != 0) return -2;      // a bounded tensor-core wait expired
            if (overlap && SC.pinned[0] < o->polish_overlap * M) {
                int nnew = 0;
                for (int a = 0; a < M; ++a)
                    if (was_active[a] && !SC.hact[a]) { was_active[a] = 0; SC.hsel[a] = pol_gen + 1; ++nnew; }
                if (nnew) {
                    ++pol_gen;
                    cudaMemcpyAsync(dsel, SC.hsel, (size_t)M * 4, cudaMemcpyHostToDevice, SC.pst);
                    polish_batch(pol_gen, SC.pst);
                }
            }
            if (SC.pinned[0] == 0) break;
            if (!overlap && few_fit(SC.pinned[0])) { run_few(SC.hact, D.eps_admm, D.max_iter); break; }
            if (o->time_budget_s > 0) {
                double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_call0).count();
                if (el > o->time_budget_s) break;
            }
        }
        return done_iters;
    };
    // the first iterations run the staged prox: the streaming form needs the budget multiplier
    // to have settled (its moves set the streaming form's margin) to keep its candidate lists short
    const bool blockwise = acct || fp64 || packed;   // every iteration inside a per-account kernel
    const int cold = (D.stream_prox && !blockwise) ? std::min(std::max(0, o->stream_after), o->max_iter) : 0;
    if (acct) {
        run_acct(0, o->eps_admm, o->max_iter, settle);
    } else if (fp64) {
        // PLAIN_FP64: every iteration of the account in one FP64 launch (block_admm.cu)
        P64.resume = 0;
        SC.prof.run(PRISM_K_BLOCK, 1, st, [&] { launch_block_admm(P64, blk_grid(P64), st); });
    }
    if (packed) {
        // ragged book, packed layout: the position lists, then one persistent FP32 launch
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] {
            launch_member_lists(M, Npad, S, member, U.d_sec_start, PA.offsets, PK.plist, PK.psec, st);
        });
        PK.resume = 0;
        SC.prof.run(PRISM_K_BLOCK, 1, st, [&] { launch_block_admm(PK, blk_grid(PK), st); });
    }
    if ((fp64 || packed) && !acct && D.stats) {
        // diagnostics: ns per phase summed over accounts, iterations, projection evaluations
        unsigned long long h[8] = {};
        BlkArgs<float> DP = PK;
        BlkArgs<double> D64 = P64;
        cudaMemsetAsync(D.stats, 0, 64, st);
        if (packed) { DP.dbg = D.stats; launch_block_admm(DP, blk_grid(DP), st); }
        else { D64.dbg = D.stats; launch_block_admm(D64, blk_grid(D64), st); }
        cudaMemcpyAsync(h, D.stats, 64, cudaMemcpyDeviceToHost, st);
        cudaStreamSynchronize(st);
        std::fprintf(stderr, "prism block stats: iterations %llu, ns: X+B'X %llu, solve %llu, x-update %llu, roots %llu, "
                     "z/y %llu, factor %llu; evaluations per iteration %.1f\n", h[6], h[0], h[1], h[2], h[3], h[4], h[5],
                     h[6] ? double(h[7]) / h[6] : 0.0);
    }
    for (int it = 0; it < cold; ++it) {
        SC.prof.run(PRISM_K_GEMM_P, 1, st, [&] { if (D.bf16) launch_tc_gemm_P(D, st); else launch_gemm_P(D, st); });
        SC.prof.run(PRISM_K_SOLVE_K, 1, st, [&] { launch_small_solve(D, st); });
        SC.prof.run(PRISM_K_GEMM_X, 1, st, [&] { if (D.bf16) launch_tc_gemm_x(D, st); else launch_gemm_x(D, st); });
        SC.prof.run(PRISM_K_PROX, 1, st, [&] { launch_prox(D, st, true); });
    }
    std::memset(SC.hsel, 0, (size_t)M * 4);
    if (D.fused && o->fold_products) { D.needP = needP_buf; D.fold = 1; }
    int total_iters = blockwise ? 0 : admm_loop(o->max_iter + check_every - cold, true);
    if (total_iters >= 0) total_iters += cold;
    if (acct_err != cudaSuccess) { set_error(std::string("ADMM launch failed: ") + cudaGetErrorString(acct_err)); return PRISM_ERR_CUDA; }
    if (total_iters == -2) { set_error("tensor-core pipeline wait timed out (error flags " + std::to_string(SC.pinned[1]) + ")"); return PRISM_ERR_CUDA; }
    if (total_iters < 0) { set_error(std::string("ADMM loop failed: ") + cudaGetErrorString(cudaGetLastError())); return PRISM_ERR_CUDA; }
    SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_mark_timeout(D, st); });   // accounts still iterating
    cudaEventRecord(SC.ev[2], st);
    if (std::getenv("PRISM_DEBUG_STATS")) {
        unsigned long long h[4] = {0, 0, 0, 0};
        cudaMemcpyAsync(h, D.stats, 32, cudaMemcpyDeviceToHost, st);
        cudaStreamSynchronize(st);
        std::fprintf(stderr, "prism stats: ADMM iterations %d, prox account-calls %llu, sector-edge evals/call %.2f, "
                     "budget evals/call %.2f, sectors from global memory/call %.2f\n", total_iters, h[0],
                     h[0] ? double(h[1]) / h[0] : 0.0, h[0] ? double(h[2]) / h[0] : 0.0,
                     h[0] ? double(h[3]) / h[0] : 0.0);
    }
    // ---- polish, with up to two returns to the iterations at a tighter target (after a new start of
    // accounts that had been waiting for their places)
    // polish rounds until no account needs another (checked after each round)
    int n_rounds_run = 0, n_retried = 0;
    // all active-set rounds of every account in one launch; each block stops when settled (one
    // launch per round measured slower: each launch waits for its slowest block)
    auto polish_rounds = [&](bool last, int accounts) -> int {
        ++n_rounds_run;
        P.retry = !last;
        SC.prof.run(PRISM_K_POLISH, 1, st, [&] { launch_polish(P, rounds, st, accounts); });
        return 0;
    };
    if (pol_gen > 0) {
        // the batches polished beside the iterations, then every account not in one of them
        // (those that stopped in the last chunk, or were still iterating at the cap)
        cudaEventRecord(SC.ev_pol, SC.pst);
        cudaStreamWaitEvent(st, SC.ev_pol, 0);
        cudaMemcpyAsync(dsel, SC.hsel, (size_t)M * 4, cudaMemcpyHostToDevice, st);
        ++n_rounds_run;
        polish_batch(0, st);
    } else {
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_classify(P, st); });
        if (polish_rounds(false, M) < 0) { set_error("polish failed"); return PRISM_ERR_CUDA; }
    }
    for (int retry = settle ? -1 : 0; retry < 2; ++retry) {   // (-1: they begin again, see settle)
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { k_unsettled<<<1, 1024, 0, st>>>(M, P.skip, P.done, D.status, err + 3); });
        PRISM_CUDA_TRY(cudaMemcpyAsync(SC.pinned + 8, err + 3, 4, cudaMemcpyDeviceToHost, st));
        PRISM_CUDA_TRY(cudaStreamSynchronize(st));
        if (SC.pinned[8] == 0) break;
        std::vector<int> done(M), skip(M), status(M);
        cudaMemcpyAsync(done.data(), P.done, M * 4, cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(skip.data(), P.skip, M * 4, cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(status.data(), D.status, M * 4, cudaMemcpyDeviceToHost, st);
        PRISM_CUDA_TRY(cudaStreamSynchronize(st));
        std::vector<int> act(M, 0);
        int n_retry = 0;
        for (int a = 0; a < M; ++a) {
            if (skip[a] || done[a] == 1 || status[a] == PRISM_NUMERICAL_FAILURE) continue;
            act[a] = 1;
            done[a] = 0;
            status[a] = 0;
            ++n_retry;
        }
        if (!n_retry) break;
        n_retried += n_retry;
        if (o->time_budget_s > 0 &&
            std::chrono::duration<double>(std::chrono::steady_clock::now() - t_call0).count() > o->time_budget_s) break;
        // iterate again, to a tighter target, only the accounts the polish could not settle
        PRISM_CUDA_TRY(cudaMemcpyAsync(D.active, act.data(), M * 4, cudaMemcpyHostToDevice, st));
        PRISM_CUDA_TRY(cudaMemcpyAsync(D.status, status.data(), M * 4, cudaMemcpyHostToDevice, st));
        PRISM_CUDA_TRY(cudaMemcpyAsync(P.done, done.data(), M * 4, cudaMemcpyHostToDevice, st));
        PRISM_CUDA_TRY(cudaStreamSynchronize(st));
        int more = 0;
        const int sent_back = n_retry;
        if (retry < 0) {
            SC.prof.run(PRISM_K_OTHER, 1, st, [&] { k_restart<<<(unsigned)cdiv64((int64_t)M * S, 256), 256, 0, st>>>(M, S, D, rho_idx0); });
            run_acct(0, o->eps_admm, o->max_iter, 0);
        } else if (acct) {
            run_acct(1, o->eps_admm * (retry == 0 ? 0.1 : 0.01), o->max_iter * (retry + 2), 0);
        } else if (few_fit(n_retry)) {
            run_few(act.data(), o->eps_admm * (retry == 0 ? 0.1 : 0.01), o->max_iter * (retry + 2));
        } else if (fp64) {
            // continue the FP64 iterations of the accounts sent back, to a tighter target
            BlkArgs<double> R = P64;
            R.resume = 1;
            R.eps = P64.eps * (retry == 0 ? 0.1 : 0.01);
            R.max_iter = P64.max_iter * (retry + 2);
            SC.prof.run(PRISM_K_BLOCK, 1, st, [&] { launch_block_admm(R, blk_grid(R), st); });
        } else if (packed) {
            BlkArgs<float> R = PK;
            R.resume = 1;
            R.eps = PK.eps * (retry == 0 ? 0.1 : 0.01);
            R.max_iter = PK.max_iter * (retry + 2);
            SC.prof.run(PRISM_K_BLOCK, 1, st, [&] { launch_block_admm(R, blk_grid(R), st); });
        } else {
            Dev saved = D;
            D.eps_admm = saved.eps_admm * (retry == 0 ? 0.1f : 0.01f);
            D.max_iter = saved.max_iter * (retry + 2);
            more = admm_loop(D.max_iter, false);
            D = saved;
        }
        if (acct_err != cudaSuccess) { set_error(std::string("ADMM launch failed: ") + cudaGetErrorString(acct_err)); return PRISM_ERR_CUDA; }
        if (more == -2) { set_error("tensor-core pipeline wait timed out"); return PRISM_ERR_CUDA; }
        if (more < 0) { set_error("ADMM retry failed"); return PRISM_ERR_CUDA; }
        total_iters += more;
        SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_classify(P, st); });
        if (polish_rounds(retry == 1, sent_back) < 0) { set_error("polish failed"); return PRISM_ERR_CUDA; }
    }
    if (std::getenv("PRISM_DEBUG_STATS"))
        std::fprintf(stderr, "prism stats: polish rounds %d, accounts sent back to the iterations %d\n", n_rounds_run,
                     n_retried);
    SC.prof.run(PRISM_K_OTHER, 2, st, [&] { launch_fallback(P, st); });
    cudaEventRecord(SC.ev[3], st);
    SC.prof.run(PRISM_K_OTHER, 1, st, [&] { launch_finish_status(P, o->eps_kkt, st); });
    cudaEventRecord(SC.ev[4], st);
    if (o->keep_for_backward) {
        if (int rc2 = make_backward_state(uh, P, D.status, PA.offsets, PA.asset_idx, nnz, st, res->state)) return rc2;
    }
    // ---- unpack
    UnpackArgs UA;
    UA.M = M; UA.Npad = Npad; UA.offsets = PA.offsets; UA.asset_idx = PA.asset_idx; UA.inv_perm = U.d_inv_perm;
    UA.W = P.W; UA.nnz = nnz;
    const bool w_dev = is_dev(res->w);
    UA.out = w_dev ? res->w : ragged_out;
    if (nnz > 0) SC.prof.run(PRISM_K_UNPACK, 1, st, [&] { k_unpack<<<(unsigned)cdiv64(nnz, 256), 256, 0, st>>>(UA); });
    // (small outputs to host memory come back through the box, and are handed out once all are there)
    struct Out { void* dst; const char* at; size_t bytes; } outs[8];
    int n_out = 0;
    size_t out_used = 0;
    auto out = [&](void* dst, const void* src, size_t bytes) {
        if (!dst) return;
        const size_t room = (bytes + 255) / 256 * 256;
        if (SC.box && bytes && room <= SolveCache::BOX / 4 && out_used + room <= SolveCache::BOX && !is_dev(dst)) {
            char* at = SC.box + SolveCache::BOX + out_used;
            out_used += room;
            cudaMemcpyAsync(at, src, bytes, cudaMemcpyDeviceToHost, st);
            outs[n_out++] = {dst, at, bytes};
            return;
        }
        cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, st);
    };
    if (!w_dev) out(res->w, ragged_out, nnz * 8);
    out(res->status, D.status, M * 4);
    out(res->iters, D.iters, M * 4);
    out(res->nu, P.nu, M * 8);
    out(res->lambda_band, P.lam, (size_t)M * S * 8);
    out(res->theta, P.theta, M * 8);
    out(res->diag, P.diag, (size_t)M * PRISM_NDIAG * 8);
    out(res->kappa, P.kappa, (size_t)M * K * 8);
    cudaEventRecord(SC.ev[5], st);
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { set_error(std::string("solve failed: ") + cudaGetErrorString(e)); return PRISM_ERR_CUDA; }
    for (int q = 0; q < n_out; ++q) std::memcpy(outs[q].dst, outs[q].at, outs[q].bytes);
    e = cudaGetLastError();
    if (e != cudaSuccess) { set_error(std::string("solve failed: ") + cudaGetErrorString(e)); return PRISM_ERR_CUDA; }
    res->t_phase_ms[0] = ms_between(SC.ev[0], SC.ev[1]);
    res->t_phase_ms[1] = ms_between(SC.ev[1], SC.ev[2]);
    res->t_phase_ms[2] = ms_between(SC.ev[2], SC.ev[3]);
    res->t_phase_ms[3] = ms_between(SC.ev[3], SC.ev[4]);
    res->t_device_ms = ms_between(SC.ev[0], SC.ev[5]);
    res->device_bytes = (int64_t)(SC.arena_bytes + U.bytes);
    int64_t nl = 0;
    for (int q = 0; q < PRISM_NKCLASS; ++q) {
        res->kernel_launches[q] = SC.prof.launches[q];
        res->kernel_ms[q] = 0.0;
        nl += SC.prof.launches[q];
    }
    for (auto& mk : SC.prof.marks) res->kernel_ms[mk.cls] += ms_between(mk.a, mk.b);
    res->stream_entries = res->stream_candidates = 0;
    if (D.pcount) {
        unsigned long long pc[2] = {0, 0};
        cudaMemcpy(pc, D.pcount, 16, cudaMemcpyDeviceToHost);
        res->stream_candidates = (int64_t)pc[0];
        res->stream_entries = (int64_t)pc[1];
    }
    res->n_launches = nl;
    res->t_call_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_call0).count();
    (void)plain;
    return PRISM_OK;
}

}  // namespace prism

extern "C" void prism_default_opts(prism_solve_opts* o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->eps_kkt = 1e-6;
    o->eps_admm = 5e-4;
    o->rho0 = 3.0;
    o->alpha = 1.5;
    o->time_budget_s = 0.0;
    o->max_iter = 4000;
    o->check_every = 20;
    o->min_iter = 20;
    o->polish_rounds = 8;
    o->precision = PRISM_BATCHED_BF16;
    o->use_graph = 1;
    o->fuse_prox = 1;
    o->stream_after = 6;
    o->adapt_every = 25;
    o->chains = 0;
    o->polish_overlap = 0.0;
    o->keep_for_backward = 0;
    o->cuda_stream = nullptr;
}

extern "C" int prism_solve_batch(prism_universe* uh, const prism_batch* b, const prism_solve_opts* opts,
                                 prism_result* res) {
    using namespace prism;
    if (!uh || !b || !res) { set_error("NULL argument"); return PRISM_ERR_ARGUMENT; }
    prism_solve_opts o;
    if (opts) o = *opts; else prism_default_opts(&o);
    if (b->n_accounts < 1) { set_error("n_accounts must be >= 1"); return PRISM_ERR_ARGUMENT; }
    if (!b->offsets || !b->w0 || !b->lower || !b->upper || !b->tc || !b->band_lo || !b->band_hi) {
        set_error("required batch array is NULL");
        return PRISM_ERR_ARGUMENT;
    }
    if (!res->w || !res->status) { set_error("result w and status are required"); return PRISM_ERR_ARGUMENT; }
    if (b->lot_offsets && (!b->lot_size || !b->lot_kappa)) { set_error("lot arrays incomplete"); return PRISM_ERR_ARGUMENT; }
    if (!(o.eps_kkt > 0) || !(o.eps_admm > 0) || !(o.rho0 > 0) || !(o.alpha > 0 && o.alpha < 2) ||
        o.max_iter < 1 || o.check_every < 1 || o.g2_sets < 0 || o.g2_sets > 64 || o.ragged_layout < 0 ||
        o.ragged_layout > 2 || o.fold_products < 0 || o.fold_products > 1 || o.adapt_every < 0 ||
        o.xupdate_form < 0 || o.xupdate_form > 1) {
        set_error("invalid options");
        return PRISM_ERR_ARGUMENT;
    }
    if (o.keep_for_backward && !res->state) { set_error("keep_for_backward needs res->state"); return PRISM_ERR_ARGUMENT; }
    if (o.keep_for_backward && (o.precision == PRISM_PLAIN_FP32 || o.precision == PRISM_PLAIN_FP64)) {
        set_error("keep_for_backward is available in the batched modes");
        return PRISM_ERR_UNSUPPORTED;
    }
    if (o.keep_for_backward && (b->w_bench || b->factor_lo || b->factor_hi)) {
        set_error("keep_for_backward does not take a benchmark or factor-exposure bounds");
        return PRISM_ERR_UNSUPPORTED;
    }
    if (o.keep_for_backward) *res->state = nullptr;
    const auto t0 = std::chrono::steady_clock::now();
    if (o.precision == PRISM_BATCHED_FP32) return solve_core(uh, b, &o, res, false, false);
    if (o.precision == PRISM_BATCHED_BF16) {
        if (!tc_available()) {
            set_error("BATCHED_BF16 needs the tcgen05 product kernels, which this build does not provide");
            return PRISM_ERR_UNSUPPORTED;
        }
        return solve_core(uh, b, &o, res, true, false);
    }
    if (o.precision != PRISM_PLAIN_FP32 && o.precision != PRISM_PLAIN_FP64) {
        set_error("unknown precision mode");
        return PRISM_ERR_ARGUMENT;
    }
    const bool fp64 = o.precision == PRISM_PLAIN_FP64;
    // PLAIN_FP32 / PLAIN_FP64: one account per launch sequence (the single-account form)
    std::vector<int64_t> offs;
    if (int rc = to_host(b->offsets, (size_t)b->n_accounts + 1, offs)) return rc;
    const int S = uh->u.S;
    double tdev = 0, tph[4] = {0, 0, 0, 0}, kms[PRISM_NKCLASS] = {};
    int64_t dbytes = 0, nlaunch = 0, kl[PRISM_NKCLASS] = {};
    for (int a = 0; a < b->n_accounts; ++a) {
        int64_t sub_off[2] = {0, offs[a + 1] - offs[a]};
        prism_batch sb = *b;
        sb.n_accounts = 1;
        sb.offsets = sub_off;
        const int64_t e0 = offs[a];
        sb.asset_idx = b->asset_idx ? b->asset_idx + e0 : nullptr;
        sb.w0 = b->w0 + e0; sb.lower = b->lower + e0; sb.upper = b->upper + e0; sb.tc = b->tc + e0;
        sb.band_lo = b->band_lo + (size_t)a * S; sb.band_hi = b->band_hi + (size_t)a * S;
        sb.turnover_cap = b->turnover_cap ? b->turnover_cap + a : nullptr;
        sb.mu_tilt = b->mu_tilt ? b->mu_tilt + e0 : nullptr;
        sb.w_bench = b->w_bench ? b->w_bench + e0 : nullptr;
        sb.factor_lo = b->factor_lo ? b->factor_lo + (size_t)a * uh->u.K : nullptr;
        sb.factor_hi = b->factor_hi ? b->factor_hi + (size_t)a * uh->u.K : nullptr;
        std::vector<int64_t> lot_sub;
        if (b->lot_offsets) {
            std::vector<int64_t> lo_all;
            if (int rc = to_host(b->lot_offsets + e0, (size_t)(sub_off[1] + 1), lo_all)) return rc;
            lot_sub.resize(lo_all.size());
            for (size_t q = 0; q < lo_all.size(); ++q) lot_sub[q] = lo_all[q] - lo_all[0];
            sb.lot_offsets = lot_sub.data();
            sb.lot_size = b->lot_size + lo_all[0];
            sb.lot_kappa = b->lot_kappa + lo_all[0];
        }
        prism_result r1 = *res;
        r1.w = res->w + e0;
        r1.status = res->status + a;
        r1.iters = res->iters ? res->iters + a : nullptr;
        r1.nu = res->nu ? res->nu + a : nullptr;
        r1.lambda_band = res->lambda_band ? res->lambda_band + (size_t)a * S : nullptr;
        r1.theta = res->theta ? res->theta + a : nullptr;
        r1.diag = res->diag ? res->diag + (size_t)a * PRISM_NDIAG : nullptr;
        r1.kappa = res->kappa ? res->kappa + (size_t)a * uh->u.K : nullptr;
        int rc = solve_core(uh, &sb, &o, &r1, false, true, fp64);
        if (rc != PRISM_OK) return rc;
        tdev += r1.t_device_ms;
        for (int q = 0; q < 4; ++q) tph[q] += r1.t_phase_ms[q];
        nlaunch += r1.n_launches;
        for (int q = 0; q < PRISM_NKCLASS; ++q) { kms[q] += r1.kernel_ms[q]; kl[q] += r1.kernel_launches[q]; }
        dbytes = std::max(dbytes, r1.device_bytes);
    }
    res->t_device_ms = tdev;
    for (int q = 0; q < 4; ++q) res->t_phase_ms[q] = tph[q];
    res->device_bytes = dbytes;
    res->n_launches = nlaunch;
    for (int q = 0; q < PRISM_NKCLASS; ++q) { res->kernel_ms[q] = kms[q]; res->kernel_launches[q] = kl[q]; }
    res->stream_entries = res->stream_candidates = 0;
    res->t_call_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return PRISM_OK;
}


