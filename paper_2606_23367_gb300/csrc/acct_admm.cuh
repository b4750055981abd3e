// acct_admm.cuh -- the account-resident ADMM: every iteration of an account in one launch. (One
// translation unit for each type of the rows of B: acct_bf16.cu, acct_fp32.cu, acct_fp64.cu.)
//
// The same splitting as the batched kernels (admm.cu; Eq. 1, Sec. 4.2) with penalty rho and
// relaxation alpha, Delta = diag(2 d + rho):
//   X  = Delta^{-1} (mu + rho z - y),  Q = C^{-1} B'X,  x = X - Delta^{-1} B Q,
//   v  = alpha x + (1 - alpha) z + y / rho,  z+ = projection of v,  y+ = rho (v - z+).
//
// What bounds it: for one account an iteration is two products with its n x K rows of B and a few
// scalar roots, that is, a chain of block-wide reductions; launched as four batched kernels the
// chain costs 21-34 us whatever its size. Here the rows of B stay in shared memory and the entries
// in registers for the whole solve, so that an iteration touches no global memory: its products
// are bound by the shared-memory reads and the FP32 issue of n K multiply-adds each, its roots by
// barriers. A thread reads its entries' rows in 16-byte chunks: B Q needs no reduction at all, and B'X
// one transposing warp reduction of 32 sums. A row takes an odd number of chunks, so that eight
// rows hit different banks. (mma.sync for the two products, the vector split into two BF16 columns,
// measured slower, 7.8 against 6.2 us an iteration at 2,000 x 32: the iteration is a chain of short
// phases, six of the eight columns are idle, and its fragments crowd the registers.)
// A thread's entries are consecutive and the positions sorted by sector, so that the sums of all
// sectors are a segmented scan over the lanes and a few additions; warp 0 alone takes the steps of
// the roots.
// Measured (ADMM phase of a solve, before and after): 37 accounts x 777 x 17 1.31 -> 0.26 ms, 64 x 2,000 x
// 32 1.24 -> 0.24, 200 x 1,924 x 48 with lots and a cap 8.0 -> 1.5, one account of 100 x 10 0.94 -> 0.09, in
// FP64 2.8 -> 0.39.
// Accounts too large for one CTA's shared memory are split over a cluster of up to eight CTAs,
// which add their partial sums by stores into each other's shared memory; every CTA then holds the
// same sums, added in the same order, and takes the same decisions.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "acct_admm.h"
#include "common.cuh"

namespace prism {
namespace cg = cooperative_groups;

constexpr int ACCT_WARPS = ACCT_THREADS / 32;
constexpr int ROOT_IT = 80;               // evaluations per safeguarded root
constexpr int PAIR_IT = 12;               // Newton steps on (nu, theta) before the nested search
constexpr int PWROW = 2 * MAXBP + 1;      // a cost row in shared memory: b_0, then (s_j, b_j+1); odd, so
                                          // that the rows of a warp hit different banks

template <typename T> struct AcctTol;
// ROOT: a budget sum accepted as 1; CAP: a turnover accepted as tau (relative); WIDTH: relative
// width at which a bracket is closed. The FP32 values are those of the batched kernels.
template <> struct AcctTol<float> { static constexpr float ROOT = 1e-6f, CAP = 1e-5f, WIDTH = 4e-7f; };
template <> struct AcctTol<double> { static constexpr double ROOT = 1e-13, CAP = 1e-12, WIDTH = 1e-15; };

// a sum and the count of its entries on a linear piece
template <typename T> struct alignas(2 * sizeof(T)) SumCount { T f; int n; };

template <typename T>
struct AcctShared {
    SumCount<T> seg[ACCT_WARPS + SMAX];   // per segment (warp w, sector s): at w + s, which is different
                                          // for every segment
    SumCount<T> turn[ACCT_WARPS];         // turnover and signed count per warp
    SumCount<T> xseg[2][ACCT_CLUSTER][SMAX];   // sector sums per CTA of the cluster
    SumCount<T> xturn[2][ACCT_CLUSTER];
    T fmx[ACCT_WARPS][7];                 // residual maxima per warp, and per CTA of the cluster
    int imx[ACCT_WARPS];
    T xmx[ACCT_CLUSTER][7];
    int ximx[ACCT_CLUSTER];
    T xs[SMAX];                           // where each sector is evaluated (nu, or its edge's root)
    T blo[SMAX], bhi[SMAX];
    T wh[SMAX], wl[SMAX];                 // last edge roots
    T part[ACCT_WARPS][KMAX];             // B'X per warp
    T xp[2][ACCT_CLUSTER][KMAX];          // and per CTA of the cluster
    T P[KMAX], Q[KMAX], P0[KMAX], tv[KMAX], s[KMAX], ys[KMAX];
    T x, t, g;                            // what warp 0 tells the block: nu, theta, turnover - tau
    int code;
    int sec[SMAX + 1];                    // sector ranges in this CTA's entries
    int npw[ACCT_WARPS], nseg[ACCT_WARPS];
};

// ---- packed FP32 arithmetic and the chunks of a row of B ------------------------------------
__device__ __forceinline__ void fma2(float2& acc, float2 a, float2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;"
        : "+l"(reinterpret_cast<unsigned long long&>(acc))
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
}
__device__ __forceinline__ void fma2(double2& acc, double2 a, double2 b) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.y = fma(a.y, b.y, acc.y);
}
template <typename T> struct Two;
template <> struct Two<float> { using type = float2; };
template <> struct Two<double> { using type = double2; };

// A 16-byte chunk as pairs of T.
template <typename T, typename BT> struct Chunk;
template <> struct Chunk<float, __nv_bfloat16> {
    static constexpr int N = 8;
    float2 v[4];
    __device__ __forceinline__ explicit Chunk(uint4 u) {
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = make_float2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
    }
};
template <> struct Chunk<float, float> {
    static constexpr int N = 4;
    float2 v[2];
    __device__ __forceinline__ explicit Chunk(uint4 u) {
        v[0] = make_float2(__uint_as_float(u.x), __uint_as_float(u.y));
        v[1] = make_float2(__uint_as_float(u.z), __uint_as_float(u.w));
    }
};
template <> struct Chunk<double, double> {
    static constexpr int N = 2;
    double2 v[1];
    __device__ __forceinline__ explicit Chunk(uint4 u) {
        v[0] = make_double2(__hiloint2double(int(u.y), int(u.x)), __hiloint2double(int(u.w), int(u.z)));
    }
};

// Chunks of a row (those of whole 4-factor tiles) and the odd number it takes.
__host__ __device__ inline int row_chunks(int K, int per) { return per == 2 ? 2 * ((K + 3) / 4) : (K + per - 1) / per; }
__host__ __device__ inline int row_stride(int K, int per) { return row_chunks(K, per) | 1; }

// Four consecutive elements of a row, the first a multiple of four.
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&o)[4]) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    o[0] = __uint_as_float(u.x << 16); o[1] = __uint_as_float(u.x & 0xffff0000u);
    o[2] = __uint_as_float(u.y << 16); o[3] = __uint_as_float(u.y & 0xffff0000u);
}
__device__ __forceinline__ void load4(const float* p, float (&o)[4]) {
    const float4 u = *reinterpret_cast<const float4*>(p);
    o[0] = u.x; o[1] = u.y; o[2] = u.z; o[3] = u.w;
}
__device__ __forceinline__ void load4(const double* p, double (&o)[4]) {
    const double2 u = reinterpret_cast<const double2*>(p)[0], w = reinterpret_cast<const double2*>(p)[1];
    o[0] = u.x; o[1] = u.y; o[2] = w.x; o[3] = w.y;
}

// ---- safeguarded Newton step for a nonincreasing piecewise-linear g -------------------------
__device__ __forceinline__ float quotient(float a, float b) { return __fdividef(a, b); }   // a step: 2 ulp do
__device__ __forceinline__ double quotient(double a, double b) { return a / b; }

template <typename T>
struct ARoot {
    T x, a, b, step;
    bool done;
    __device__ __forceinline__ void init(T x0, T st) { x = x0; a = -T(FLT_MAX); b = T(FLT_MAX); step = st; done = false; }
    // g = S(x) - target, cnt entries of slope -1/rho
    __device__ __forceinline__ void update(T g, int cnt, T rho, T tol) {
        if (fabs(g) <= tol) { done = true; return; }
        if (g > T(0)) a = x; else b = x;
        T xn = x;
        bool ok = false;
        if (cnt > 0) {
            xn = x + quotient(g * rho, T(cnt));
            ok = xn > a && xn < b;
        }
        const bool closed = a > -T(FLT_MAX) && b < T(FLT_MAX);
        if (!ok) {
            if (closed) xn = T(0.5) * (a + b);
            else { xn = (g > T(0)) ? x + step : x - step; step *= T(2); }
        }
        if (closed && (b - a) <= AcctTol<T>::WIDTH * fmax(T(1e-6), fabs(a) + fabs(b))) {
            x = T(0.5) * (a + b);
            done = true;
            return;
        }
        x = xn;
    }
};

__device__ __forceinline__ float acct_rho(float, int j) { return float(RHO_MIN) * exp10f(float(j) / float(RHO_PER_DECADE)); }
__device__ __forceinline__ double acct_rho(double, int) { return 0.0; }    // (FP64 penalties are on no grid)

__device__ __forceinline__ float warp_maxv(float v) {      // of values >= 0 (a NaN is reported apart)
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_maxv(double v) { return warp_max(v); }

template <typename T, typename BT, int E, int THREADS, bool GEN, bool CL>
__global__ void __launch_bounds__(THREADS, 1) k_acct_admm(AcctArgs<T> A) {
    using T2 = typename Two<T>::type;
    using Ch = Chunk<T, BT>;
    constexpr int PC = Ch::N;                       // elements per chunk
    extern __shared__ __align__(16) unsigned char acct_smem[];
    AcctShared<T>& sh = *reinterpret_cast<AcctShared<T>*>(acct_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = NT >> 5;
    const int K = A.K, S = A.S;
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = CL ? int(cluster.num_blocks()) : 1, rank = CL ? int(cluster.block_rank()) : 0;
    const int slot = CL ? int(blockIdx.x) / CS : int(blockIdx.x);
    const int a = A.order ? A.order[slot] : slot;
    if (!A.active[a]) return;                       // the same answer in every CTA of the cluster
    if constexpr (CL) cluster.sync();               // a CTA's shared memory may be written to once it has started
    constexpr bool own = sizeof(T) == 8;            // C^{-1} formed and inverted here
    const bool fac = GEN && A.flo != nullptr;
    // ---- shared memory behind the fixed part: C^{-1}, G, 1 / (2 d + rho) (own), the rows of B, cost rows
    const int ldc = ((K + 31) / 32) * 32 + 8;
    T* Ci = reinterpret_cast<T*>(acct_smem + (sizeof(AcctShared<T>) + 15) / 16 * 16);
    T* Gm = Ci + K * ldc;
    const int nc = row_chunks(K, PC), ncs = row_stride(K, PC);
    // ---- this CTA's entries
    const size_t base = (size_t)a * A.Npad;
    const int n = A.N;
    const int per = CL ? (n + CS - 1) / CS : n;
    const int i0 = rank * per, my = max(0, min(per, n - i0));
    // A thread's entries are consecutive: entry e of lane l of warp w is number 32 E w + E l + e. Their
    // rows of B sit at slot 32 E w + 32 e + l, so that a warp's rows are consecutive for each e;
    // slots without an entry hold zeros.
    const int slots = NT * E;
    T* Cj = Gm + (fac ? K * ldc : 0);                // (own) the other buffer of the inversion
    T* wrow = Cj + (own ? K * ldc : 0);
    uint4* Brow = reinterpret_cast<uint4*>(wrow + (own ? slots : 0));
    T* pwrow = reinterpret_cast<T*>(Brow + (size_t)slots * ncs);
    for (int s = tid; s <= S; s += NT)
        sh.sec[s] = max(0, min(my, A.sec_start[s] - i0));
    for (int s = tid; s < S; s += NT) {
        sh.blo[s] = A.band_lo[a * S + s];
        sh.bhi[s] = A.band_hi[a * S + s];
        sh.wh[s] = T(A.eta_hi[a * S + s]);          // NaN before the first solve
        sh.wl[s] = T(A.eta_lo[a * S + s]);
    }
    if (tid < KMAX) { sh.P[tid] = T(0); sh.Q[tid] = T(0); }
    if (fac && tid < K) {
        sh.s[tid] = A.resume ? A.s[(size_t)a * K + tid] : T(0);
        sh.ys[tid] = A.resume ? A.ys[(size_t)a * K + tid] : T(0);
    }
    for (int e = tid; e < slots * nc; e += NT) {
        const int i = e / nc, c = e - i * nc;         // entry i of this CTA, its slot
        const int r = i % (32 * E), sl = i - r + 32 * (r % E) + r / E;
        uint4 u = make_uint4(0, 0, 0, 0);
        if (i < my) {
            const int p = i0 + i;
            if constexpr (sizeof(BT) == 2) u = reinterpret_cast<const uint4*>(A.B16p + (size_t)p * KMAX)[c];
            else if constexpr (sizeof(BT) == 4) u = reinterpret_cast<const uint4*>(A.B32p + (size_t)p * KMAX)[c];
            else {
                const double* q = A.B64 + (size_t)p * K + 2 * c;
                const double b0 = 2 * c < K ? q[0] : 0.0, b1 = 2 * c + 1 < K ? q[1] : 0.0;
                u = make_uint4(__double2loint(b0), __double2hiint(b0), __double2loint(b1), __double2hiint(b1));
            }
        }
        Brow[(size_t)sl * ncs + c] = u;
    }
    T z[E], y[E], v[E], w0[E], lo[E], up[E], c1[E], mu[E];
    int pw[E];
    unsigned long long secp = 0;                    // sector of each entry, 8 bits each (255: no entry)
    const bool has_pw = GEN && A.pw_idx != nullptr;
    __syncthreads();
    const int ib = tid * E, slot0 = warp * 32 * E + lane;
    int n_row = 0, n_seg = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = ib + e;
        const bool in = i < my;
        const int p = in ? i0 + i : 0;
        w0[e] = in ? A.w0[base + p] : T(0);
        lo[e] = in ? A.lo[base + p] : T(0);
        up[e] = in ? A.up[base + p] : T(0);
        c1[e] = in ? A.c[base + p] : T(0);
        mu[e] = in ? A.mu[p] + (A.tilt ? A.tilt[base + p] : T(0)) : T(0);
        z[e] = (A.resume && in) ? A.z[base + p] : fmin(fmax(w0[e], lo[e]), up[e]);
        // (the tilt belongs to the costs that the projection prices, as in the batched kernels' cost rows:
        // with y + tilt in the place of y that is the iteration with mu + tilt, started from y = tilt)
        y[e] = !in ? T(0) : (A.resume ? A.y[base + p] : (A.tilt ? A.tilt[base + p] : T(0)));
        pw[e] = (has_pw && in) ? A.pw_idx[base + p] : -1;
        n_row += pw[e] >= 0;
        if (pw[e] >= 0) n_seg = max(n_seg, A.pw_nbp[pw[e]] - 1);
        v[e] = T(0);
        int s = 255;
        if (in) {
            s = 0;
            int b = S;                               // the sector range that holds i
            while (b - s > 1) {
                const int m = (s + b) >> 1;
                if (sh.sec[m] <= i) s = m; else b = m;
            }
        }
        secp |= (unsigned long long)s << (8 * e);
    }
    // runs of one sector: brk bit e: entry e begins another sector than e - 1 of this thread; the run
    // that ends in a thread began in lane run0; cont: the thread's first run began in an earlier lane
    unsigned brk = 0;
#pragma unroll
    for (int e = 1; e < E; ++e) brk |= (((secp >> (8 * e)) ^ (secp >> (8 * e - 8))) & 255ull) ? 1u << e : 0u;
    const bool any_brk = __any_sync(0xffffffffu, brk != 0);
    const int s_first = int(secp & 255u), s_last = int((secp >> (8 * (E - 1))) & 255u);
    const int prev = __shfl_up_sync(0xffffffffu, s_last, 1), next = __shfl_down_sync(0xffffffffu, s_first, 1);
    const bool cont = lane > 0 && prev == s_first;
    const unsigned starts = __ballot_sync(0xffffffffu, brk != 0 || !cont);
    const int run0 = 31 - __clz(starts & (0xffffffffu >> (31 - lane)));
    const bool ends = s_last != 255 && (lane == 31 || next != s_last);
    // cost rows of this CTA in shared memory when they fit (else read from the tables)
    bool rows_here = false;
    if (has_pw) {
        const int warp_rows = __reduce_add_sync(0xffffffffu, n_row);
        n_seg = __reduce_max_sync(0xffffffffu, n_seg);
        if (lane == 0) { sh.npw[warp] = warp_rows; sh.nseg[warp] = n_seg; }
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < NW; ++w) {
            if (w < warp) before += sh.npw[w];
            total += sh.npw[w];
            n_seg = max(n_seg, sh.nseg[w]);
        }
        rows_here = total <= A.pw_rows;
        if (rows_here) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const unsigned b = __ballot_sync(0xffffffffu, pw[e] >= 0);
                if (pw[e] >= 0) {
                    // rows shorter than the longest end in segments of no length
                    const int q = before + __popc(b & ((1u << lane) - 1u)), nb = A.pw_nbp[pw[e]];
                    const T* bp = A.pw_bp + (size_t)pw[e] * MAXBP;
                    const T* sl = A.pw_sl + (size_t)pw[e] * (MAXBP - 1);
                    T* r = pwrow + (size_t)q * PWROW;
                    r[0] = bp[0];
                    for (int j = 0; j < n_seg; ++j) {
                        r[1 + 2 * j] = j + 1 < nb ? sl[j] : T(0);
                        r[2 + 2 * j] = j + 1 < nb ? bp[j + 1] : bp[nb - 1];
                    }
                    pw[e] = q;
                }
                before += __popc(b);
            }
        }
    }
    int j = A.rho_idx[a];
    T rho = own ? (A.resume ? A.rho_state[a] : A.rho0) : acct_rho(T(0), j), irho = T(1) / rho;
    T nu = T(A.nu[a]), theta = T(0);
    if (GEN) theta = own ? (A.resume ? A.theta_state[a] : T(0)) : T(A.theta[a]);
    int it = A.iters[a];
    const T tau = (GEN && A.tau) ? A.tau[a] : T(INFINITY);
    const bool has_cap = GEN && isfinite(tau);
    int xb = 0;                                      // buffer of the cluster's exchange

    // ---- the entries at a multiplier ----------------------------------------------------------
    auto sector_of = [&](int e) { return int((secp >> (8 * e)) & 255u); };
    // z_e at (arg_e, th): the prox of (phi + th |. - w0|) / rho on [l, u] at v - arg / rho; lin: on a
    // linear piece, sgn: its side of w0
    T zz[E];
    int lin[E], sgn[E];
    auto prox = [&](bool each, T x, T th) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const T t = v[e] - (each ? sh.xs[sector_of(e) & (SMAX - 1)] : x) * irho;
            const T k = (c1[e] + th) * irho;
            T r = (t > w0[e] + k) ? t - k : ((t < w0[e] - k) ? t + k : w0[e]);
            r = fmin(fmax(r, lo[e]), up[e]);
            lin[e] = (r > lo[e] && r < up[e] && r != w0[e]) ? 1 : 0;
            if (GEN) sgn[e] = r > w0[e] ? lin[e] : -lin[e];
            zz[e] = r;
        }
        if (!GEN || !has_pw) return;
        if (rows_here) {
            // the last segment whose minimiser lies right of its left end holds the answer; all the
            // thread's rows side by side, so that their loads overlap
            T t[E], left[E];
            const T* r[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                t[e] = v[e] - (each ? sh.xs[sector_of(e) & (SMAX - 1)] : x) * irho;
                r[e] = pwrow + max(pw[e], 0) * PWROW;
                left[e] = r[e][0];
                if (pw[e] >= 0) { zz[e] = left[e]; lin[e] = 0; sgn[e] = 0; }
            }
            for (int q = 0; q < n_seg; ++q) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const T sq = r[e][1 + 2 * q], right = r[e][2 + 2 * q];
                    const bool above = left[e] + right > T(2) * w0[e];
                    const T cand = fmin(t[e] - (sq + (above ? th : -th)) * irho, right);
                    if (pw[e] >= 0 && cand > left[e]) {
                        zz[e] = cand;
                        lin[e] = cand < right;
                        sgn[e] = cand < right ? (above ? 1 : -1) : 0;
                    }
                    left[e] = right;
                }
            }
            return;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (pw[e] < 0) continue;
            const T t = v[e] - (each ? sh.xs[sector_of(e) & (SMAX - 1)] : x) * irho;
            const T* bp = A.pw_bp + (size_t)pw[e] * MAXBP;
            const T* sl = A.pw_sl + (size_t)pw[e] * (MAXBP - 1);
            const int nb = A.pw_nbp[pw[e]];
            zz[e] = bp[nb - 1]; lin[e] = 0; sgn[e] = 0;
            for (int q = 0; q + 1 < nb; ++q) {
                const int sg = (bp[q] + bp[q + 1] > T(2) * w0[e]) ? 1 : -1;
                const T cand = t - (sl[q] + (sg > 0 ? th : -th)) * irho;
                if (cand <= bp[q]) { zz[e] = bp[q]; break; }
                if (cand < bp[q + 1]) { zz[e] = cand; lin[e] = 1; sgn[e] = sg; break; }
            }
        }
    };
    // Every sector at x (each: sector s at sh.xs[s]): afterwards warp 0 can gather() the sector sums of the
    // whole account, and with two also the turnover. Block-collective (cluster-collective).
    auto eval = [&](bool each, T x, T th, bool sums, bool two) {
        prox(each, x, th);
        if (sums) {
            T f = zz[0];
            int m = lin[0];
            T head = T(0);
            int hm = 0;
            if (any_brk) {
                bool first = true;
#pragma unroll
                for (int e = 1; e < E; ++e) {
                    if (brk & (1u << e)) {            // the run of entry e - 1 ends
                        if (first) { head = f; hm = m; first = false; }
                        else if (sector_of(e - 1) != 255) sh.seg[warp + sector_of(e - 1)] = {f, m};
                        f = T(0); m = 0;
                    }
                    f += zz[e]; m += lin[e];
                }
            } else {
#pragma unroll
                for (int e = 1; e < E; ++e) { f += zz[e]; m += lin[e]; }
            }
            // segmented inclusive scan of the threads' last runs
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const T fo = __shfl_up_sync(0xffffffffu, f, o);
                const int mo = __shfl_up_sync(0xffffffffu, m, o);
                if (lane - o >= run0) { f += fo; m += mo; }
            }
            if (any_brk) {
                const T fo = __shfl_up_sync(0xffffffffu, f, 1);
                const int mo = __shfl_up_sync(0xffffffffu, m, 1);
                if (brk && s_first != 255) sh.seg[warp + s_first] = {cont ? head + fo : head, cont ? hm + mo : hm};
            }
            if (ends) sh.seg[warp + s_last] = {f, m};
        }
        if (GEN && two) {
            T u = T(0);
            int m = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) { u += fabs(zz[e] - w0[e]); m += sgn[e]; }
            u = warp_sum(u);
            m = __reduce_add_sync(0xffffffffu, m);
            if (lane == 0) sh.turn[warp] = {u, m};
        }
        __syncthreads();
        if constexpr (CL) {
            auto here = [&](int s) {
                SumCount<T> t{T(0), 0};
                const int b = sh.sec[s], e = sh.sec[s + 1];
                if (e > b)
                    for (int q = b / (32 * E); q <= (e - 1) / (32 * E); ++q) { t.f += sh.seg[q + s].f; t.n += sh.seg[q + s].n; }
                return t;
            };
            for (int r = warp; r < CS; r += NW) {     // warp r tells CTA r
                AcctShared<T>* o = cluster.map_shared_rank(&sh, r);
                if (sums)
                    for (int s = lane; s < S; s += 32) o->xseg[xb][rank][s] = here(s);
                if (GEN && two && lane == 0) {
                    SumCount<T> t{T(0), 0};
                    for (int w = 0; w < NW; ++w) { t.f += sh.turn[w].f; t.n += sh.turn[w].n; }
                    o->xturn[xb][rank] = t;
                }
            }
            cluster.sync();
            xb ^= 1;
        }
    };
    // (warp 0) the sums of its lanes' sectors over the account, and their counts
    const int s0 = lane, s1 = lane + 32;
    const bool wide = S > 32;
    auto segments = [&](int s) {                      // the warps that hold entries of sector s: first, last
        const int b = s < S ? sh.sec[s] : 0, e = s < S ? sh.sec[s + 1] : 0;
        return e > b ? make_int2(b / (32 * E), (e - 1) / (32 * E)) : make_int2(0, -1);
    };
    const int2 g0 = segments(s0), g1 = segments(s1);
    const T lo0 = s0 < S ? sh.blo[s0] : T(0), hi0 = s0 < S ? sh.bhi[s0] : T(0);
    const T lo1 = s1 < S ? sh.blo[s1] : T(0), hi1 = s1 < S ? sh.bhi[s1] : T(0);
    auto gather = [&](int s, int2 g) {
        SumCount<T> t{T(0), 0};
        if constexpr (CL) {
            if (s < S)
                for (int r = 0; r < CS; ++r) { const SumCount<T> c = sh.xseg[xb ^ 1][r][s]; t.f += c.f; t.n += c.n; }
        } else {
            for (int q = g.x; q <= g.y; ++q) { const SumCount<T> c = sh.seg[q + s]; t.f += c.f; t.n += c.n; }
        }
        return t;
    };
    auto gather_turn = [&]() {
        SumCount<T> t{T(0), 0};
        if constexpr (CL) {
            for (int r = 0; r < CS; ++r) { t.f += sh.xturn[xb ^ 1][r].f; t.n += sh.xturn[xb ^ 1][r].n; }
        } else {
            for (int w = 0; w < NW; ++w) { t.f += sh.turn[w].f; t.n += sh.turn[w].n; }
        }
        return t;
    };
    bool clamped = false;                             // some sector sits on its band edge (all threads alike)
    auto over = [&](T v_, T edge) { return v_ > edge + AcctTol<T>::ROOT * fmax(edge, T(1e-3)); };
    auto under = [&](T v_, T edge) { return v_ < edge - AcctTol<T>::ROOT * fmax(fabs(edge), T(1e-3)); };
    // (warp 0) its lanes' sector sums; the clamped budget sum and the count that moves it
    SumCount<T> c0{T(0), 0}, c1s{T(0), 0};
    auto budget = [&](int& m) -> T {
        c0 = gather(s0, g0);
        T t = fmin(fmax(c0.f, lo0), hi0);             // (no sector: 0 within [0, 0])
        m = (c0.f > lo0 && c0.f < hi0) ? c0.n : 0;
        if (wide) {
            c1s = gather(s1, g1);
            t += fmin(fmax(c1s.f, lo1), hi1);
            if (c1s.f > lo1 && c1s.f < hi1) m += c1s.n;
        }
        m = __reduce_add_sync(0xffffffffu, m);
        return warp_sum(t);
    };
    auto leaves_band = [&]() -> bool {
        bool out = over(c0.f, hi0) || under(c0.f, lo0);
        if (wide) out |= over(c1s.f, hi1) || under(c1s.f, lo1);
        return __any_sync(0xffffffffu, out);
    };
    // The projection at a given th: the budget reads sum_s clamp(S_s(nu), lo_s, hi_s) = 1, S_s
    // nonincreasing; then each sector outside its band gets its edge's root, all of them at
    // once. Returns nu; leaves `clamped` and, when it is set, sh.xs.
    // `stale` is set when zz is not at the point returned (see close).
    bool stale = false;
    T close = T(0);
    auto project = [&](T nu0, T th) -> T {
        const T step = T(0.05) * rho + T(1e-6);
        ARoot<T> R;
        R.init(nu0, step);
        T x = nu0;
        int code = 0;
        for (int q = 0; q < ROOT_IT + 2; ++q) {
            eval(false, x, th, true, false);
            if (warp == 0) {
                int m;
                const T t = budget(m);
                const bool near = !has_cap && m > 0 && fabs(t - T(1)) <= close;
                if (!R.done) R.update(t - T(1), m, rho, AcctTol<T>::ROOT);
                // done at the point just evaluated: 1, or 2 when some sector leaves its band there. Closer than
                // the iterations' own residual the step is taken without a look at where it leads (3):
                // the sums are linear between kinks, so that it is off by much less again
                int c = 0;
                if ((R.done && R.x == x) || q + 1 == ROOT_IT + 2) c = leaves_band() ? 2 : 1;
                else if (near && !leaves_band()) c = 3;
                if (lane == 0) { sh.x = (c == 1 || c == 2) ? x : R.x; sh.code = c; }
            }
            __syncthreads();
            x = sh.x;
            code = sh.code;
            if (code) break;
        }
        clamped = code == 2;
        stale = code == 3;
        if (!clamped) return x;
        __syncthreads();                              // (every warp has read sh.code)
        // edges: lane l of warp 0 owns sectors l and l + 32
        ARoot<T> E0, E1;
        T t0 = T(0), t1 = T(0);
        auto edge = [&](int s, T Sv, ARoot<T>& Q, T& target) {
            Q.init(x, step);
            Q.done = true;
            if (s >= S) return;
            if (over(Sv, sh.bhi[s])) {
                target = sh.bhi[s];
                const T w = sh.wh[s];
                Q.init((w > x && w < T(FLT_MAX)) ? w : x, step);
                Q.a = x;
            } else if (under(Sv, sh.blo[s])) {
                target = sh.blo[s];
                const T w = sh.wl[s];
                Q.init((w < x && w > -T(FLT_MAX)) ? w : x, step);
                Q.b = x;
            }
        };
        if (warp == 0) {
            edge(s0, c0.f, E0, t0);
            edge(s1, c1s.f, E1, t1);
        }
        for (int q = 0; q <= ROOT_IT; ++q) {
            if (warp == 0) {
                if (s0 < S) sh.xs[s0] = E0.x;
                if (s1 < S) sh.xs[s1] = E1.x;
                const bool more = __any_sync(0xffffffffu, !E0.done || !E1.done);
                if (lane == 0) sh.code = more;
            }
            __syncthreads();
            const bool more = sh.code != 0;
            if (!more || q == ROOT_IT) break;
            eval(true, x, th, true, false);
            if (warp == 0) {
                c0 = gather(s0, g0);
                if (!E0.done) E0.update(c0.f - t0, c0.n, rho, AcctTol<T>::ROOT * fmax(fabs(t0), T(1e-3)));
                if (wide) {
                    c1s = gather(s1, g1);
                    if (!E1.done) E1.update(c1s.f - t1, c1s.n, rho, AcctTol<T>::ROOT * fmax(fabs(t1), T(1e-3)));
                }
            }
        }
        __syncthreads();                              // (sh.code has been read)
        return x;
    };
    auto turnover = [&](T x, T th) -> T {             // - tau
        eval(clamped, x, th, false, true);
        if (warp == 0) {
            const T u = gather_turn().f - tau;
            if (lane == 0) sh.g = u;
        }
        __syncthreads();
        return sh.g;
    };

    // ---- capacitance ------------------------------------------------------------------------
    // C^{-1} at the penalty into shared memory: from the universe's table (index j), or (FP64) formed from
    // the rows of B and inverted here
    T idl[E];
    auto capacitance = [&]() -> bool {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            idl[e] = T(0);
            if (ib + e < my) {
                idl[e] = T(1) / (T(2) * A.d[i0 + ib + e] + rho);
            }
            if (own) wrow[slot0 + 32 * e] = idl[e];
        }
        __syncthreads();
        if constexpr (!own) {
            for (int e = tid; e < K * K; e += NT) {
                const int r = e / K, c = e - r * K;
                Ci[r * ldc + c] = T(A.Cinv[(size_t)j * K * K + e]);
                if (fac) Gm[r * ldc + c] = T(A.G[(size_t)j * K * K + e]);
            }
            __syncthreads();
            return true;
        }
        // G by 4 x 4 tiles of factors, the rows cut into as many groups as the threads allow
        const BT* Bs = reinterpret_cast<const BT*>(Brow);
        const int ldb = ncs * PC;
        const int kb = (K + 3) / 4, tiles = kb * kb, groups = max(1, NT / tiles);
        for (int t0 = 0; t0 < tiles; t0 += NT) {
            const int tile = t0 + (groups > 1 ? tid % tiles : tid), g = groups > 1 ? tid / tiles : 0;
            const bool on = tile < tiles && g < groups;
            T acc[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = T(0);
            const int r0 = on ? 4 * (tile / kb) : 0, k0 = on ? 4 * (tile % kb) : 0;
            if (on) {
#pragma unroll 2
                for (int i = g; i < slots; i += groups) {
                    T br[4], bc[4];
                    load4(Bs + (size_t)i * ldb + r0, br);
                    load4(Bs + (size_t)i * ldb + k0, bc);
                    const T w = wrow[i];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const T bw = br[r] * w;
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[r][c] = fma(bw, bc[c], acc[r][c]);
                    }
                }
            }
            for (int h = 0; h < groups; ++h) {        // the groups add in turn
                if (on && g == h)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (r0 + r < K && k0 + c < K) {
                                T* o = &Ci[(r0 + r) * ldc + k0 + c];
                                *o = (h == 0) ? acc[r][c] : *o + acc[r][c];
                            }
                __syncthreads();
            }
        }
        for (int r = warp; r < K; r += NW)
            for (int c = lane; c < K; c += 32) {
                const T g = Ci[r * ldc + c];
                if (fac) Gm[r * ldc + c] = g;
                if (r == c) Ci[r * ldc + c] = g + (fac ? T(1) / (T(2) * A.f[r] + rho) : T(1) / (T(2) * A.f[r]));
            }
        __syncthreads();
        // Gauss-Jordan inversion, positive definite, so without pivoting; each step from one buffer into the
        // other, one barrier a step
        bool fine = true;
        T *from = Ci, *to = Cj;
        for (int k = 0; k < K; ++k) {
            const T piv = from[k * ldc + k];
            fine = fine && piv > T(0) && isfinite(piv);
            const T ip = T(1) / piv;
            for (int r = warp; r < K; r += NW) {
                const T f = -from[r * ldc + k] * ip;
                for (int c = lane; c < K; c += 32) {
                    const T p = from[k * ldc + c];
                    T q = (r == k) ? p * ip : fma(f, p, from[r * ldc + c]);
                    if (c == k) q = (r == k) ? ip : f;
                    to[r * ldc + c] = q;
                }
            }
            __syncthreads();
            T* t = from; from = to; to = t;
        }
        if (K & 1) {
            for (int r = warp; r < K; r += NW)
                for (int c = lane; c < K; c += 32) Ci[r * ldc + c] = Cj[r * ldc + c];
            __syncthreads();
        }
        return fine;
    };
    // sum_j M[k][j] x[j] for k < K to out (shared): eight lanes per row
    auto matvec = [&](const T* Mx, const T* x, auto&& out) {
        for (int k0 = 0; k0 < K; k0 += NT / 8) {
            const int k = k0 + (tid >> 3), sub = tid & 7;
            if (k0 + 4 * warp >= K) break;            // (a warp's four rows are past the end)
            T acc = T(0);
            if (k < K)
                for (int q = sub; q < K; q += 8) acc = fma(Mx[k * ldc + q], x[q], acc);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            if (sub == 0 && k < K) out(k, acc);
        }
        __syncthreads();
    };
    // B'X of this warp's entries for factors h .. h + W - 1: per thread over its rows, then a transposing
    // reduction that leaves factor h + lane's sum in lane
    T X[E];
    auto products = [&](int h, auto width) {
        constexpr int W = decltype(width)::value;
        T2 acc[W / 2];
#pragma unroll
        for (int q = 0; q < W / 2; ++q) acc[q].x = acc[q].y = T(0);
#pragma unroll
        for (int cq = 0; cq < W / PC; ++cq) {
            const int c = h / PC + cq;
            if (c < nc) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const Ch b(Brow[(slot0 + 32 * e) * ncs + c]);
                    T2 xx;
                    xx.x = xx.y = X[e];
#pragma unroll
                    for (int q = 0; q < PC / 2; ++q) fma2(acc[cq * (PC / 2) + q], xx, b.v[q]);
                }
            }
        }
        T r[W];
#pragma unroll
        for (int q = 0; q < W / 2; ++q) { r[2 * q] = acc[q].x; r[2 * q + 1] = acc[q].y; }
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) {
            const bool hi = lane & o;
#pragma unroll
            for (int q = 0; q < o; ++q) {
                const T send = hi ? r[q] : r[q + o], keep = hi ? r[q + o] : r[q];
                r[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
#pragma unroll
        for (int o = W; o < 32; o <<= 1) r[0] += __shfl_xor_sync(0xffffffffu, r[0], o);
        if (lane < W) sh.part[warp][h + lane] = r[0];
    };

    bool go = true, fresh = true;                     // fresh: a new penalty
    int status = 0;
    bool stopped = false;                             // out of time, still iterating
    bool closing = false;                             // stopped: the last iterate's root is taken to its tolerance
    bool watch = false;                               // near the target: the entries' places are followed
    unsigned held = 0;                                // this thread's entries' places, two bits each
    int quiet = 0, met = 0;                           // iterations without a change; where the target was met
    int pbuf = 0;
    while (go) {
        T rps = T(0), rds = T(0);
        if (!closing) {
            if (fresh) {
                if (!capacitance()) { status = PRISM_NUMERICAL_FAILURE; break; }
                fresh = false;
            }
            // ---- X and P = B'X
#pragma unroll
            for (int e = 0; e < E; ++e) X[e] = (mu[e] + rho * z[e] - y[e]) * idl[e];
            for (int h = 0; h < K; h += 32) {
                if (K - h > 16) products(h, std::integral_constant<int, 32>());
                else products(h, std::integral_constant<int, 16>());
            }
            __syncthreads();
            if constexpr (CL) {
                if (tid < K) {
                    T t = T(0);
                    for (int w = 0; w < NW; ++w) t += sh.part[w][tid];
                    for (int r = 0; r < CS; ++r) cluster.map_shared_rank(&sh, r)->xp[pbuf][rank][tid] = t;
                }
                cluster.sync();
                if (tid < K) {
                    T t = T(0);
                    for (int r = 0; r < CS; ++r) t += sh.xp[pbuf][r][tid];
                    sh.P[tid] = t;
                }
                pbuf ^= 1;
            } else if (tid < K) {
                T t0 = T(0), t1 = T(0);
                int w = 0;
                for (; w + 1 < NW; w += 2) { t0 += sh.part[w][tid]; t1 += sh.part[w + 1][tid]; }
                if (w < NW) t0 += sh.part[w][tid];
                sh.P[tid] = t0 + t1;
            }
            __syncthreads();
            // ---- Q = C^{-1} P; with the factor block (s = B'x, dual ys) Q' = C^{-1}(P + G tv) - tv,
            // tv = rho s - ys, and B'x = P - G Q'
            if (fac) {
                if (tid < K) { sh.tv[tid] = rho * sh.s[tid] - sh.ys[tid]; sh.P0[tid] = sh.P[tid]; }
                __syncthreads();
                matvec(Gm, sh.tv, [&](int k, T g) { sh.P[k] = sh.P0[k] + g; });
                matvec(Ci, sh.P, [&](int k, T q) { sh.Q[k] = q - sh.tv[k]; });
                T rp = T(0), rd = T(0);
                int bad = 0;
                matvec(Gm, sh.Q, [&](int k, T g) {
                    const T bx = sh.P0[k] - g, so = sh.s[k], yo = sh.ys[k];
                    const T xh = A.alpha * bx + (T(1) - A.alpha) * so;
                    const T sn = fmin(fmax(xh + yo * irho, A.flo[(size_t)a * K + k]), A.fhi[(size_t)a * K + k]);
                    sh.s[k] = sn;
                    sh.ys[k] = yo + rho * (xh - sn);
                    rp = fmax(rp, fabs(xh - sn));
                    rd = fmax(rd, rho * fabs(sn - so));
                    bad |= !(isfinite(xh) && isfinite(sn));
                });
                rps = bad ? T(INFINITY) : rp;
                rds = bad ? T(INFINITY) : rd;
            } else {
                matvec(Ci, sh.P, [&](int k, T q) { sh.Q[k] = q; });
            }
            // ---- B Q, x and v
            T bq[E];
            {
                T2 acc[E];
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e].x = acc[e].y = T(0);
#pragma unroll 2
                for (int c = 0; c < nc; ++c) {
                    T2 q2[PC / 2];
#pragma unroll
                    for (int q = 0; q < PC / 2; ++q) q2[q] = reinterpret_cast<const T2*>(sh.Q)[c * (PC / 2) + q];
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const Ch b(Brow[(slot0 + 32 * e) * ncs + c]);
#pragma unroll
                        for (int q = 0; q < PC / 2; ++q) fma2(acc[e], b.v[q], q2[q]);
                    }
                }
#pragma unroll
                for (int e = 0; e < E; ++e) bq[e] = acc[e].x + acc[e].y;
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const T x = X[e] - bq[e] * idl[e];
                v[e] = A.alpha * x + (T(1) - A.alpha) * z[e] + y[e] * irho;
            }
        }
        // ---- the projection's multipliers
        T th = T(0);
        bool settled = false;
        if (has_cap && theta > T(0) && !clamped) {
            // the cap held last time: Newton on (nu, theta) together. On the linear entries
            // dz/dnu = -1/rho and dz/dtheta = -sign/rho, so with n of them and sign sum s the
            // system is (1/rho) [n s; s n]
            T x = nu, t = theta;
            for (int q = 0; q < PAIR_IT; ++q) {
                eval(false, x, t, true, true);
                if (warp == 0) {
                    int m;
                    const T g1 = budget(m) - T(1);
                    const bool out = leaves_band();
                    const SumCount<T> u = gather_turn();
                    const T g2 = u.f - tau;
                    int c = 0;
                    T xn = x, tn = t;
                    if (fabs(g1) <= AcctTol<T>::ROOT && fabs(g2) <= AcctTol<T>::CAP * tau) {
                        c = out ? 2 : 1;
                    } else {
                        const T det = T(m) * T(m) - T(u.n) * T(u.n);
                        xn = x + rho * (T(m) * g1 - T(u.n) * g2) / det;
                        tn = t + rho * (T(m) * g2 - T(u.n) * g1) / det;
                        if (!(det > T(0)) || !(tn > T(0))) c = 2;
                    }
                    if (lane == 0) { sh.x = xn; sh.t = tn; sh.code = c; }
                }
                __syncthreads();
                const int c = sh.code;
                x = sh.x; t = sh.t;
                if (c) { settled = c == 1; break; }
            }
            __syncthreads();                          // (sh.code has been read)
            if (settled) { nu = x; th = t; stale = false; }
        }
        if (!settled) {
            // without a cap one projection; with one, theta by a bracketed secant (Illinois) on the
            // turnover, nonincreasing in theta: at 0, then up until the cap holds, then inside
            int phase = 0, side = 0;
            T t_lo = T(0), u_lo = T(0), t_hi = T(0), u_hi = T(0);
            for (int q = 0; q < 104; ++q) {
                nu = project(nu, th);
                if (!has_cap) break;
                const T u = turnover(nu, th);
                if (phase == 0) {
                    if (u <= tau * AcctTol<T>::CAP) break;
                    u_lo = u;
                    th = fmax(theta, T(1e-4));
                    phase = 1;
                    continue;
                }
                if (phase == 1) {
                    if (u > T(0) && q < 41) { t_lo = th; u_lo = u; th *= T(4); continue; }
                    t_hi = th; u_hi = u;
                    phase = 2;
                } else {
                    if (fabs(u) <= AcctTol<T>::CAP * tau || (t_hi - t_lo) <= T(0.25) * AcctTol<T>::WIDTH * t_hi) break;
                    if (u > T(0)) {
                        t_lo = th; u_lo = u;
                        if (side == -1) u_hi *= T(0.5);
                        side = -1;
                    } else {
                        t_hi = th; u_hi = u;
                        if (side == 1) u_lo *= T(0.5);
                        side = 1;
                    }
                }
                T tn = t_hi - u_hi * (t_hi - t_lo) / (u_hi - u_lo);
                if (!(tn > t_lo && tn < t_hi)) tn = T(0.5) * (t_lo + t_hi);
                th = tn;
            }
        }
        if (has_cap) theta = th;
        // ---- z, y and the residuals (the norms only where the penalty may adapt)
        const bool adapt = (it + 1) % A.adapt_every == 0;
        T rp = T(0), rd = T(0), nx = T(0), nz = T(0), ny = T(0);
        int flags = 0;
        unsigned codes = 0;
        if (clamped || stale) prox(clamped, nu, th);  // (else zz holds it: nu is where the last evaluation was)
        if (closing) {
#pragma unroll
            for (int e = 0; e < E; ++e) { z[e] = zz[e]; y[e] = rho * (v[e] - zz[e]); }
            break;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const T zn = zz[e];
            const T yn = rho * (v[e] - zn);
            if (ib + e < my) {
                rp = fmax(rp, fabs(yn - y[e]) * irho);
                rd = fmax(rd, rho * fabs(zn - z[e]));
                if (adapt) {
                    nx = fmax(nx, fabs(v[e] - y[e] * irho));
                    nz = fmax(nz, fabs(zn));
                    ny = fmax(ny, fabs(A.tilt ? yn - A.tilt[base + i0 + ib + e] : yn));
                }
                flags |= !(isfinite(zn) && isfinite(yn));
                // its place: inside a linear piece above or below w0, or at a breakpoint, and the same one
                const unsigned code = lin[e] ? (zn > w0[e] ? 1u : 2u) : 0u;
                codes |= code << (2 * e);
                if (watch && (((held >> (2 * e)) & 3u) != code || (code == 0 && zn != z[e]))) flags |= 4;
                z[e] = zn;
                y[e] = yn;
            }
        }
        if (A.budget_ns && rank == 0 && tid == 0) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (now - *A.t0 > A.budget_ns) flags |= 2;
        }
        rp = warp_maxv(rp); rd = warp_maxv(rd);
        if (fac) { rps = warp_maxv(rps); rds = warp_maxv(rds); }
        if (adapt) { nx = warp_maxv(nx); nz = warp_maxv(nz); ny = warp_maxv(ny); }
        flags = __reduce_or_sync(0xffffffffu, unsigned(flags));
        if (lane == 0) {
            T* m = sh.fmx[warp];
            m[0] = rp; m[1] = rd;
            if (adapt) { m[2] = nx; m[3] = nz; m[4] = ny; }
            if (fac) { m[5] = rps; m[6] = rds; }
            sh.imx[warp] = flags;
        }
        __syncthreads();
        auto gather_max = [&](const T (*m)[7], const int* f, int count) {
            const bool in = lane < count;
            rp = warp_maxv(in ? m[lane][0] : T(0)); rd = warp_maxv(in ? m[lane][1] : T(0));
            if (adapt) {
                nx = warp_maxv(in ? m[lane][2] : T(0)); nz = warp_maxv(in ? m[lane][3] : T(0));
                ny = warp_maxv(in ? m[lane][4] : T(0));
            }
            if (fac) { rps = warp_maxv(in ? m[lane][5] : T(0)); rds = warp_maxv(in ? m[lane][6] : T(0)); }
            flags = __reduce_or_sync(0xffffffffu, in ? unsigned(f[lane]) : 0u);
        };
        gather_max(sh.fmx, sh.imx, NW);
        if constexpr (CL) {
            if (tid < CS) {
                AcctShared<T>* o = cluster.map_shared_rank(&sh, tid);
                T* m = o->xmx[rank];
                m[0] = rp; m[1] = rd; m[2] = nx; m[3] = nz; m[4] = ny; m[5] = rps; m[6] = rds;
                o->ximx[rank] = flags;
            }
            cluster.sync();
            gather_max(sh.xmx, sh.ximx, CS);
        }
        ++it;
        // the factor block's residuals take part in the stopping test; the penalty follows the entries' alone
        const T ep = rp, ed = rd;
        rp = fmax(rp, rps); rd = fmax(rd, rds);
        close = rp;
        // The residuals having met their target, the account goes on until its entries have kept their places
        // for A.settle iterations: the polish starts from those places
        held = codes;
        quiet = (watch && !(flags & 4)) ? quiet + 1 : 0;
        watch = A.settle && rp <= T(8) * A.eps && rd <= T(8) * A.eps;
        if (!met && it >= A.min_iter && rp <= A.eps && rd <= A.eps) met = it;
        // ---- control, the same in every thread
        int newj = j;
        T newrho = rho;
        if (flags & 1) { status = PRISM_NUMERICAL_FAILURE; go = false; }
        else if (met && (quiet >= A.settle || it - met >= A.settle_max)) go = false;
        else if (it >= A.max_iter || (flags & 2)) {
            // (past the target it only waited for its entries to settle)
            if (!met && it >= A.max_iter) status = PRISM_TIMEOUT;
            else stopped = !met;
            go = false;
        }
        else if (adapt && own) {
            // FP64 (as in block_admm.cu): any penalty, followed by all residuals, once they are a factor of
            // four apart
            const T tiny = T(1e-35);
            const T pr = rp / fmax(fmax(nx, nz), tiny), du = rd / fmax(ny, tiny);
            const T ratio = sqrt(pr / fmax(du, tiny));
            if (ratio > T(2) || ratio < T(0.5)) newrho = rho * fmin(fmax(ratio, T(0.1)), T(10));
            newrho = fmin(fmax(newrho, T(1e-6)), T(1e6));
        } else if (adapt) {
            const T pr = ep / fmax(fmax(nx, nz), T(1e-12));
            const T du = ed / fmax(ny, T(1e-12));
            const T ratio = sqrt(pr / fmax(du, T(1e-20)));
            int dj = int(lrint(double(RHO_PER_DECADE) * log10(double(fmax(ratio, T(1e-12))))));
            dj = max(-4, min(4, dj));
            newj = max(0, min(NRHO - 1, j + dj));
        }
        // a point whose budget sum nobody looked at (stale) is closed once: an account that does not certify
        // is returned as it stops
        if (!go && stale && !(flags & 1)) { go = closing = true; close = T(0); }
        if (tid < S && clamped) {
            // warm starts of the edges
            const T x = sh.xs[tid];
            if (x > nu) sh.wh[tid] = x;
            if (x < nu) sh.wl[tid] = x;
        }
        if (newj != j || newrho != rho) {
            j = newj;
            rho = own ? newrho : acct_rho(T(0), j);
            irho = T(1) / rho;
            fresh = true;
        }
    }
    // ---- what the polish and a second pass read
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (ib + e < my) {
            const size_t p = base + i0 + ib + e;
            A.z[p] = z[e];
            A.y[p] = y[e];
            if constexpr (sizeof(T) == 8) A.zf[p] = float(z[e]);
        }
    if (rank == 0) {
        for (int s = tid; s < S; s += NT) {
            const T x = clamped ? sh.xs[s] : nu;
            // held at its upper edge: x > nu, at its lower: x < nu. The FP32 copies keep that order
            const float nf = float(nu), xf = float(x);
            A.eta_hi[a * S + s] = x > nu ? fmaxf(xf, nextafterf(nf, FLT_MAX)) : -FLT_MAX;
            A.eta_lo[a * S + s] = x < nu ? fminf(xf, nextafterf(nf, -FLT_MAX)) : FLT_MAX;
        }
        if (fac && tid < K) {
            const T sk = sh.s[tid];
            A.sflag[(size_t)a * K + tid] = sk >= A.fhi[(size_t)a * K + tid] ? 1 : (sk <= A.flo[(size_t)a * K + tid] ? -1 : 0);
            A.s[(size_t)a * K + tid] = sk;
            A.ys[(size_t)a * K + tid] = sh.ys[tid];
        }
        if (tid == 0) {
            A.nu[a] = float(nu);
            A.theta[a] = float(theta);
            A.rho_idx[a] = j;
            if constexpr (own) {
                A.rho_state[a] = rho;
                A.theta_state[a] = theta;
            }
            A.iters[a] = it;
            if (status) A.status[a] = status;
            if (!stopped) A.active[a] = 0;
        }
    }
    if constexpr (CL) cluster.sync();                 // no CTA leaves while another may write to it
}

template <typename T, typename BT, int E, int THREADS, bool GEN, bool CL>
static cudaError_t launch_one(const AcctArgs<T>& A0, const AcctShape& sh, int n_accounts, cudaStream_t st) {
    AcctArgs<T> A = A0;
    A.pw_rows = sh.pw_rows;
    auto* k = k_acct_admm<T, BT, E, THREADS, GEN, CL>;
    // (the limit belongs to the process: every thread sets the same one, whatever it launches with)
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ACCT_SMEM);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_accounts * sh.cluster);
    cfg.blockDim = dim3(sh.threads);
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = sh.cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, A);
}

// The shapes that acct_shape gives.
template <typename BT, bool GEN>
static cudaError_t launch_acct_gen(const AcctArgs<float>& A, const AcctShape& sh, int n, cudaStream_t st) {
    const bool small = sh.threads <= 256;             // (with twice the registers a thread)
    if (sh.cluster > 1) {
        if (small) return launch_one<float, BT, 4, 256, GEN, true>(A, sh, n, st);
        return launch_one<float, BT, 4, 512, GEN, true>(A, sh, n, st);
    }
    if (sh.E == 1) return launch_one<float, BT, 1, 256, GEN, false>(A, sh, n, st);
    if (small) return launch_one<float, BT, 4, 256, GEN, false>(A, sh, n, st);
    return launch_one<float, BT, 4, 512, GEN, false>(A, sh, n, st);
}
template <typename BT>
static cudaError_t launch_acct_float(const AcctArgs<float>& A, const AcctShape& sh, int n, cudaStream_t st) {
    if (A.pw_idx || A.flo || A.tau) return launch_acct_gen<BT, true>(A, sh, n, st);
    return launch_acct_gen<BT, false>(A, sh, n, st);
}

}  // namespace prism
