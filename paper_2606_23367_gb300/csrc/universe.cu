// universe.cu -- prism_create_universe / prism_destroy_universe.
//
// The risk model Sigma = B F B' + D (Eq. 1, factor-structured risk with O(N K)
// products, Sec. 4.2) is copied to the device once, in an asset order that
// makes each sector a contiguous range (the projection step reduces per
// sector). Alongside the FP64 copy the library keeps FP32 and BF16 copies of
// B (row-major and transposed for the tensor-core products) and, for each
// point of the penalty grid rho_j, the inverse of the Woodbury capacitance
//     C_j = (2F)^{-1} + B' Delta_j^{-1} B,   Delta_j = diag(2 d + rho_j),
// which turns the ADMM x-update (2 Sigma + rho I) x = r into K x K work.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <numeric>

#include "common.cuh"

namespace prism {

static thread_local std::string g_last_error;
void set_error(const std::string& msg) { g_last_error = msg; }
const char* last_error() { return g_last_error.c_str(); }

// G_j[k1][k2] = sum_i B[i][k1] B[i][k2] / (2 d_i + rho_j), FP32 products summed
// in FP32 over chunks of 128 assets and in FP64 across chunks. One block per
// (j, 8-row stripe of k1); B rows staged through shared memory.
// blockIdx.z: B in FP32 or as rounded to BF16.
__global__ void k_gram(const float* __restrict__ B32, const __nv_bfloat16* __restrict__ B16,
                       const float* __restrict__ d, int N, int K, double* __restrict__ Gs) {
    const int j = blockIdx.x;
    double* G = Gs + (size_t)blockIdx.z * NRHO * K * K;
    const int k1_0 = blockIdx.y * 8;
    const float rho = float(RHO_MIN * pow(10.0, double(j) / RHO_PER_DECADE));
    __shared__ float sB[128][KMAX + 1];
    __shared__ float sw[128];
    const int t = threadIdx.x;            // 256 threads: pair (k1 = k1_0 + t/32 ... )
    // each thread owns up to 2 (k1, k2) pairs: k1 = k1_0 + (t >> 5), k2 = (t & 31) and +32
    const int k1 = k1_0 + (t >> 5);
    const int k2a = t & 31, k2b = (t & 31) + 32;
    double acc_a = 0.0, acc_b = 0.0;
    for (int i0 = 0; i0 < N; i0 += 128) {
        __syncthreads();
        for (int e = t; e < 128 * K; e += 256) {
            int r = e / K, c = e % K;
            int i = i0 + r;
            sB[r][c] = (i < N) ? (blockIdx.z ? __bfloat162float(B16[(size_t)i * K + c]) : B32[(size_t)i * K + c]) : 0.f;
        }
        for (int r = t; r < 128; r += 256) {
            int i = i0 + r;
            sw[r] = (i < N) ? 1.0f / (2.0f * d[i] + rho) : 0.f;
        }
        __syncthreads();
        if (k1 < K) {
            float pa = 0.f, pb = 0.f;
            for (int r = 0; r < 128; ++r) {
                float bw = sB[r][k1] * sw[r];
                if (k2a < K) pa = fmaf(bw, sB[r][k2a], pa);
                if (k2b < K) pb = fmaf(bw, sB[r][k2b], pb);
            }
            acc_a += pa;
            acc_b += pb;
        }
    }
    if (k1 < K) {
        if (k2a < K) G[((size_t)j * K + k1) * K + k2a] = acc_a;
        if (k2b < K) G[((size_t)j * K + k1) * K + k2b] = acc_b;
    }
}

// Cinv_j = ((2F)^{-1} + G_j)^{-1} in FP64 (Gauss-Jordan, positive definite, so without pivoting; each step
// from one buffer into the other, one barrier a step), rounded to FP32. blockIdx.y: bit 0 the BF16 B, bit
// 1 the capacitance of the x-update when the factor exposures are split off with the same
// penalty, whose diagonal term is (2 f_k + rho_j)^{-1}. A block per inverse, all 4 x 33 in one launch:
// bound by the FP64 rate, K^3 / 2 cycles each. (Four launches of one 64-thread Cholesky per inverse, a
// thread per column of it, took 0.6 of the 1.4 ms of a 2,000 x 32 universe.)
struct CinvArgs {
    const double* G;                       // 2 x NRHO x K x K
    const double* f;
    int K;
    float* out[4];
    float* G_out[2];                       // FP32 copies of the Gram matrices
};

__global__ void __launch_bounds__(256) k_cinv(CinvArgs A) {
    extern __shared__ double cinv_smem[];
    const int K = A.K, ld = K + 1, j = blockIdx.x, which = blockIdx.y, t = threadIdx.x;
    const int lane = t & 31, warp = t >> 5, NW = blockDim.x >> 5;
    double *from = cinv_smem, *to = cinv_smem + K * ld;
    const double* G = A.G + ((size_t)(which & 1) * NRHO + j) * K * K;
    const double rho = RHO_MIN * pow(10.0, double(j) / RHO_PER_DECADE);
    for (int e = t; e < K * K; e += blockDim.x) {
        const int r = e / K, c = e - r * K;
        double v = G[e];
        if (which < 2) A.G_out[which][(size_t)j * K * K + e] = float(v);
        if (r == c) v += (which & 2) ? 1.0 / (2.0 * A.f[r] + rho) : 1.0 / (2.0 * A.f[r]);
        from[r * ld + c] = v;
    }
    __syncthreads();
    for (int k = 0; k < K; ++k) {
        const double ip = 1.0 / from[k * ld + k];
        for (int r = warp; r < K; r += NW) {
            const double m = -from[r * ld + k] * ip;
            for (int c = lane; c < K; c += 32) {
                const double p = from[k * ld + c];
                double q = (r == k) ? p * ip : fma(m, p, from[r * ld + c]);
                if (c == k) q = (r == k) ? ip : m;
                to[r * ld + c] = q;
            }
        }
        __syncthreads();
        double* x = from; from = to; to = x;
    }
    float* out = A.out[which] + (size_t)j * K * K;
    for (int e = t; e < K * K; e += blockDim.x) {
        const int r = e / K, c = e - r * K;
        out[e] = float(from[r * ld + c]);
    }
}

// The copies of B in sorted order from the caller's (a warp per position; padding rows are zero), and
// sum_k |B_ik|. A non-finite entry sets *bad.
struct ConvArgs {
    const double* raw;                     // N x K, the caller's order
    const int* perm;                       // sorted position -> asset
    int N, Npad, K;
    double* B64;
    float *B32, *B32p;
    __nv_bfloat16 *B16, *Bt16, *B16p, *Bt16p;
    double* Bn1;
    float* Bn1f;
    int* bad;
};

__global__ void k_convert_B(ConvArgs A) {
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (p >= A.Npad) return;
    const int K = A.K;
    const double* row = p < A.N ? A.raw + (size_t)A.perm[p] * K : nullptr;
    double n1 = 0.0;
    for (int k = lane; k < KMAX; k += 32) {
        const double b = (row && k < K) ? row[k] : 0.0;
        const float f = float(b);
        const __nv_bfloat16 h = __float2bfloat16_rn(f);
        if (!isfinite(b)) *A.bad = 1;
        n1 += fabs(b);
        if (k < K) {
            A.B64[(size_t)p * K + k] = b;
            A.B32[(size_t)p * K + k] = f;
            A.B16[(size_t)p * K + k] = h;
            A.Bt16[(size_t)k * A.Npad + p] = h;
        }
        A.B32p[(size_t)p * KMAX + k] = f;
        A.B16p[(size_t)p * KMAX + k] = h;
        A.Bt16p[(size_t)k * A.Npad + p] = h;
    }
    n1 = warp_sum(n1);
    if (lane == 0) { A.Bn1[p] = n1; A.Bn1f[p] = float(n1); }
}

static bool is_device_ptr(const void* p) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

// Whether a kernel on device `dev` may read p where it is.
static bool on_device(const void* p, int dev) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return attr.type == cudaMemoryTypeManaged || (attr.type == cudaMemoryTypeDevice && attr.device == dev);
}

// Copy n elements of T from a host or device pointer to a host vector.
template <typename T>
static int fetch(const T* src, size_t n, std::vector<T>& dst) {
    dst.resize(n);
    if (n == 0) return PRISM_OK;
    if (is_device_ptr(src)) {
        PRISM_CUDA_TRY(cudaMemcpy(dst.data(), src, n * sizeof(T), cudaMemcpyDeviceToHost));
    } else {
        std::memcpy(dst.data(), src, n * sizeof(T));
    }
    return PRISM_OK;
}

static void free_universe(Universe& U) {
    if (U.d_block) cudaFree(U.d_block);
    if (U.stream) cudaStreamDestroy(U.stream);
    U = Universe();
}

static int create(const prism_universe_desc* desc, Universe& U) {
    if (!desc) { set_error("desc is NULL"); return PRISM_ERR_ARGUMENT; }
    const int N = desc->n_assets, K = desc->n_factors, S = desc->n_sectors;
    if (N < 1 || K < 1 || K > KMAX || S < 1 || S > SMAX) {
        set_error("universe sizes out of range (N >= 1, 1 <= K <= 64, 1 <= S <= 64)");
        return PRISM_ERR_ARGUMENT;
    }
    if (!desc->B || !desc->f || !desc->d || !desc->mu || !desc->sector) {
        set_error("universe array is NULL");
        return PRISM_ERR_ARGUMENT;
    }
    int ndev = 0;
    PRISM_CUDA_TRY(cudaGetDeviceCount(&ndev));
    if (desc->device < 0 || desc->device >= ndev) {
        set_error("device ordinal out of range");
        return PRISM_ERR_ARGUMENT;
    }
    PRISM_CUDA_TRY(cudaSetDevice(desc->device));
    std::vector<double> f, d, mu;
    std::vector<int32_t> sec;
    int rc;
    if ((rc = fetch(desc->f, K, f)) || (rc = fetch(desc->d, N, d)) || (rc = fetch(desc->mu, N, mu)) ||
        (rc = fetch(desc->sector, N, sec)))
        return rc;
    for (int k = 0; k < K; ++k)
        if (!(f[k] > 0) || !std::isfinite(f[k])) { set_error("f must be positive and finite"); return PRISM_ERR_ARGUMENT; }
    for (int i = 0; i < N; ++i) {
        if (!(d[i] > 0) || !std::isfinite(d[i])) { set_error("d must be positive and finite"); return PRISM_ERR_ARGUMENT; }
        if (!std::isfinite(mu[i])) { set_error("mu has a non-finite entry"); return PRISM_ERR_ARGUMENT; }
        if (sec[i] < 0 || sec[i] >= S) { set_error("sector id out of range"); return PRISM_ERR_ARGUMENT; }
    }
    U.device = desc->device;
    U.N = N; U.K = K; U.S = S;
    U.dmin = *std::min_element(d.begin(), d.end());
    U.Npad = (N + 63) / 64 * 64;
    const int Npad = U.Npad;
    // stable sort of assets by sector
    U.perm.resize(N);
    std::iota(U.perm.begin(), U.perm.end(), 0);
    std::stable_sort(U.perm.begin(), U.perm.end(), [&](int a, int b) { return sec[a] < sec[b]; });
    U.inv_perm.resize(N);
    for (int p = 0; p < N; ++p) U.inv_perm[U.perm[p]] = p;
    U.sec_start.assign(S + 1, 0);
    for (int i = 0; i < N; ++i) U.sec_start[sec[i] + 1]++;
    for (int s = 0; s < S; ++s) U.sec_start[s + 1] += U.sec_start[s];
    std::vector<double> ds(Npad, 1.0), mus(Npad, 0.0);
    std::vector<int> secs(Npad, -1);
    for (int p = 0; p < N; ++p) {
        int i = U.perm[p];
        ds[p] = d[i];
        mus[p] = mu[i];
        secs[p] = sec[i];
    }
    std::vector<float> f32(f.begin(), f.end()), d32(ds.begin(), ds.end()), mu32(mus.begin(), mus.end());
    // quarter / sector segments (sorted positions: sector ids are nondecreasing in p)
    U.nq = Npad / 32;
    std::vector<int> qseg(U.nq + 1, 0), sseg(S + 1, 0);
    for (int q = 0; q < U.nq; ++q) {
        int n = 0;
        for (int p = 32 * q; p < std::min(32 * q + 32, N); ++p)
            if (p == 32 * q || secs[p] != secs[p - 1]) { ++n; ++sseg[secs[p] + 1]; }
        qseg[q + 1] = qseg[q] + n;
    }
    for (int s = 0; s < S; ++s) sseg[s + 1] += sseg[s];
    U.nseg = qseg[U.nq];
    cudaError_t se = cudaStreamCreateWithFlags(&U.stream, cudaStreamNonBlocking);
    if (se != cudaSuccess) { set_error(cudaGetErrorString(se)); return PRISM_ERR_CUDA; }
    // One device block: what the host fills first (uploaded in one copy), then what the kernels fill. (27 allocations and 15 copies cost 0.5 ms here and their frees as much again.)
    std::vector<char> image;
    size_t off = 0;
    std::vector<std::pair<void**, size_t>> at;
    auto place = [&](auto** p, size_t n) {
        at.push_back({(void**)p, off});
        off += (n * sizeof(**p) + 255) / 256 * 256;
    };
    auto upload = [&](auto** p, const auto* src, size_t n) {
        const size_t o = off;
        place(p, n);
        image.resize(off);
        std::memcpy(image.data() + o, src, n * sizeof(**p));
    };
    int* d_bad = nullptr;
    const int zero = 0;
    upload(&U.d_inv_perm, U.inv_perm.data(), N);
    upload(&U.d_perm, U.perm.data(), N);
    upload(&U.d_sec_start, U.sec_start.data(), S + 1);
    upload(&U.d_sector, secs.data(), Npad);
    upload(&U.d_qseg, qseg.data(), U.nq + 1);
    upload(&U.d_sseg, sseg.data(), S + 1);
    upload(&U.d_f64, f.data(), K);
    upload(&U.d_d64, ds.data(), Npad);
    upload(&U.d_mu64, mus.data(), Npad);
    upload(&U.d_f32, f32.data(), K);
    upload(&U.d_d32, d32.data(), Npad);
    upload(&U.d_mu32, mu32.data(), Npad);
    upload(&d_bad, &zero, 1);
    place(&U.d_B64, (size_t)Npad * K);
    place(&U.d_Bn1, Npad);
    place(&U.d_Bn1f, Npad);
    place(&U.d_B32, (size_t)Npad * K);
    place(&U.d_B32p, (size_t)Npad * KMAX);
    place(&U.d_B16, (size_t)Npad * K);
    place(&U.d_Bt16, (size_t)K * Npad);
    place(&U.d_B16p, (size_t)Npad * KMAX);
    place(&U.d_Bt16p, (size_t)KMAX * Npad);
    place(&U.d_Cinv32, (size_t)NRHO * K * K);
    place(&U.d_Cinv16, (size_t)NRHO * K * K);
    place(&U.d_G32, (size_t)NRHO * K * K);
    place(&U.d_G16, (size_t)NRHO * K * K);
    place(&U.d_CinvF32, (size_t)NRHO * K * K);
    place(&U.d_CinvF16, (size_t)NRHO * K * K);
    // what only the setup needs: the Gram matrices, and B in the caller's order unless it is there already
    const bool here = on_device(desc->B, desc->device);
    struct Scratch {
        double* p = nullptr;
        ~Scratch() { if (p) cudaFree(p); }
    } scratch;
    const size_t nG = 2 * (size_t)NRHO * K * K;
    if (cudaMalloc((void**)&U.d_block, off) != cudaSuccess ||
        cudaMalloc((void**)&scratch.p, (nG + (here ? 0 : (size_t)N * K)) * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc (universe) failed");
        free_universe(U);
        return PRISM_ERR_ALLOCATION;
    }
    double *const G = scratch.p, *const raw = scratch.p + nG;
    U.bytes = off;
    for (auto& q : at) *q.first = U.d_block + q.second;
    // (the default stream's copies order the upload behind what the caller queued there; they return
    // once the host memory may be reused, and the kernels' stream is told to follow them)
    if (cudaMemcpy(U.d_block, image.data(), image.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        (!here && cudaMemcpy(raw, desc->B, (size_t)N * K * sizeof(double), cudaMemcpyDefault) != cudaSuccess) ||
        cudaStreamSynchronize(0) != cudaSuccess) {
        cudaGetLastError();
        set_error("universe upload failed");
        free_universe(U);
        return PRISM_ERR_CUDA;
    }
    ConvArgs CA;
    CA.raw = here ? desc->B : raw;
    CA.perm = U.d_perm; CA.N = N; CA.Npad = Npad; CA.K = K;
    CA.B64 = U.d_B64; CA.B32 = U.d_B32; CA.B32p = U.d_B32p;
    CA.B16 = U.d_B16; CA.Bt16 = U.d_Bt16; CA.B16p = U.d_B16p; CA.Bt16p = U.d_Bt16p;
    CA.Bn1 = U.d_Bn1; CA.Bn1f = U.d_Bn1f; CA.bad = d_bad;
    k_convert_B<<<(unsigned)cdiv64((int64_t)Npad * 32, 256), 256, 0, U.stream>>>(CA);
    k_gram<<<dim3(NRHO, cdiv(K, 8), 2), 256, 0, U.stream>>>(U.d_B32, U.d_B16, U.d_d32, N, K, G);
    CinvArgs IA;
    IA.G = G; IA.f = U.d_f64; IA.K = K;
    IA.out[0] = U.d_Cinv32; IA.out[1] = U.d_Cinv16; IA.out[2] = U.d_CinvF32; IA.out[3] = U.d_CinvF16;
    IA.G_out[0] = U.d_G32; IA.G_out[1] = U.d_G16;
    const int smem = 2 * K * (K + 1) * (int)sizeof(double);
    // (the limit belongs to the process: every thread sets the same one, whatever its K)
    cudaFuncSetAttribute(k_cinv, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * KMAX * (KMAX + 1) * (int)sizeof(double));
    k_cinv<<<dim3(NRHO, 4), 256, smem, U.stream>>>(IA);
    int bad = 0;
    cudaError_t e = cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, U.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(U.stream);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error(std::string("universe setup kernels failed: ") + cudaGetErrorString(e));
        free_universe(U);
        return PRISM_ERR_CUDA;
    }
    if (bad) {
        set_error("B has a non-finite entry");
        free_universe(U);
        return PRISM_ERR_ARGUMENT;
    }
    return PRISM_OK;
}

}  // namespace prism

extern "C" int prism_create_universe(const prism_universe_desc* desc, prism_universe** out) {
    if (!out) { prism::set_error("out is NULL"); return PRISM_ERR_ARGUMENT; }
    *out = nullptr;
    prism_universe* h = new (std::nothrow) prism_universe();
    if (!h) { prism::set_error("host allocation failed"); return PRISM_ERR_ALLOCATION; }
    int rc = prism::create(desc, h->u);
    if (rc != PRISM_OK) { delete h; return rc; }
    *out = h;
    prism::set_error("");
    return PRISM_OK;
}

extern "C" void prism_destroy_universe(prism_universe* u) {
    if (!u) return;
    cudaSetDevice(u->u.device);
    prism::free_universe(u->u);
    delete u;
}

extern "C" const char* prism_last_error(void) { return prism::last_error(); }
extern "C" const char* prism_version(void) { return "prism-gb300 0.1 (sm_103a)"; }
