// MBAR free energies of the states of one window segment (Shirts & Chodera
// 2008), the estimator the paper applies within each GPU segment before summing
// the segments ("Simulation protocol").
//
// The dimensionless free energies solve
//     f_i = -ln sum_n exp(-u_in) / sum_k N_k exp(f_k - u_kn),   f_0 = 0,
// for the K x N matrix of reduced potentials u_kn, by self-consistent
// iteration in FP64 with every iteration on the device. One iteration applies
// the map above once, in one of two exact arrangements:
//  A (log space): ld_n = ln sum_k exp(ln N_k + f_k - u_kn) per sample, then per
//    state f_i = -ln sum_n exp(-u_in - ld_n); 2 K N exponentials.
//  B (scaled linear): with a reference f^r and the stored matrix
//    c_kn = exp(f^r_k - u_kn - b_n), b_n = max over sampled k of f^r_k - u_kn,
//    D_n = sum_k N_k exp(f_k - f^r_k) c_kn and f_i = f^r_i - ln sum_n c_in / D_n:
//    two FP64 multiply-adds per element, no exponential.
// B is the same map (multiply numerator and denominator by exp(-b_n)); c_kn
// lies in [0, 1] with a 1 for the largest sampled term of every sample, so D_n
// cannot underflow while |f - f^r| stays moderate. The loop starts with c at f = 0
// and runs B, refreshing c whenever f drifts more than 20 from f^r; an iteration
// that moved f by more than 40 from f^r, or whose sums are not finite, is done
// again in A. Terms c_kn below 2^-160 are stored as zeros: against sums of at
// least exp(-40) even 10^12 of them stay below the last bit.
// The state machine lives in device memory: a pass is k_mbar_main (A's ld_n, a
// refresh, or all of B), k_mbar_part (A's second half) and k_mbar_reduce, each
// returning at once when it is not its turn, and the graph's while-node body holds
// four passes (a conditional node costs 6 us), so there are no host round trips.
// The log-sum-exps take the maximum first and skip terms more than 60 below it
// (relative weight < 1e-26). Reductions have a fixed order: deterministic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include "abfe.h"
#include "abfe_internal.cuh"

namespace {

constexpr int MB_THREADS = 256;
constexpr int MB_CHUNK = 16384;        // samples per partial of k_mbar_part
constexpr double MB_SKIP = -60.0;      // exp(x - max) not evaluated below this
constexpr double MB_ZERO = -110.9;     // ln 2^-160: smaller c_kn are zero
constexpr int MB_SMEM_MAX = 160 * 1024;  // dynamic shared memory of k_mbar_main, any K
constexpr int MB_PASSES = 4;           // passes in the body of the graph's while node

enum : int { MODE_A = 0, MODE_REFRESH = 1, MODE_B = 2 };
constexpr double MB_DRIFT = 20.0;      // refresh c when max |f - f^r| exceeds this
constexpr double MB_REDO = 40.0;       // redo the iteration in A when it exceeds this

struct MbarDev {
    const double* u;       // [K][N]
    double* c;             // [K][N] scaled weights of arrangement B
    long long N;
    int K, nch;
    int nb, tn;            // blocks of arrangement B, samples per tile
    const double* logN;    // [K] ln N_k (-inf for N_k = 0)
    double* lognf;         // [K] ln N_k + f_k
    double* f;             // [K]
    double* fr;            // [K] reference f of c
    double* fn;            // [K] f of the iteration, before normalisation
    double* ld;            // [N] ld_n (A)
    double2* part;         // [K][nch] (max, sum) (A)
    double* bpart;         // [K][nb] (B)
    int* iter;             // iterations done
    int* status;           // bit 0 converged, bit 1 non-finite
    int* mode;             // MODE_*
    int* stop;             // 1: converged, failed or max_iter reached
    int* done;             // blocks of k_mbar_reduce that have finished
    double tol;
    int max_iter;
};

__device__ __forceinline__ double block_max(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = sh[0];
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) t = fmax(t, sh[i]);
    return t;  // all threads
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sh[i];
    return t;  // all threads
}

// A, first half: ld_n for every sample (thread per sample; u rows read coalesced)
__device__ void mbar_ld(const MbarDev& M, double* s_lognf) {
    for (int k = threadIdx.x; k < M.K; k += blockDim.x) s_lognf[k] = M.lognf[k];
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < M.N; n += stride) {
        double m = -INFINITY;
        for (int k = 0; k < M.K; ++k) {
            const double a = s_lognf[k];
            if (a > -INFINITY) m = fmax(m, a - M.u[(long long)k * M.N + n]);
        }
        double s = 0.0;
        for (int k = 0; k < M.K; ++k) {
            const double a = s_lognf[k];
            if (a > -INFINITY) {
                const double x = a - M.u[(long long)k * M.N + n] - m;
                if (x > MB_SKIP) s += exp(x);
            }
        }
        const double v = m + log(s);
        M.ld[n] = v;
        if (!isfinite(v)) atomicOr(M.status, 2);
    }
}

// c_kn = exp(f_k - u_kn - b_n) at the current f, which becomes the reference
__device__ void mbar_refresh(const MbarDev& M, double* s_f) {   // [K] f, [K] 1 if sampled
    for (int k = threadIdx.x; k < M.K; k += blockDim.x) {
        s_f[k] = M.f[k];
        s_f[M.K + k] = M.logN[k] > -INFINITY ? 1.0 : 0.0;
    }
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < M.N; n += stride) {
        double b = -INFINITY;
        for (int k = 0; k < M.K; ++k)
            if (s_f[M.K + k] != 0.0) b = fmax(b, s_f[k] - M.u[(long long)k * M.N + n]);
        for (int k = 0; k < M.K; ++k) {
            const double x = s_f[k] - M.u[(long long)k * M.N + n] - b;
            M.c[(long long)k * M.N + n] = x > MB_ZERO ? exp(x) : 0.0;
        }
    }
}

// B: D_n and the partial sums over the block's samples of c_in / D_n, in tiles of
// tn samples that are read once and held in shared memory ([K][tn + 1]: the odd
// stride keeps both directions free of bank conflicts). First half: thread per
// sample (256 / tn threads each take a share of the states); second half: thread
// per state (256 / K threads each take a share of the samples), the sums in
// registers over all tiles. Bound by the FP64 pipe (63 issue cycles per warp
// multiply-add, 1/64 of FP32's rate; 75% active, measured): a group of
// multiply-adds whose elements are all zero is skipped (tested as integers: an
// FP64 compare takes the same pipe). 80 states x 160,000 samples: 126 us per
// iteration with two passes over c in kernels of their own, 86 now, 73 of them
// here (42 for the multiply-adds alone at that rate). Two blocks per SM: three,
// four, six and eight with smaller tiles took 91, 94, 113 and 118 us.
constexpr int MB_SUMS = 4;   // states per thread (ABFE_MBAR_MAX_K / MB_THREADS)
static_assert(ABFE_MBAR_MAX_K <= MB_SUMS * MB_THREADS, "k_mbar_main keeps MB_SUMS sums per thread");
__device__ void mbar_linear(const MbarDev& M, double* sm) {
    const int K = M.K, tn = M.tn, ls = tn + 1;
    double* const s_c = sm;                       // [K][ls]
    double* const s_w = sm + (size_t)K * ls;      // [K]
    double* const s_d = s_w + K;                  // [256]
    const int tid = threadIdx.x;
    for (int k = tid; k < K; k += MB_THREADS)
        s_w[k] = M.logN[k] > -INFINITY ? exp(M.logN[k] + M.f[k] - M.fr[k]) : 0.0;
    const long long n0 = M.N * blockIdx.x / M.nb, n1 = M.N * (blockIdx.x + 1) / M.nb;
    const int g1 = MB_THREADS / tn, n_of = tid % tn, g_of = tid / tn;
    const int seg = K < MB_THREADS ? MB_THREADS / K : 1;
    const int i_of = K < MB_THREADS ? tid % K : tid, s_of = K < MB_THREADS ? tid / K : 0;
    double sum[MB_SUMS] = {0.0, 0.0, 0.0, 0.0};
    for (long long t0 = n0; t0 < n1; t0 += tn) {
        const int cnt = (int)(n1 - t0 < tn ? n1 - t0 : tn);
        __syncthreads();   // the last tile's second half is over
        // (asynchronous copies: every load of the tile is in flight at once)
        for (int k = g_of; k < K; k += g1) {
            const unsigned int dst = (unsigned int)__cvta_generic_to_shared(s_c + k * ls + n_of);
            const double* src = M.c + (long long)k * M.N + t0 + (n_of < cnt ? n_of : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src),
                         "r"(n_of < cnt ? 8 : 0) : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        double d[4] = {0.0, 0.0, 0.0, 0.0};
        if (tn < 32 || __any_sync(0xffffffffu, n_of < cnt)) {
            for (int k = g_of; k < K; k += 4 * g1) {
                double v[4], w[4];
                bool nz = false;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int kq = k + q * g1;
                    v[q] = kq < K ? s_c[kq * ls + n_of] : 0.0;
                    w[q] = kq < K ? s_w[kq] : 0.0;
                    nz |= __double_as_longlong(v[q]) != 0ll;
                }
                // (below 32 samples per tile a warp's threads take different states)
                if (tn < 32 ? nz : __any_sync(0xffffffffu, nz)) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) d[q] = fma(w[q], v[q], d[q]);
                }
            }
        }
        s_d[tid] = (d[0] + d[1]) + (d[2] + d[3]);
        __syncthreads();
        double inv = 0.0;   // (samples beyond the block's: their c are zeros)
        if (tid < cnt) {
            double t = 0.0;
            for (int g = 0; g < g1; ++g) t += s_d[g * tn + tid];
            inv = 1.0 / t;
        }
        __syncthreads();
        if (tid < tn) s_d[tid] = inv;
        __syncthreads();
        // the longest segment's trip count and whole warps for all lanes (segments change
        // within a warp and some lanes have none), so that the votes take full warps
        const int m0 = cnt * s_of / seg, m1 = cnt * (s_of + 1) / seg, len = (cnt + seg - 1) / seg;
#pragma unroll
        for (int q = 0; q < MB_SUMS; ++q) {
            if (q * MB_THREADS >= K) break;
            const int i = i_of + q * MB_THREADS;
            const int end = s_of < seg && i < K ? m1 : 0;
            const double* row = s_c + (size_t)i * ls;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            for (int m = m0; m < m0 + len; m += 4) {
                double v[4], r[4];
                bool nz = false;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const bool on = m + p < end;
                    v[p] = on ? row[m + p] : 0.0;
                    r[p] = on ? s_d[m + p] : 0.0;
                    nz |= __double_as_longlong(v[p]) != 0ll;
                }
                if (__any_sync(0xffffffffu, nz)) {
#pragma unroll
                    for (int p = 0; p < 4; ++p) s[p] = fma(v[p], r[p], s[p]);
                }
            }
            sum[q] += (s[0] + s[1]) + (s[2] + s[3]);
        }
    }
    // the segments of a state, in order
    __syncthreads();
    if (seg > 1) {
        s_d[tid] = sum[0];
        __syncthreads();
        if (tid < K) {
            double s = 0.0;
            for (int g = 0; g < seg; ++g) s += s_d[g * K + tid];
            M.bpart[(long long)tid * M.nb + blockIdx.x] = s;
        }
    } else {
        for (int q = 0; q < MB_SUMS; ++q) {
            const int i = tid + q * MB_THREADS;
            if (i < K) M.bpart[(long long)i * M.nb + blockIdx.x] = sum[q];
        }
    }
}

__global__ void __launch_bounds__(MB_THREADS) k_mbar_main(MbarDev M) {
    extern __shared__ double sm[];
    if (*M.stop) return;
    switch (*M.mode) {
        case MODE_A: mbar_ld(M, sm); break;
        case MODE_REFRESH: mbar_refresh(M, sm); break;
        default: mbar_linear(M, sm); break;
    }
}

// A, second half: partial log-sum-exp of -u_in - ld_n over one chunk of samples,
// per state i
__global__ void __launch_bounds__(MB_THREADS) k_mbar_part(MbarDev M) {
    if (*M.stop || *M.mode != MODE_A) return;
    __shared__ double sh[MB_THREADS / 32];
    const int i = blockIdx.y, j = blockIdx.x;
    const long long n0 = (long long)j * MB_CHUNK;
    const long long n1 = n0 + MB_CHUNK < M.N ? n0 + MB_CHUNK : M.N;
    const double* ui = M.u + (long long)i * M.N;
    double m = -INFINITY;
    for (long long n = n0 + threadIdx.x; n < n1; n += blockDim.x) m = fmax(m, -ui[n] - M.ld[n]);
    m = block_max(m, sh);
    double s = 0.0;
    for (long long n = n0 + threadIdx.x; n < n1; n += blockDim.x) {
        const double x = -ui[n] - M.ld[n] - m;
        if (x > MB_SKIP) s += exp(x);
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) M.part[(long long)i * M.nch + j] = make_double2(m, s);
}

// A block per state combines its partials; the last block to finish normalises,
// tests convergence, chooses the next mode and sets the loop condition.
constexpr int MR_THREADS = 128;
__global__ void __launch_bounds__(MR_THREADS) k_mbar_reduce(MbarDev M, cudaGraphConditionalHandle h,
                                                            int use_handle) {
    __shared__ double sh[MR_THREADS / 32];
    __shared__ int s_last;
    if (*M.stop) return;   // (the while condition was cleared with the flag)
    const int mode = *M.mode, i = blockIdx.x;
    if (mode == MODE_A) {
        if (threadIdx.x == 0) {
            const double2* p = M.part + (long long)i * M.nch;
            double mx = -INFINITY;
            for (int j = 0; j < M.nch; ++j) mx = fmax(mx, p[j].x);
            double s = 0.0;
            for (int j = 0; j < M.nch; ++j) s += p[j].y * exp(p[j].x - mx);
            M.fn[i] = -(mx + log(s));
        }
    } else if (mode == MODE_B) {
        double s = 0.0;
        for (int b = threadIdx.x; b < M.nb; b += MR_THREADS) s += M.bpart[(long long)i * M.nb + b];
        s = block_sum(s, sh);
        if (threadIdx.x == 0) M.fn[i] = M.fr[i] - log(s);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(M.done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) *M.done = 0;
    if (mode == MODE_REFRESH) {
        for (int k = threadIdx.x; k < M.K; k += MR_THREADS) M.fr[k] = M.f[k];
        if (threadIdx.x == 0) *M.mode = MODE_B;
        return;
    }
    const double f0 = __ldcg(&M.fn[0]);
    double d = 0.0, drift = 0.0;
    bool bad = false;
    for (int k = threadIdx.x; k < M.K; k += MR_THREADS) {
        const double fk = __ldcg(&M.fn[k]) - f0;
        if (!isfinite(fk)) bad = true;
        d = fmax(d, fabs(fk - M.f[k]));
        if (mode == MODE_B) drift = fmax(drift, fabs(fk - M.fr[k]));
    }
    const int bad_any = __syncthreads_or(bad);
    d = block_max(bad_any ? INFINITY : d, sh);
    drift = block_max(drift, sh);
    if (mode == MODE_B && (bad_any || drift > MB_REDO)) {
        // the sums left the range of arrangement B: redo this iteration in log space
        if (threadIdx.x == 0) *M.mode = MODE_A;
        return;
    }
    for (int k = threadIdx.x; k < M.K; k += MR_THREADS) {
        const double fk = __ldcg(&M.fn[k]) - f0;
        M.f[k] = fk;
        M.lognf[k] = M.logN[k] > -INFINITY ? M.logN[k] + fk : -INFINITY;
    }
    if (threadIdx.x == 0) {
        const int it = *M.iter + 1;
        *M.iter = it;
        int st = *M.status;
        if (bad_any) st |= 2;
        if (d < M.tol) st |= 1;
        *M.status = st;
        if (mode == MODE_A || drift > MB_DRIFT) *M.mode = MODE_REFRESH;
        if ((st & 3) || it >= M.max_iter) {
            *M.stop = 1;
            if (use_handle) cudaGraphSetConditional(h, 0u);
        }
    }
}

// non-finite inputs would otherwise drop out of the max-first sums unnoticed
__global__ void k_mbar_check(MbarDev M) {
    const long long total = (long long)M.K * M.N;
    const long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride)
        bad |= !isfinite(M.u[t]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(M.status, 2);
}

__global__ void k_mbar_init(MbarDev M) {
    for (int i = threadIdx.x; i < M.K; i += blockDim.x) {
        M.f[i] = 0.0;
        M.lognf[i] = M.logN[i];
    }
    if (threadIdx.x == 0) {
        *M.iter = 0;
        *M.status = 0;
        *M.mode = MODE_REFRESH;
        *M.stop = 0;
        *M.done = 0;
    }
}

struct Scratch {
    std::vector<std::pair<void*, size_t>> a;
    cudaStream_t s;
    bool ok = true;
    template <class T>
    T* get(size_t n) {
        const size_t b = n * sizeof(T);
        void* p = abfe::lib_alloc(b, s);
        if (!p) ok = false;
        a.push_back({p, b});
        return (T*)p;
    }
    ~Scratch() {
        cudaStreamSynchronize(s);
        for (auto& x : a) abfe::lib_free(x.first, x.second, s);
    }
};

cudaStream_t mbar_stream() {
    // one stream for every call, so that allocator pools tied to a stream are reused
    static std::once_flag once;
    static cudaStream_t s = nullptr;
    std::call_once(once, [] {
        if (cudaStreamCreate(&s) != cudaSuccess) {
            cudaGetLastError();
            s = nullptr;
        }
    });
    return s;
}

abfe_status fail(abfe_status st, const std::string& m) {
    abfe::set_free_error(m.c_str());
    return st;
}

// samples per tile and dynamic shared memory of k_mbar_main: the widest tile that
// leaves room for two blocks per SM
int mbar_tile(int K) {
    int tn = 256;
    while (tn > 16 && (size_t)K * (tn + 1) * sizeof(double) > 100 * 1024) tn /= 2;
    return tn;
}
size_t mbar_smem(int K, int tn) {
    return sizeof(double) * ((size_t)K * (tn + 1) + K + MB_THREADS);
}

void enqueue_pass(const MbarDev& M, cudaStream_t s, cudaGraphConditionalHandle h, int use_handle) {
    k_mbar_main<<<M.nb, MB_THREADS, mbar_smem(M.K, M.tn), s>>>(M);
    k_mbar_part<<<dim3(M.nch, M.K), MB_THREADS, 0, s>>>(M);
    k_mbar_reduce<<<M.K, MR_THREADS, 0, s>>>(M, h, use_handle);
}

abfe_status mbar_run(const double* u_src, bool u_host, const int32_t* N_k, int32_t K, int64_t N,
                     double tol, int32_t max_iter, double* f_out, int32_t* n_iter,
                     cudaStream_t caller) {
    if (!u_src || !N_k || !f_out) return fail(ABFE_ERR_INVALID_ARG, "mbar: NULL pointer");
    if (K < 1 || K > ABFE_MBAR_MAX_K || N < 1 || !(tol > 0.0) || max_iter < 1)
        return fail(ABFE_ERR_INVALID_ARG,
                    "mbar: need 1 <= K <= ABFE_MBAR_MAX_K, N >= 1, tol > 0, max_iter >= 1");
    int64_t tot = 0;
    std::vector<double> logN(K);
    for (int k = 0; k < K; ++k) {
        if (N_k[k] < 0) return fail(ABFE_ERR_INVALID_ARG, "mbar: negative N_k");
        tot += N_k[k];
        logN[k] = N_k[k] > 0 ? std::log((double)N_k[k]) : -INFINITY;
    }
    if (tot != N) return fail(ABFE_ERR_INVALID_ARG, "mbar: sum of N_k differs from N");
    cudaStream_t s = mbar_stream();
    if (!s) return fail(ABFE_ERR_CUDA, "mbar: stream creation failed");
    cudaEvent_t ev = nullptr;
    if (caller) {
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventRecord(ev, caller) != cudaSuccess || cudaStreamWaitEvent(s, ev, 0) != cudaSuccess) {
            if (ev) cudaEventDestroy(ev);
            cudaGetLastError();
            return fail(ABFE_ERR_CUDA, "mbar: cannot order after the caller's stream");
        }
    }
    MbarDev M{};
    M.N = N;
    M.K = K;
    M.nch = (int)((N + MB_CHUNK - 1) / MB_CHUNK);
    M.tol = tol;
    M.max_iter = max_iter;
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    M.nb = (int)std::min<int64_t>(2 * (int64_t)n_sm, (N + 31) / 32);
    M.tn = mbar_tile(K);
    // (the attribute belongs to the kernel: set to what any K needs)
    static_assert(8 * (ABFE_MBAR_MAX_K * 17 + ABFE_MBAR_MAX_K + MB_THREADS) <= MB_SMEM_MAX, "");
    if (mbar_smem(K, M.tn) > MB_SMEM_MAX ||
        cudaFuncSetAttribute(k_mbar_main, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             MB_SMEM_MAX) != cudaSuccess) {
        if (ev) cudaEventDestroy(ev);
        cudaGetLastError();
        return fail(ABFE_ERR_CUDA, "mbar: shared memory");
    }
    Scratch sc;
    sc.s = s;
    double* d_u = u_host ? sc.get<double>((size_t)K * N) : nullptr;
    double* d_logN = sc.get<double>(K);
    M.lognf = sc.get<double>(K);
    M.f = sc.get<double>(K);
    M.fr = sc.get<double>(K);
    M.fn = sc.get<double>(K);
    M.bpart = sc.get<double>((size_t)K * M.nb);
    M.c = sc.get<double>((size_t)K * N);
    M.ld = sc.get<double>(N);
    M.part = sc.get<double2>((size_t)K * M.nch);
    int* d_ints = sc.get<int>(5);
    if (ev) cudaEventDestroy(ev);
    if (!sc.ok) return fail(ABFE_ERR_OUT_OF_MEMORY, "mbar: device scratch");
    M.iter = d_ints;
    M.status = d_ints + 1;
    M.mode = d_ints + 2;
    M.stop = d_ints + 3;
    M.done = d_ints + 4;
    M.logN = d_logN;
    if (u_host) {
        if (cudaMemcpyAsync(d_u, u_src, sizeof(double) * (size_t)K * N, cudaMemcpyHostToDevice, s) !=
            cudaSuccess)
            return fail(ABFE_ERR_CUDA, "mbar: copy of u_kn");
        M.u = d_u;
    } else {
        M.u = u_src;
    }
    if (cudaMemcpyAsync(d_logN, logN.data(), sizeof(double) * K, cudaMemcpyHostToDevice, s) !=
        cudaSuccess)
        return fail(ABFE_ERR_CUDA, "mbar: copy of ln N_k");
    k_mbar_init<<<1, 1024, 0, s>>>(M);
    k_mbar_check<<<n_sm * 4, MB_THREADS, 0, s>>>(M);
    {
        int h_st = 0;
        if (cudaMemcpyAsync(&h_st, M.status, sizeof h_st, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return fail(ABFE_ERR_CUDA, "mbar: input check");
        if (h_st & 2) return fail(ABFE_ERR_NONFINITE, "mbar: non-finite u_kn");
    }

    // the whole iteration as one graph: while (condition) { passes }
    bool graph_done = false;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t gx = nullptr;
    if (cudaGraphCreate(&g, 0) == cudaSuccess) {
        cudaGraphConditionalHandle h;
        cudaGraphNodeParams np = {};
        cudaGraphNode_t node;
        if (cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) == cudaSuccess) {
            np.type = cudaGraphNodeTypeConditional;
            np.conditional.handle = h;
            np.conditional.type = cudaGraphCondTypeWhile;
            np.conditional.size = 1;
            if (cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np) == cudaSuccess) {
                cudaGraph_t body = np.conditional.phGraph_out[0];
                cudaStream_t cs = nullptr;
                if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess) {
                    if (cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0,
                                                      cudaStreamCaptureModeRelaxed) == cudaSuccess) {
                        for (int q = 0; q < MB_PASSES; ++q) enqueue_pass(M, cs, h, 1);
                        const bool cap = cudaStreamEndCapture(cs, &body) == cudaSuccess;
                        if (cap && cudaGraphInstantiate(&gx, g, 0) == cudaSuccess &&
                            cudaGraphLaunch(gx, s) == cudaSuccess)
                            graph_done = true;
                    }
                    cudaStreamDestroy(cs);
                }
            }
        }
    }
    if (!graph_done) {
        cudaGetLastError();
        // host-driven fallback: the device still tests convergence; the host looks at
        // its flag every 16 passes
        int h_stop = 0;
        while (!h_stop) {
            for (int b = 0; b < 16; ++b) enqueue_pass(M, s, 0, 0);
            if (cudaMemcpyAsync(&h_stop, M.stop, sizeof h_stop, cudaMemcpyDeviceToHost, s) !=
                    cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                break;
        }
    }
    int h_ints[2] = {0, 0};
    cudaMemcpyAsync(h_ints, d_ints, sizeof h_ints, cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(f_out, M.f, sizeof(double) * K, cudaMemcpyDeviceToHost, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (gx) cudaGraphExecDestroy(gx);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) return fail(ABFE_ERR_CUDA, std::string("mbar: ") + cudaGetErrorString(e));
    if (n_iter) *n_iter = h_ints[0];
    if (h_ints[1] & 2) return fail(ABFE_ERR_NONFINITE, "mbar: non-finite u_kn or free energy");
    return ABFE_OK;
}

}  // namespace

extern "C" {

abfe_status abfe_mbar(const double* h_u_kn, const int32_t* h_N_k, int32_t K, int64_t N,
                      double tol, int32_t max_iter, double* h_f_k, int32_t* h_n_iter) {
    return mbar_run(h_u_kn, true, h_N_k, K, N, tol, max_iter, h_f_k, h_n_iter, nullptr);
}

abfe_status abfe_mbar_device(const double* d_u_kn, const int32_t* h_N_k, int32_t K, int64_t N,
                             double tol, int32_t max_iter, double* h_f_k, int32_t* h_n_iter,
                             void* stream) {
    return mbar_run(d_u_kn, false, h_N_k, K, N, tol, max_iter, h_f_k, h_n_iter,
                    (cudaStream_t)stream);
}

}  // extern "C"
