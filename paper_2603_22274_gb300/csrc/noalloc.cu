// abfe_ukn_frame_noalloc: the lambda-dependent part of one frame's u_kn row for
// callers that cannot allocate device memory (for example a plugin inside a
// host MD engine whose device memory belongs to the host application's own
// allocator). It uses no context and calls no cudaMalloc/cudaFree: its only
// scratch is the file-scope array below, shared by every call on a device.
//
// One launch. Every block takes a strided share of the atoms (neighbours in the
// caller's order are neighbours in space: strided, the pairs near the ligand
// spread over all blocks) and tests them against all ligand atoms in FP32, with a
// margin above its rounding; what passes is queued in shared memory in a fixed
// order. For 256 queued pairs at a time, a thread per pair evaluates the exact
// (FP64) cutoff and exclusion tests, the unit-charge Coulomb energy and r^6 /
// sigma^6, and then the warps share out the states: with t = r^6 / sigma^6 the
// softcore LJ of a pair at (lambda_v, A) is lambda_v 4 eps (x^2 - x), x = 1 / (A +
// t), one division per pair and distinct lambda_v. Blocks leave a row of partial
// sums; the last one to finish adds them in block order (deterministic), with the
// charge-scaled Coulomb terms and lambda_r,k times the restraint energy that one
// block of its own evaluates, and writes du[k]. A ligand index outside [0, n) is
// never dereferenced: it makes the sums, and so every du[k] of that call, NaN.
// Sums and energies are FP64.
//
// Bound by the FP64 pipe (63 issue cycles per warp operation, a division 335): the
// form before this one evaluated every atom's minimum image in FP64 three times (a
// pass per 16 states) in 240 blocks and took 1,277 us for one 60,000-atom frame
// with a 60-atom ligand at 42 states (22 distinct lambda_v); 72 us now, 30 of them
// FP64 pipe time.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "abfe.h"

namespace {

constexpr int NA_MAX_BLOCKS = ABFE_NOALLOC_MAX_BLOCKS;
constexpr int NA_MAX_K = ABFE_NOALLOC_MAX_K;
constexpr int NA_SLOTS = NA_MAX_K + 2;  // LJ sums + ligand-env and ligand-ligand Coulomb
constexpr int NA_THREADS = 256;
constexpr int NA_WARPS = NA_THREADS / 32;
constexpr int NA_MAX_LIG = ABFE_NOALLOC_MAX_LIG;
constexpr int NA_TILE = 8;      // ligand atoms tested between two looks at the queues
constexpr int NA_QUEUE = 512;   // queued pairs per warp
static_assert(ABFE_NOALLOC_MAX_ATOMS <= 1 << 22 && NA_MAX_LIG <= 1 << 10,
              "a queued pair is an atom (22 bits) and a ligand atom (10 bits)");

// Scratch: one row of NA_SLOTS partial sums per block (about 1 MB), the restraint
// energy and the count of finished blocks (cleared before each launch). Every call
// overwrites the rows it uses before reading them.
static __device__ __align__(256) double g_noalloc_scratch[NA_MAX_BLOCKS * NA_SLOTS + 2];

struct NaParams {
    int n, n_lig, K, nv, nb, mode, has_boresch;
    double box[3], rc2, beta, ke;
    float boxf[3], rcf;
    const float* pos;
    const float* q;
    const float* sig;
    const float* eps;
    const unsigned char* lig;
    const int* lig_idx;
    const int* lig_excl;
    double lam_r[NA_MAX_K], lam_q[NA_MAX_K];
    double lam_v[NA_MAX_K], A[NA_MAX_K];      // per distinct lambda_v
    unsigned char v_of[NA_MAX_K];             // state -> distinct lambda_v
    int anc[6];
    double b_r0, th0[2], cph0[3], sph0[3], kr, kth, kph;
};

// nearest image of anchors' separations; the number of box lengths in FP32 (the
// same but for separations of half a box length)
__device__ __forceinline__ double mi1(double d, double L) {
    return fma(-L, (double)rintf((float)d / (float)L), d);
}

struct V3 {
    double x, y, z;
};
__device__ V3 vsub(V3 a, V3 b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ double vdot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ V3 vcross(V3 a, V3 b) {
    return V3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// term t of the restraint energy U_B of the six anchors (P1 P2 P3 L1 L2 L3),
// nearest images: 0 distance, 1-2 angles, 3-5 dihedrals
__device__ double boresch_term(const NaParams& P, int t) {
    const int atoms[6][4] = {{0, 3, 3, 3}, {0, 3, 4, 4}, {3, 0, 1, 1},
                             {1, 0, 3, 4}, {0, 3, 4, 5}, {3, 0, 1, 2}};
    V3 p[4];
    for (int i = 0; i < 4; ++i) {
        const int a = P.anc[atoms[t][i]];
        p[i] = V3{(double)P.pos[3 * a], (double)P.pos[3 * a + 1], (double)P.pos[3 * a + 2]};
    }
    auto sep = [&](int from, int to) {
        V3 d = vsub(p[to], p[from]);
        d.x = mi1(d.x, P.box[0]); d.y = mi1(d.y, P.box[1]); d.z = mi1(d.z, P.box[2]);
        return d;
    };
    if (t == 0) {
        const V3 d = sep(0, 1);
        const double r = sqrt(vdot(d, d));
        return 0.5 * P.kr * (r - P.b_r0) * (r - P.b_r0);
    }
    if (t < 3) {
        const V3 u = sep(1, 0), v = sep(1, 2);
        double c = vdot(u, v) / sqrt(vdot(u, u) * vdot(v, v));
        c = fmin(1.0, fmax(-1.0, c));
        const double th = acos(c);
        return 0.5 * P.kth * (th - P.th0[t - 1]) * (th - P.th0[t - 1]);
    }
    // cos(phi - phi0) by addition, phi = atan2(y, x) without the angle itself
    const V3 b1 = sep(0, 1), b2 = sep(1, 2), b3 = sep(2, 3);
    const V3 n1 = vcross(b1, b2), n2 = vcross(b2, b3);
    const double x = vdot(n1, n2), y = sqrt(vdot(b2, b2)) * vdot(b1, n2);
    const double h2 = x * x + y * y, ih = 1.0 / sqrt(h2);
    const double c = h2 == 0.0 ? 1.0 : x * ih, s = h2 == 0.0 ? 0.0 : y * ih;
    return P.kph * (1.0 - (c * P.cph0[t - 3] + s * P.sph0[t - 3]));
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// dynamic shared memory: ligand atoms (position, index; n_lig), queues, the
// evaluated pairs, sums [nv][32] (lane partials; the warp v % NA_WARPS owns row v)
__host__ __device__ constexpr size_t na_smem(int n_lig, int nv) {
    return sizeof(float4) * (size_t)n_lig + sizeof(double) * (2 * NA_THREADS + 32 * (size_t)nv) +
           sizeof(unsigned int) * NA_WARPS * NA_QUEUE;
}

__global__ void __launch_bounds__(NA_THREADS) k_na_frame(const __grid_constant__ NaParams P,
                                                         double* scratch, double* du) {
    extern __shared__ __align__(16) unsigned char na_raw[];
    float4* const s_lig = reinterpret_cast<float4*>(na_raw);
    double* const s_t = reinterpret_cast<double*>(s_lig + P.n_lig);   // r^6 / sigma^6
    double* const s_e = s_t + NA_THREADS;                             // 4 eps
    double* const s_acc = s_e + NA_THREADS;
    unsigned int* const s_q = reinterpret_cast<unsigned int*>(s_acc + 32 * P.nv);
    __shared__ int s_cnt[NA_WARPS];
    __shared__ float s_max[NA_WARPS];
    __shared__ double s_c[NA_WARPS][2];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    double* const ub = scratch + (size_t)NA_MAX_BLOCKS * NA_SLOTS;
    int* const done = reinterpret_cast<int*>(ub + 1);
    if ((int)blockIdx.x == P.nb) {
        // the restraint, a lane per term
        if (w == 0) {
            const double u = lane < 6 && P.has_boresch ? boresch_term(P, lane) : 0.0;
            const double s = warp_sum(u);
            if (lane == 0) *ub = s;
        }
    } else {
        bool bad = false;
        float amax = fmaxf(P.boxf[0], fmaxf(P.boxf[1], P.boxf[2]));
        for (int l = tid; l < P.n_lig; l += NA_THREADS) {
            const int a = P.lig_idx[l];
            float4 x = make_float4(0.f, 0.f, 0.f, __int_as_float(a));
            if (a < 0 || a >= P.n) {
                bad = true;
            } else {
                x.x = P.pos[3 * a]; x.y = P.pos[3 * a + 1]; x.z = P.pos[3 * a + 2];
                amax = fmaxf(amax, fmaxf(fabsf(x.x), fmaxf(fabsf(x.y), fabsf(x.z))));
            }
            s_lig[l] = x;
        }
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        if (lane == 0) s_max[w] = amax;
        for (int k = tid; k < 32 * P.nv; k += NA_THREADS) s_acc[k] = 0.0;
        const bool any_bad = __syncthreads_or(bad);
        for (int k = 0; k < NA_WARPS; ++k) amax = fmaxf(amax, s_max[k]);
        double cle = 0.0, cll = 0.0;   // ligand-environment, ligand-ligand (unit scale)
        int cnt = 0;                   // this warp's queued pairs
        // queued pairs: exact tests and per-pair values, then the states
        auto flush = [&]() {
            if (lane == 0) s_cnt[w] = cnt;
            __syncthreads();
            int pre[NA_WARPS + 1];
            pre[0] = 0;
#pragma unroll
            for (int k = 0; k < NA_WARPS; ++k) pre[k + 1] = pre[k] + s_cnt[k];
            const int total = pre[NA_WARPS];
            for (int p0 = 0; p0 < total; p0 += NA_THREADS) {
                const int p = p0 + tid;
                double tt = 0.0, e4 = 0.0;   // e4 = 0: no pair
                if (p < total) {
                    int k = 0;
#pragma unroll
                    for (int q = 1; q < NA_WARPS; ++q) k += p >= pre[q] ? 1 : 0;
                    int first = 0;
#pragma unroll
                    for (int q = 1; q < NA_WARPS; ++q) first = k == q ? pre[q] : first;
                    const unsigned int e = s_q[k * NA_QUEUE + (p - first)];
                    const int b = (int)(e & 0x3FFFFFu), l = (int)(e >> 22);
                    const float4 xa = s_lig[l];
                    const int a = __float_as_int(xa.w);
                    const bool bl = P.lig[b] != 0;
                    // each ligand-ligand pair once; decoupled ones are lambda independent
                    bool on = b != a && !(bl && (b < a || P.mode == 1));
                    if (on) {
#pragma unroll
                        for (int q = 0; q < ABFE_NOALLOC_MAX_EXCL; ++q)
                            on = on && P.lig_excl[l * ABFE_NOALLOC_MAX_EXCL + q] != b;
                    }
                    if (on) {
                        auto mi = [](double d, double L) { return d - L * rint(d / L); };
                        const double dx = mi((double)P.pos[3 * b] - (double)xa.x, P.box[0]);
                        const double dy = mi((double)P.pos[3 * b + 1] - (double)xa.y, P.box[1]);
                        const double dz = mi((double)P.pos[3 * b + 2] - (double)xa.z, P.box[2]);
                        const double r2 = dx * dx + dy * dy + dz * dz;
                        if (r2 < P.rc2) {
                            const double r = sqrt(r2);
                            const double u = P.ke * (double)P.q[a] * (double)P.q[b] * erfc(P.beta * r) / r;
                            if (bl) cll += u; else cle += u;
                            const double s = 0.5 * ((double)P.sig[a] + (double)P.sig[b]);
                            const double s2 = s * s;
                            tt = r2 * r2 * r2 / (s2 * s2 * s2);
                            e4 = 4.0 * sqrt((double)P.eps[a] * (double)P.eps[b]);
                        }
                    }
                }
                s_t[tid] = tt;
                s_e[tid] = e4;
                __syncthreads();
                const int nq = min(NA_WARPS, (total - p0 + 31) >> 5);   // warps' worth of pairs
                for (int v = w; v < P.nv; v += NA_WARPS) {
                    const double A = P.A[v];
                    double acc = s_acc[32 * v + lane];
                    for (int q = 0; q < nq; ++q) {
                        const double e = s_e[32 * q + lane];
                        // (a zero well depth adds nothing, whatever t; integer test)
                        if (__double_as_longlong(e) != 0ll) {
                            const double x = 1.0 / (A + s_t[32 * q + lane]);
                            acc = fma(e, fma(x, x, -x), acc);
                        }
                    }
                    s_acc[32 * v + lane] = acc;
                }
                __syncthreads();
            }
            cnt = 0;
        };
        // block b's warp w takes atoms b + nb (w + 8 (lane + 32 i))
        const int nw = P.nb * NA_WARPS;
        const int first = (int)blockIdx.x + P.nb * w;
        const int rounds = any_bad ? 0 : (P.n + nw * 32 - 1) / (nw * 32);
        for (int i = 0; i < rounds; ++i) {
            const long long bb = (long long)first + (long long)nw * (lane + 32 * i);
            const int b = bb < P.n ? (int)bb : -1;
            float x = 0.f, y = 0.f, z = 0.f;
            if (b >= 0) {
                x = P.pos[3 * b]; y = P.pos[3 * b + 1]; z = P.pos[3 * b + 2];
            }
            // FP32 rounding of a separation: a few ulps of the largest coordinate or box
            // length in it; not-a-numbers pass to the exact test
            const float m = fmaxf(amax, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
            const float lim = P.rcf * 1.00001f + 4.0e-6f * m;
            for (int l0 = 0; l0 < P.n_lig; l0 += NA_TILE) {
#pragma unroll
                for (int l = l0; l < l0 + NA_TILE; ++l) {
                    bool hit = false;
                    if (l < P.n_lig && b >= 0) {
                        const float4 a = s_lig[l];
                        float dx = x - a.x, dy = y - a.y, dz = z - a.z;
                        dx = fmaf(-P.boxf[0], rintf(dx / P.boxf[0]), dx);
                        dy = fmaf(-P.boxf[1], rintf(dy / P.boxf[1]), dy);
                        dz = fmaf(-P.boxf[2], rintf(dz / P.boxf[2]), dz);
                        hit = !(dx * dx + dy * dy + dz * dz >= lim * lim);
                    }
                    const unsigned int bal = __ballot_sync(0xffffffffu, hit);
                    if (hit)
                        s_q[w * NA_QUEUE + cnt + __popc(bal & ((1u << lane) - 1u))] =
                            (unsigned int)b | ((unsigned int)l << 22);
                    cnt += __popc(bal);
                }
                // room for the next tile in every warp's queue?
                if (__syncthreads_or(cnt > NA_QUEUE - 32 * NA_TILE)) flush();
            }
        }
        flush();
        // the block's row of partial sums: four lanes' worth per state and thread
        const double sle = warp_sum(cle), sll = warp_sum(cll);
        if (lane == 0) {
            s_c[w][0] = sle;
            s_c[w][1] = sll;
        }
        __syncthreads();
        double* const row = scratch + (size_t)blockIdx.x * NA_SLOTS;
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        for (int v = w; v < P.nv; v += NA_WARPS) {
            const double s = warp_sum(s_acc[32 * v + lane]);
            if (lane == 0) row[v] = any_bad ? nan : P.lam_v[v] * s;
        }
        if (tid < 2) {
            double s = 0.0;
            for (int k = 0; k < NA_WARPS; ++k) s += s_c[k][tid];
            row[P.nv + tid] = any_bad ? nan : s;
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(done, 1) == P.nb;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the last block: every slot's rows in order, a warp per slot
    for (int v = w; v < P.nv + 2; v += NA_WARPS) {
        double s = 0.0;
        for (int r = lane; r < P.nb; r += 32) s += __ldcg(scratch + (size_t)r * NA_SLOTS + v);
        s = warp_sum(s);
        if (lane == 0) s_t[v] = s;
    }
    const double u = __ldcg(ub);
    __syncthreads();
    const double cle = s_t[P.nv], cll = s_t[P.nv + 1];
    for (int k = tid; k < P.K; k += NA_THREADS) {
        const double lq = P.lam_q[k];
        du[k] = s_t[P.v_of[k]] + lq * cle + lq * lq * cll + P.lam_r[k] * u;
    }
}

std::mutex g_na_mutex;
double* g_na_ptr[64] = {nullptr};
int g_na_sm[64] = {0};

}  // namespace

extern "C" abfe_status abfe_ukn_frame_noalloc(const abfe_noalloc_frame* f, double* d_du,
                                              void* cuda_stream) {
    if (!f || !d_du || !f->pos || !f->charge || !f->sigma || !f->epsilon || !f->is_ligand ||
        !f->lig_idx || !f->lig_excl)
        return ABFE_ERR_INVALID_ARG;
    if (f->n_atoms < 1 || f->n_atoms > ABFE_NOALLOC_MAX_ATOMS || f->n_lig < 1 ||
        f->n_lig > ABFE_NOALLOC_MAX_LIG || f->K < 1 || f->K > NA_MAX_K)
        return ABFE_ERR_INVALID_ARG;  // sizes beyond the documented maxima
    if (!(f->cutoff > 0) || !(f->sc_p >= 1.0) || (f->ligand_mode != 0 && f->ligand_mode != 1))
        return ABFE_ERR_INVALID_ARG;
    for (int d = 0; d < 3; ++d)
        if (!(f->cutoff < 0.5 * f->box[d])) return ABFE_ERR_CUTOFF_TOO_LARGE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return ABFE_ERR_CUDA;
    }
    double* scratch = nullptr;
    int n_sm = 0;
    {
        // first call on a device: look up the device address of the scratch
        // array with that device current
        std::lock_guard<std::mutex> lk(g_na_mutex);
        if (!g_na_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return ABFE_ERR_CUDA;
            }
            if (cudaDeviceGetAttribute(&g_na_sm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
                cudaFuncSetAttribute(k_na_frame, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)na_smem(NA_MAX_LIG, NA_MAX_K)) != cudaSuccess) {
                cudaGetLastError();
                return ABFE_ERR_CUDA;
            }
            g_na_ptr[dev] = static_cast<double*>(p);
        }
        scratch = g_na_ptr[dev];
        n_sm = g_na_sm[dev];
    }
    NaParams P;
    P.n = f->n_atoms;
    P.n_lig = f->n_lig;
    P.K = f->K;
    P.mode = f->ligand_mode;
    P.has_boresch = f->has_boresch ? 1 : 0;
    for (int d = 0; d < 3; ++d) P.box[d] = f->box[d];
    P.rc2 = f->cutoff * f->cutoff;
    P.beta = f->ewald_beta;
    P.ke = f->coulomb_k;
    for (int d = 0; d < 3; ++d) P.boxf[d] = (float)f->box[d];
    P.rcf = (float)f->cutoff;
    P.nv = 0;
    P.pos = f->pos;
    P.q = f->charge;
    P.sig = f->sigma;
    P.eps = f->epsilon;
    P.lig = f->is_ligand;
    P.lig_idx = f->lig_idx;
    P.lig_excl = f->lig_excl;
    for (int k = 0; k < f->K; ++k) {
        const double lr = f->lam_r[k], lq = f->lam_q[k], lv = f->lam_v[k];
        if (!(lr >= 0 && lr <= 1 && lq >= 0 && lq <= 1 && lv >= 0 && lv <= 1))
            return ABFE_ERR_INVALID_ARG;
        P.lam_r[k] = lr;
        P.lam_q[k] = lq;
        int v = 0;
        while (v < P.nv && P.lam_v[v] != lv) ++v;
        if (v == P.nv) {
            P.lam_v[v] = lv;
            P.A[v] = f->sc_alpha * std::pow(1.0 - lv, f->sc_p);
            ++P.nv;
        }
        P.v_of[k] = (unsigned char)v;
    }
    for (int i = 0; i < 6; ++i) {
        P.anc[i] = f->anchors[i];
        if (P.has_boresch && (P.anc[i] < 0 || P.anc[i] >= P.n)) return ABFE_ERR_INVALID_ARG;
    }
    P.b_r0 = f->b_r0;
    P.th0[0] = f->b_theta0[0]; P.th0[1] = f->b_theta0[1];
    for (int i = 0; i < 3; ++i) {
        P.cph0[i] = std::cos(f->b_phi0[i]);
        P.sph0[i] = std::sin(f->b_phi0[i]);
    }
    P.kr = f->b_kr; P.kth = f->b_ktheta; P.kph = f->b_kphi;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // one block per SM for small frames, two for large ones (4,500 atoms: 51 against
    // 60 us; 60,000: 78 against 72; 100,000 with cutoff 1.2 nm: 142 against 129);
    // a block more for the restraint
    const int sm = n_sm > 0 ? n_sm : 1;
    P.nb = std::min(std::min((P.n >= 32768 ? 2 : 1) * sm, NA_MAX_BLOCKS), (P.n + 7) / 8);
    if (cudaMemsetAsync(scratch + (size_t)NA_MAX_BLOCKS * NA_SLOTS + 1, 0, sizeof(double), s) != cudaSuccess) {
        cudaGetLastError();
        return ABFE_ERR_CUDA;
    }
    k_na_frame<<<P.nb + 1, NA_THREADS, na_smem(P.n_lig, P.nv), s>>>(P, scratch, d_du);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ABFE_OK : ABFE_ERR_CUDA;
}
