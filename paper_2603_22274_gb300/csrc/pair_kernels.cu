// Nonbonded pair kernels.
//
// * k_env_rows: environment-environment pairs (lambda independent): plain
//   12-6 LJ with Lorentz-Berthelot mixing plus real-space Ewald Coulomb, hard
//   cutoff, over the inner list of j rows. A warp owns one i-cluster (8 atoms,
//   held in shared memory) and walks its rows 32 at a time, a lane per row:
//   the lane loads the row's j atom once and evaluates it against all 8 i atoms,
//   dropping those that the row does not cover (atoms 4-7 or 0-3 of a half row,
//   excluded ones of a masked row); its j force goes to the 64-bit fixed-point
//   accumulators once per row and the i forces stay in registers until the item
//   ends. FP32 forces: the Coulomb force is
//   qq G(r) / r^3 with G from a quadratic table in r held in shared memory
//   (ewald_G); FP32 energies (energy steps only) use erfc from a second table and
//   the force's reciprocal root, corrected.
// * k_env_rows_f64: the same pairs in FP64 contexts, erfc from Taylor coefficients.
// * k_lig: ligand-involved pairs at the replica's own state (outer list, 4x8
//   half tiles: lane = jj + 8 ii): Beutler softcore LJ, lambda_q-scaled
//   charges, dU/dlambda_v and dU/dlambda_q; pair arithmetic in the kernel's
//   precision, energy sums (energy steps only) in FP64.
// * k_lig_ukn: the same pairs at every distinct lambda_v of the replica's
//   schedule, plus the unit-charge Coulomb sums, for the u_kn row.
// * k_count_rows / k_count: in-cutoff pair counts through the inner rows and the
//   ligand list (list parity checks) and the computed pair lanes.
#include <cuda_runtime.h>

#include "abfe_internal.cuh"

namespace abfe {

namespace {

constexpr unsigned FULL = 0xffffffffu;

template <typename T>
struct T3 {
    T x, y, z;
};

template <typename T>
struct Atom {
    T x, y, z, q, sh, e2;  // position, q sqrt(ke), sigma/2, 2 sqrt(eps)
};

template <typename T>
struct KC {
    T rc2, beta, tbsp, nb2l2e, dke_sqrt;
    const float4* tab;    // FP32 path: the Ewald force table in shared memory
    const float4* etab;   // and that of erfc (energy steps)
    const double2* dtab;  // FP64 path: erfc's expansions (see erfc_table)
    float inv_h;
};

template <typename T>
__device__ __forceinline__ KC<T> make_kc(const DevPtrs& P);
template <>
__device__ __forceinline__ KC<float> make_kc<float>(const DevPtrs& P) {
    return KC<float>{P.rc2, P.beta, P.tbsp, P.nb2l2e, P.sqrt_ke, nullptr, nullptr, nullptr, P.ewtab_inv_h};
}
template <>
__device__ __forceinline__ KC<double> make_kc<double>(const DevPtrs& P) {
    return KC<double>{P.drc2, P.dbeta, 2.0 * P.dbeta / sqrt(3.14159265358979323846), 0.0,
                      sqrt(P.dke), nullptr, nullptr, P.erfc_tab, 0.0f};
}

template <typename T>
__device__ __forceinline__ Atom<T> load_atom(const DevPtrs& P, int slot, const RepDev& R,
                                             const KC<T>& K);
template <>
__device__ __forceinline__ Atom<float> load_atom<float>(const DevPtrs& P, int slot, const RepDev&,
                                                        const KC<float>&) {
    const float4 x = P.xq[slot];
    const float2 s = P.se[slot];
    return Atom<float>{x.x, x.y, x.z, x.w, s.x, s.y};
}
template <>
__device__ __forceinline__ Atom<double> load_atom<double>(const DevPtrs& P, int slot,
                                                          const RepDev& R, const KC<double>& K) {
    const float4 x = P.xq[slot];
    const int o = P.orig[slot];
    Atom<double> a{(double)x.x, (double)x.y, (double)x.z, 0.0, 0.0, 0.0};
    if (o >= 0) {
        const int sys_atom_off = R.sys_atom_off;
        const dbl4 p = P.sys_prmd[sys_atom_off + o];
        // alchemical oxygens: q0 + (1 - lambda_q) dq
        a.q = fma(1.0 - R.dlam_q, P.sys_dqd[sys_atom_off + o], p.x) * K.dke_sqrt;
        a.sh = p.y;
        a.e2 = p.z;
    }
    return a;
}


// G(r) from the shared-memory table: the nearest grid point j = round(t),
// t = r / h (clamped to the table), and the centred quadratic in f = t - j.
// Adding 1.5 * 2^23 leaves round(t) in the low mantissa bits (t < 2^22), so no
// conversion instruction is needed.
__device__ __forceinline__ float ewald_G(float r, const float4* tab, float inv_h) {
    const float t = fminf(r * inv_h, (float)(EW_NT - 1));
    const float tr = t + 12582912.0f;
    const int j = __float_as_int(tr) - 0x4B400000;
    const float f = t - (tr - 12582912.0f);
    const float4 c = tab[j];
    return fmaf(fmaf(c.z, f, c.y), f, c.x);
}

// erfc(beta r) from its table, the centred quadratic about the nearest point of the
// same grid (see ewald_G). The offset is one multiply-add, so r's own rounding is the
// only one in it; the value at the point is held to twice binary32 (c.x + c.w), since
// its rounding would be common to every pair near that point.
__device__ __forceinline__ float ewald_erfc(float r, const float4* tab, float inv_h) {
    const float t = fminf(r * inv_h, (float)(EW_NT - 1));
    const float tr = t + 12582912.0f;
    const int j = __float_as_int(tr) - 0x4B400000;
    const float f = fmaf(r, inv_h, -(tr - 12582912.0f));
    const float4 c = tab[j];
    return c.x + fmaf(fmaf(c.z, f, c.y), f, c.w);
}

// correctly rounded / library-accurate variants, used for ligand pairs (dU/dlambda and
// u_kn)
__device__ __forceinline__ float t_sqrt_acc(float x) { return __fsqrt_rn(x); }
__device__ __forceinline__ float t_rcp_acc(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double t_rcp_acc(double x) { return 1.0 / x; }
__device__ __forceinline__ void ewald_acc(float r, float r2, const KC<float>& K, float& erfcv,
                                          float& ex) {
    ex = expf(-(K.beta * K.beta) * r2);
    erfcv = erfcf(K.beta * r);
}
__device__ __forceinline__ void ewald_acc(double r, double, const KC<double>& K, double& erfcv,
                                          double& ex) {
    double d;   // erfc'(x) = -2 / sqrt(pi) exp(-x^2)
    erfc_table(K.beta * r, K.dtab, erfcv, d);
    ex = -0.88622692545275801 * d;
}

// r, 1 / r and 1 / r^2: for energies and ligand pairs
__device__ __forceinline__ void root_acc(float r2, float& r, float& rinv, float& rinv2) {
    r = t_sqrt_acc(r2);
    rinv = t_rcp_acc(r);
    rinv2 = t_rcp_acc(r2);
}
__device__ __forceinline__ void root_acc(double r2, double& r, double& rinv, double& rinv2) {
    rinv = rsqrt(r2);
    const double r0 = r2 * rinv;
    r = fma(fma(-r0, r0, r2), 0.5 * rinv, r0);
    rinv2 = rinv * rinv;
}

// x_j + s - c (image shift s, reference atom c of the i-cluster): the box
// length is only subtracted from a coordinate near it (exact), so an image
// pair's separation carries no rounding of a box-sized sum
template <typename T>
__device__ __forceinline__ T rel_img(float xj, float s, float c) {
    return s > 0.f ? (T)xj + (T)(s - c) : ((T)xj + (T)s) - (T)c;
}

// Inner-list item `it` of the iteration space over all replicas' regions: from
// the replica of its block of 256 items, forward to the last replica r with
// ritem_pref[r] <= it (an empty replica shares its successor's prefix).
__device__ __forceinline__ const RowItem& row_item(const DevPtrs& P, int it) {
    int r = P.ritem_blk[it >> 8];
    while (r + 1 < P.R && P.ritem_pref[r + 1] <= it) ++r;
    return P.ritems[P.ritem_base[r] + (it - P.ritem_pref[r])];
}

// ------------------------------------------------------------------ env pair
// (a pair that is not kept adds exact zeros)
template <bool ENERGY>
__device__ __forceinline__ void pair_env(const Atom<float>& ai, const Atom<float>& aj, bool keep,
                                         T3<float>& fi, T3<float>& fj, float& elj, float& ec,
                                         const KC<float>& K) {
    const float dx = aj.x - ai.x, dy = aj.y - ai.y, dz = aj.z - ai.z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    keep = keep && (r2 < K.rc2);
    const float rinv = rsqrt_fast(r2);
    const float rinv2 = rinv * rinv;
    const float qq = ai.q * aj.q;
    // Coulomb force times r^2: qq G(r) / r from the table
    const float fcr = qq * ewald_G(r2 * rinv, K.tab, K.inv_h) * rinv;
    const float sig = ai.sh + aj.sh;
    const float eps4 = ai.e2 * aj.e2;
    const float s2 = sig * sig * rinv2;
    const float s6 = s2 * s2 * s2;
    // F / r = [Coulomb r^2 + 4 eps s6 (12 s6 - 6)] / r^2
    const float fs = keep ? fmaf(eps4 * s6, fmaf(12.f, s6, -6.f), fcr) * rinv2 : 0.f;
    // explicit FMAs (never left to contraction), so the force and energy
    // variants of the kernel add every pair force with the same roundings
    fi.x = fmaf(-fs, dx, fi.x); fi.y = fmaf(-fs, dy, fi.y); fi.z = fmaf(-fs, dz, fi.z);
    fj.x = fmaf(fs, dx, fj.x);  fj.y = fmaf(fs, dy, fj.y);  fj.z = fmaf(fs, dz, fj.z);
    if (ENERGY) {
        // (energy steps only.) The force's fast reciprocal root, corrected to r, 1 / r
        // and 1 / r^2 of about half a unit in the last place each, and erfc from its
        // table. sqrt, two reciprocals and erfcf, each accurate by itself, took 195
        // issue cycles a pair, most of the pass (24 windows of 25,000 atoms: 1489 us
        // with them, 750 us).
        const float r0 = r2 * rinv;
        const float re = fmaf(fmaf(-r0, r0, r2), 0.5f * rinv, r0);
        const float y = fmaf(rinv, fmaf(-re, rinv, 1.f), rinv);
        const float r2inv = fmaf(rinv2, fmaf(-r2, rinv2, 1.f), rinv2);
        const float vce = qq * ewald_erfc(re, K.etab, K.inv_h) * y;
        const float s2e = sig * sig * r2inv;
        const float s6e = s2e * s2e * s2e;
        const float vlj = eps4 * fmaf(s6e, s6e, -s6e);
        elj += keep ? vlj : 0.f;
        ec += keep ? vce : 0.f;
    }
}

template <typename T>
__device__ __forceinline__ void red_jforce(const DevPtrs& P, int ja, int ii, T3<T> fj) {
    fj.x += __shfl_xor_sync(FULL, fj.x, 8);
    fj.y += __shfl_xor_sync(FULL, fj.y, 8);
    fj.z += __shfl_xor_sync(FULL, fj.z, 8);
    fj.x += __shfl_xor_sync(FULL, fj.x, 16);
    fj.y += __shfl_xor_sync(FULL, fj.y, 16);
    fj.z += __shfl_xor_sync(FULL, fj.z, 16);
    const T v = ii == 0 ? fj.x : (ii == 1 ? fj.y : fj.z);
    if (ii < 3 && v != (T)0) {
        long long* dst = ii == 0 ? P.fx : (ii == 1 ? P.fy : P.fz);
        add_fixed(dst + ja, (sizeof(T) == 4) ? to_fixed((float)v) : to_fixed_d((double)v));
    }
}

// i-forces: sum over the 8 lanes sharing ii, then lanes jj=0..2 write atom ii
// and lanes jj=3..5 write atom ii+4.
template <typename T>
__device__ __forceinline__ void red_iforce(const DevPtrs& P, int base_slot, int ii, int jj,
                                           T3<T> f0, T3<T> f1) {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        f0.x += __shfl_xor_sync(FULL, f0.x, o);
        f0.y += __shfl_xor_sync(FULL, f0.y, o);
        f0.z += __shfl_xor_sync(FULL, f0.z, o);
        f1.x += __shfl_xor_sync(FULL, f1.x, o);
        f1.y += __shfl_xor_sync(FULL, f1.y, o);
        f1.z += __shfl_xor_sync(FULL, f1.z, o);
    }
    if (jj < 6) {
        const T3<T> f = jj < 3 ? f0 : f1;
        const int c = jj % 3;
        const T v = c == 0 ? f.x : (c == 1 ? f.y : f.z);
        if (v != (T)0) {
            long long* dst = c == 0 ? P.fx : (c == 1 ? P.fy : P.fz);
            const int a = base_slot + ii + (jj < 3 ? 0 : 4);
            add_fixed(dst + a, (sizeof(T) == 4) ? to_fixed((float)v) : to_fixed_d((double)v));
        }
    }
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Sums of 24 per-lane values over the warp by halving exchanges: at lane bit
// 4, 3, 2 each lane keeps the half of its values that matches its bit and adds
// the partner's copy of that half (12, 6, 3 shuffles), then bits 1 and 0 sum
// the remaining three in full. On return v[0] holds the sum of value
// 12 b4 + 6 b3 + 3 b2 + (lane & 3) for lane & 3 < 3 (the index is returned).
template <typename T>
__device__ __forceinline__ int warp_sum_24(T (&v)[24], int lane) {
    const bool b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        const T keep = b4 ? v[j + 12] : v[j], give = b4 ? v[j] : v[j + 12];
        v[j] = keep + __shfl_xor_sync(FULL, give, 16);
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const T keep = b3 ? v[j + 6] : v[j], give = b3 ? v[j] : v[j + 6];
        v[j] = keep + __shfl_xor_sync(FULL, give, 8);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const T keep = b2 ? v[j + 3] : v[j], give = b2 ? v[j] : v[j + 3];
        v[j] = keep + __shfl_xor_sync(FULL, give, 4);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        v[j] += __shfl_xor_sync(FULL, v[j], 2);
        v[j] += __shfl_xor_sync(FULL, v[j], 1);
    }
    const int q = lane & 3;
    const T out = q == 1 ? v[1] : (q == 2 ? v[2] : v[0]);
    v[0] = out;
    return 12 * b4 + 6 * b3 + 3 * b2 + (q < 3 ? q : 0);
}

// ------------------------------------------------------------------ env rows
// Lane per j row: lane l of a warp takes row k0 + l of its item, loads the
// row's j atom once and evaluates it against the cluster's 8 i atoms, read as
// broadcasts from the warp's copy of the i-cluster in shared memory. The j force
// stays in the lane and goes to the fixed-point accumulators once per row; the i
// forces stay in registers (8 atoms x 3) until the item ends and are then summed
// over the warp. Rounds of 32 full rows evaluate eight pairs per lane without a
// check; the last one or two rounds of an item (the remaining full rows, rows with
// only atoms 0-3 or 4-7 in range, masked rows, idle lanes) check each pair.
constexpr int ENV_WARPS_MAX = 8;

// one i atom in shared memory: x, y, z, q sqrt(ke), sigma/2, 2 sqrt(eps), -, -
__device__ __forceinline__ Atom<float> ld_iatom(const float* p) {
    const float4 a = reinterpret_cast<const float4*>(p)[0];
    const float2 b = reinterpret_cast<const float2*>(p)[2];
    return Atom<float>{a.x, a.y, a.z, a.w, b.x, b.y};
}
__device__ __forceinline__ void st_iatom(float* p, const Atom<float>& a) {
    p[0] = a.x; p[1] = a.y; p[2] = a.z; p[3] = a.q; p[4] = a.sh; p[5] = a.e2;
    p[6] = 0.f; p[7] = 0.f;
}

// adds a force component to an accumulator unless it is zero (no pair in range)
__device__ __forceinline__ void red_nonzero(long long* p, float f) {
    const long long v = to_fixed(f);
    if (f != 0.f) add_fixed(p, v);
}
__device__ __forceinline__ void red_nonzero(long long* p, double f) {
    const long long v = to_fixed_d(f);
    if (v != 0) add_fixed(p, v);
}

// Image shifts of a replica's box, by code, for the lane's code: x_j + s - c for image
// shift s and reference atom c is evaluated as (x_j + u) - v with u = s - c, v = 0
// where s > 0 (then c lies near the box length, and s - c is exact) and u = s, v = c
// otherwise (x_j + s is exact where s < 0, x_j lying near the box length): no box-sized
// sum is rounded.
__device__ __forceinline__ void row_shifts(const RepDev& R, const float4& c, int lane, float4* sh) {
    if (lane < 27) {
        const float sx = (float)(lane % 3 - 1) * R.box[0],
                    sy = (float)((lane / 3) % 3 - 1) * R.box[1],
                    sz = (float)(lane / 9 - 1) * R.box[2];
        sh[lane] = make_float4(sx > 0.f ? sx - c.x : sx, sy > 0.f ? sy - c.y : sy,
                               sz > 0.f ? sz - c.z : sz, 0.f);
        sh[32 + lane] = make_float4(sx > 0.f ? 0.f : c.x, sy > 0.f ? 0.f : c.y,
                                    sz > 0.f ? 0.f : c.z, 0.f);
    }
}

// One row of a lane against the i atoms; CHECK: minus those in `em`.
template <bool ENERGY, bool CHECK>
__device__ __forceinline__ void env_row(const DevPtrs& P, const KC<float>& K, const float* s_ia,
                                        const float4* sh, unsigned int word, unsigned int em,
                                        const Atom<float>& aj, T3<float> (&fi)[CL], double& elj_d,
                                        double& ec_d) {
    // the j atom relative to the cluster's reference atom c, (x_j + u) - v
    // with (u, v) from the row's image code
    const int code = (int)(word >> ROW_SLOT_BITS);
    const float4 u = sh[code], v = sh[32 + code];
    Atom<float> a = aj;
    a.x = (aj.x + u.x) - v.x;
    a.y = (aj.y + u.y) - v.y;
    a.z = (aj.z + u.z) - v.z;
    T3<float> fj{0.f, 0.f, 0.f};
    float elj = 0, ec = 0;
#pragma unroll
    for (int ii = 0; ii < CL; ++ii)
        pair_env<ENERGY>(ld_iatom(s_ia + ii * 8), a, !(CHECK && ((em >> ii) & 1u)), fi[ii], fj, elj, ec, K);
    if (ENERGY) {
        elj_d += (double)elj;
        ec_d += (double)ec;
    }
    const int ja = (int)(word & ROW_SLOT_MASK);
    red_nonzero(P.fx + ja, fj.x);
    red_nonzero(P.fy + ja, fj.y);
    red_nonzero(P.fz + ja, fj.z);
}

// row k of an item (I: the words of a RowItem) beyond its full rounds: plain
// rows (full | atoms 0-3 only | atoms 4-7 only), then masked rows; the i atoms
// that it must not meet (all of them past the last row)
__device__ __forceinline__ void env_tail_row(const DevPtrs& P, const volatile int* I, int k,
                                             unsigned int& word, unsigned int& em) {
    const int n_full = I[3] & 0xFFFF, n_lo_end = n_full + I[4], n_plain = n_lo_end + I[5],
              n = n_plain + (I[3] >> 16);
    const int kk = min(k, n - 1);
    if (kk < n_plain) {
        word = P.rows[(unsigned int)I[1] + (unsigned int)kk];
        em = kk < n_full ? 0u : (kk < n_lo_end ? 0xF0u : 0x0Fu);
    } else {
        const int2 xr = P.xrows[I[2] + (kk - n_plain)];
        word = (unsigned int)xr.x;
        em = (unsigned int)xr.y;
    }
    if (k >= n) em = 0xFFu;
}

// A warp's first item is its own index, dealt over the blocks, so that a small
// system needs no claims (4,864 warps claiming one counter take 3 us) and its
// idle blocks leave at once; later items are claimed, up to four at a time (one
// claim per item serialised on the counter: +0.5 ms per launch on the
// 1,152-window batch), fewer when there are few items per warp. MINB: blocks of
// 256 threads per SM that the registers allow (4: 64 registers, for many items
// per warp; fewer for small systems, see env_small).
//
// The item and the claim counters live in shared memory (volatile: read again
// where they are needed), so that 64 registers hold the round loop: with them in
// registers it spilled inside the loop (24 x 25k atoms: 472 us, 427 from shared
// memory). On that workload it buys the claim scheme and no time: the prefetch of
// the next round's atom with the former claims, in registers, took 429.
template <bool ENERGY, int MINB>
__global__ void __launch_bounds__(256, MINB) k_env_rows(DevPtrs P) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __shared__ float4 s_ewtab[EW_NT];
    __shared__ float4 s_etab[ENERGY ? EW_NT : 1];
    // per warp and image code: u (0-26) and v (32-58) of the shifted j atom
    // relative to the i-cluster's reference atom
    __shared__ float4 s_shift[ENV_WARPS_MAX][64];
    __shared__ __align__(16) float s_iat[ENV_WARPS_MAX][CL * 8];
    __shared__ int s_item[ENV_WARPS_MAX][8];   // the warp's RowItem
    __shared__ int s_next[ENV_WARPS_MAX][2];   // its next item, end of the claimed ones
    volatile int* const I = s_item[w];
    volatile int* const N = s_next[w];
    KC<float> K = make_kc<float>(P);
    {
        const int n_items = P.ritem_pref[P.R];
        if ((int)blockIdx.x >= n_items) return;   // no warp of this block has an item
        for (int i = threadIdx.x; i < EW_NT; i += blockDim.x) s_ewtab[i] = P.ewtab[i];
        K.tab = s_ewtab;
        if constexpr (ENERGY) {
            for (int i = threadIdx.x; i < EW_NT; i += blockDim.x) s_etab[i] = P.ewtab[EW_NT + i];
            K.etab = s_etab;
        }
        if (lane == 0) {
            N[0] = w * (int)gridDim.x + (int)blockIdx.x;
            N[1] = min(N[0] + 1, n_items);
        }
        __syncthreads();
    }
    float4* const sh = s_shift[w];
    float* const s_ia = s_iat[w];
    for (;;) {
        {
            __syncwarp();
            int it = N[0];
            const int it_end = N[1];
            __syncwarp();
            if (it >= it_end) {
                const int nw = (int)(gridDim.x * (blockDim.x >> 5)), n_items = P.ritem_pref[P.R];
                if (nw >= n_items) break;
                const int chunk = max(1, min(4, n_items / (nw * 8)));
                if (lane == 0) it = nw + atomicAdd(&P.cnt->env_next, chunk);
                it = __shfl_sync(FULL, it, 0);
                if (it >= n_items) break;
                if (lane == 0) N[1] = min(it + chunk, n_items);
            }
            if (lane == 0) N[0] = it + 1;
            const RowItem& item = row_item(P, it);
            if (lane < 8) I[lane] = reinterpret_cast<const int*>(&item)[lane];
            __syncwarp();
            // image shifts; the i-cluster's atoms relative to its first atom (the
            // reference c; same cluster: exact)
            const RepDev& R = P.reps[P.rep_of_cl[I[0]]];
            const float4 c = P.xq[I[0] * CL];
            row_shifts(R, c, lane, sh);
            if (lane < CL) {
                Atom<float> ai = load_atom<float>(P, I[0] * CL + lane, R, K);
                ai.x -= c.x;
                ai.y -= c.y;
                ai.z -= c.z;
                st_iatom(s_ia + lane * 8, ai);
            }
            __syncwarp();
        }
        T3<float> fi[CL];
#pragma unroll
        for (int ii = 0; ii < CL; ++ii) fi[ii] = T3<float>{0.f, 0.f, 0.f};
        double elj = 0.0, ec = 0.0;
        const RepDev& R = P.reps[0];   // (FP32 atoms hold their own parameters)
        {
            // full rounds: the next round's row word is loaded a round ahead, its atom
            // is not (the other warps cover that latency at fewer registers) unless
            // there are no other warps
            int nf = (I[3] & 0xFFFF) >> 5;
            const unsigned int* rp = P.rows + ((unsigned int)I[1] + (unsigned int)lane);
            unsigned int word = nf > 0 ? *rp : 0u;
            if (MINB == 1) {
                Atom<float> aj{};
                if (nf > 0) aj = load_atom<float>(P, (int)(word & ROW_SLOT_MASK), R, K);
                for (; nf > 0; --nf) {
                    rp += 32;
                    unsigned int word_n = word;
                    Atom<float> aj_n = aj;
                    if (nf > 1) {
                        word_n = *rp;
                        aj_n = load_atom<float>(P, (int)(word_n & ROW_SLOT_MASK), R, K);
                    }
                    env_row<ENERGY, false>(P, K, s_ia, sh, word, 0u, aj, fi, elj, ec);
                    word = word_n;
                    aj = aj_n;
                }
            } else {
                for (; nf > 0; --nf) {
                    rp += 32;
                    const unsigned int word_n = nf > 1 ? *rp : 0u;
                    const Atom<float> aj = load_atom<float>(P, (int)(word & ROW_SLOT_MASK), R, K);
                    env_row<ENERGY, false>(P, K, s_ia, sh, word, 0u, aj, fi, elj, ec);
                    word = word_n;
                }
            }
        }
        for (int k0 = (I[3] & 0xFFFF) & ~31; k0 < (I[3] & 0xFFFF) + I[4] + I[5] + (I[3] >> 16); k0 += 32) {
            unsigned int word, em;
            env_tail_row(P, I, k0 + lane, word, em);
            const Atom<float> aj = load_atom<float>(P, (int)(word & ROW_SLOT_MASK), R, K);
            env_row<ENERGY, true>(P, K, s_ia, sh, word, em, aj, fi, elj, ec);
        }
        // i forces: the 24 values 3 ii + c summed over the warp (transposed);
        // value v ends on the four lanes of group v / 3, and the lane with
        // lane % 4 == v % 3 < 3 writes it
        float v[3 * CL];
#pragma unroll
        for (int ii = 0; ii < CL; ++ii) {
            v[3 * ii] = fi[ii].x;
            v[3 * ii + 1] = fi[ii].y;
            v[3 * ii + 2] = fi[ii].z;
        }
        const int vi = warp_sum_24<float>(v, lane);
        if ((lane & 3) < 3 && v[0] != 0.f) {
            const int c = vi % 3;
            long long* d = c == 0 ? P.fx : (c == 1 ? P.fy : P.fz);
            add_fixed(d + I[0] * CL + vi / 3, to_fixed(v[0]));
        }
        if (ENERGY) {
            const double sl = warp_sum<double>(elj);
            const double sc = warp_sum<double>(ec);
            if (lane == 0) {
                const int rep = P.rep_of_cl[I[0]];
                if (!isfinite(sl) || !isfinite(sc)) set_err(P.cnt, ERRB_NONFINITE, rep);
                add_fixed(P.eacc + (size_t)rep * EA_N + EA_ENV_LJ, to_fixed_d(sl));
                add_fixed(P.eacc + (size_t)rep * EA_N + EA_ENV_C, to_fixed_d(sc));
            }
        }
    }
}

// FP64 environment rows (precision 1: energies on every pass), bound by the FP64 pipe,
// which takes 64 cycles per warp instruction. So no FP64 work is spent on pairs out of
// range: a row's eight pairs are tested in FP32 with a margin (5e-5 of r_c, far above
// the rounding of the binary32 positions), and a lane then works off its row's set bits
// pair by pair with the exact test, taking the next free row of the warp when it has
// none left. Rows are handed out by ballot ranks once ENVD_REFILL lanes wait: the order
// depends on the item alone. erfc and its derivative come from one table lookup, and
// energies share the force's root. The forces of the eight i atoms are kept per lane in
// shared memory, since a lane's i atom varies. An item is worked off by ENVD_SEG warps,
// each with a part of its rows. (12 frames of 672 atoms: 1531 us with eight pairs per
// row and exp and erfc evaluated for the force and for the energy, 301 us; the pipe is
// 81% busy while a multiprocessor works.)
// The block has the tuning's size; the state of each of its warps is in dynamic shared
// memory. (128 registers per thread at any of those sizes.)
struct EnvdWarp {
    float4 p[CL], shift[64];
    double f[3 * CL][32];
    Atom<double> i[CL];
    int item[8];
};
__global__ void __launch_bounds__(ENV_WARPS_MAX * 32, 2) k_env_rows_f64(DevPtrs P) {
    extern __shared__ __align__(16) unsigned char envd_raw[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    EnvdWarp& W = reinterpret_cast<EnvdWarp*>(envd_raw)[w];
    const KC<double> K = make_kc<double>(P);
    const float near2 = fmaf(P.rc2, 1e-4f, P.rc2) + 1e-5f;
    const int n_units = P.ritem_pref[P.R] * ENVD_SEG;
    const int nw = (int)(gridDim.x * (blockDim.x >> 5));
    const unsigned int below = (1u << lane) - 1u;
    volatile int* const I = W.item;
    float4* const sh = W.shift;
    double (*const fl)[32] = W.f;
    int unit = w * (int)gridDim.x + (int)blockIdx.x;
    while (unit < n_units) {
        __syncwarp();
        const RowItem& item = row_item(P, unit / ENVD_SEG);
        if (lane < 8) I[lane] = reinterpret_cast<const int*>(&item)[lane];
        __syncwarp();
        const int rep = P.rep_of_cl[I[0]];
        const RepDev& R = P.reps[rep];
        const float4 c = P.xq[I[0] * CL];
        row_shifts(R, c, lane, sh);
        if (lane < CL) {
            const float4 x = P.xq[I[0] * CL + lane];
            W.p[lane] = make_float4(x.x - c.x, x.y - c.y, x.z - c.z, 0.f);
            Atom<double> ai = load_atom<double>(P, I[0] * CL + lane, R, K);
            ai.x -= (double)c.x;
            ai.y -= (double)c.y;
            ai.z -= (double)c.z;
            W.i[lane] = ai;
        }
#pragma unroll
        for (int q = 0; q < 3 * CL; ++q) fl[q][lane] = 0.0;
        __syncwarp();
        const int n = (I[3] & 0xFFFF) + (I[3] >> 16) + I[4] + I[5];
        const int part = (n + ENVD_SEG - 1) / ENVD_SEG;
        int next = (unit % ENVD_SEG) * part;
        const int end = min(n, next + part);
        unsigned int mask = 0u;   // pairs of this lane's row still to do
        int ja = 0;
        Atom<double> a{};
        T3<double> fj{0.0, 0.0, 0.0};
        double elj = 0.0, ec = 0.0;
        for (;;) {
            const unsigned int need = __ballot_sync(FULL, mask == 0u);
            if (next < end) {
                if (__popc(need) >= ENVD_REFILL) {
                    const int k = next + __popc(need & below);
                    if (mask == 0u && k < end) {
                        unsigned int word, em;
                        env_tail_row(P, I, k, word, em);
                        ja = (int)(word & ROW_SLOT_MASK);
                        const int code = (int)(word >> ROW_SLOT_BITS);
                        const float4 u = sh[code], v = sh[32 + code], x = P.xq[ja];
                        const float px = (x.x + u.x) - v.x, py = (x.y + u.y) - v.y, pz = (x.z + u.z) - v.z;
#pragma unroll
                        for (int ii = 0; ii < CL; ++ii) {
                            const float4 p = W.p[ii];
                            const float dx = px - p.x, dy = py - p.y, dz = pz - p.z;
                            mask |= fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < near2 ? 1u << ii : 0u;
                        }
                        mask &= ~em;
                        if (mask) {
                            a = load_atom<double>(P, ja, R, K);
                            a.x = ((double)x.x + (double)u.x) - (double)v.x;
                            a.y = ((double)x.y + (double)u.y) - (double)v.y;
                            a.z = ((double)x.z + (double)u.z) - (double)v.z;
                            fj = T3<double>{0.0, 0.0, 0.0};
                        }
                    }
                    next += __popc(need);
                }
            } else if (need == FULL) {
                break;
            }
            if (mask) {
                const int ii = __ffs(mask) - 1;
                mask &= mask - 1u;
                const Atom<double> ai = W.i[ii];
                const double dx = a.x - ai.x, dy = a.y - ai.y, dz = a.z - ai.z;
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                if (r2 < K.rc2) {
                    double r, rinv, rinv2, e, d;
                    root_acc(r2, r, rinv, rinv2);
                    erfc_table(K.beta * r, K.dtab, e, d);
                    const double qq = ai.q * a.q;
                    const double vc = qq * e * rinv;
                    const double fcr = fma(-(qq * K.beta), d, vc);   // Coulomb force times r^2
                    const double sig = ai.sh + a.sh;
                    const double s2 = sig * sig * rinv2;
                    const double s6 = s2 * s2 * s2;
                    const double es = ai.e2 * a.e2 * s6;
                    const double fs = fma(es, fma(12.0, s6, -6.0), fcr) * rinv2;
                    fl[3 * ii][lane] = fma(-fs, dx, fl[3 * ii][lane]);
                    fl[3 * ii + 1][lane] = fma(-fs, dy, fl[3 * ii + 1][lane]);
                    fl[3 * ii + 2][lane] = fma(-fs, dz, fl[3 * ii + 2][lane]);
                    fj.x = fma(fs, dx, fj.x);
                    fj.y = fma(fs, dy, fj.y);
                    fj.z = fma(fs, dz, fj.z);
                    elj += fma(es, s6, -es);
                    ec += vc;
                }
                if (mask == 0u) {
                    red_nonzero(P.fx + ja, fj.x);
                    red_nonzero(P.fy + ja, fj.y);
                    red_nonzero(P.fz + ja, fj.z);
                }
            }
        }
        __syncwarp();
        // i forces: lane v sums value v = 3 ii + c over the warp's lanes
        if (lane < 3 * CL) {
            double s = 0.0;
#pragma unroll 8
            for (int l = 0; l < 32; ++l) s += fl[lane][(l + lane) & 31];
            const int cc = lane % 3;
            red_nonzero((cc == 0 ? P.fx : (cc == 1 ? P.fy : P.fz)) + I[0] * CL + lane / 3, s);
        }
        const double sl = warp_sum<double>(elj);
        const double sc = warp_sum<double>(ec);
        if (lane == 0) {
            if (!isfinite(sl) || !isfinite(sc)) set_err(P.cnt, ERRB_NONFINITE, rep);
            add_fixed(P.eacc + (size_t)rep * EA_N + EA_ENV_LJ, to_fixed_d(sl));
            add_fixed(P.eacc + (size_t)rep * EA_N + EA_ENV_C, to_fixed_d(sc));
        }
        if (nw >= n_units) break;
        if (lane == 0) unit = nw + atomicAdd(&P.cnt->env_next, 1);
        unit = __shfl_sync(FULL, unit, 0);
    }
}

// ------------------------------------------------------------------ ligand pair
template <typename T>
struct LigState {
    T lq, lv, A, dA, cs, dcs;
    bool soft;
};

template <typename T>
__device__ __forceinline__ void pair_lig(const Atom<T>& ai, const Atom<T>& aj, bool keep,
                                         const LigState<T>& S, T3<T>& fi, T3<T>& fj, T& elj,
                                         T& ec, T& dv, T& dq, const KC<T>& K) {
    const T dx = aj.x - ai.x, dy = aj.y - ai.y, dz = aj.z - ai.z;
    const T r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    keep = keep && (r2 < K.rc2);
    // (FP64: 64 cycles of its pipe per instruction, so a vote pays)
    if (sizeof(T) == 8 && !__any_sync(FULL, keep)) return;
    T r, rinv, rinv2;
    root_acc(r2, r, rinv, rinv2);
    const T qq = ai.q * aj.q;
    T erfcv, ex;
    ewald_acc(r, r2, K, erfcv, ex);
    const T u1 = qq * erfcv * rinv;
    const T f1 = fma(qq * K.tbsp, ex, u1) * rinv2;
    const T sig = ai.sh + aj.sh;
    const T eps4 = ai.e2 * aj.e2;
    const T sig2 = sig * sig;
    const T sig6 = sig2 * sig2 * sig2;
    T ulj, flj, dudl;
    if (S.soft) {
        // Beutler: s6 = A sig^6 + r^6, A = alpha (1 - lambda)^p
        const T r4 = r2 * r2;
        const T s6 = fma(S.A, sig6, r4 * r2);
        const T inv = t_rcp_acc(s6);
        const T a = sig6 * inv;
        const T g = eps4 * fma(a, a, -a);
        const T dg = eps4 * fma((T)-2 * a, a, a) * inv;   // d g / d s6
        ulj = S.lv * g;
        flj = -S.lv * dg * (T)6 * r4;
        dudl = fma(S.lv * dg, S.dA * sig6, g);
    } else {
        const T s2 = sig2 * rinv2;
        const T s6 = s2 * s2 * s2;
        ulj = eps4 * fma(s6, s6, -s6);
        flj = eps4 * s6 * fma((T)12, s6, (T)-6) * rinv2;
        dudl = (T)0;
    }
    const T fs = keep ? fma(S.cs, f1, flj) : (T)0;
    fi.x = fma(-fs, dx, fi.x); fi.y = fma(-fs, dy, fi.y); fi.z = fma(-fs, dz, fi.z);
    fj.x = fma(fs, dx, fj.x);  fj.y = fma(fs, dy, fj.y);  fj.z = fma(fs, dz, fj.z);
    elj += keep ? ulj : (T)0;
    ec += keep ? S.cs * u1 : (T)0;
    dv += keep ? dudl : (T)0;
    dq += keep ? S.dcs * u1 : (T)0;
}

template <typename T>
__device__ __forceinline__ LigState<T> lig_state(const DevPtrs& P, const RepDev& R, int jlig);
template <>
__device__ __forceinline__ LigState<float> lig_state<float>(const DevPtrs& P, const RepDev& R,
                                                            int jlig) {
    LigState<float> S;
    S.lq = R.lam_q; S.lv = R.lam_v; S.A = R.sc_A; S.dA = R.sc_dA;
    const bool dec = P.ligand_mode == 1;
    S.soft = !(jlig && dec);
    if (!jlig) { S.cs = S.lq; S.dcs = 1.f; }
    else if (!dec) { S.cs = S.lq * S.lq; S.dcs = 2.f * S.lq; }
    else { S.cs = 1.f; S.dcs = 0.f; }
    return S;
}
template <>
__device__ __forceinline__ LigState<double> lig_state<double>(const DevPtrs& P, const RepDev& R,
                                                              int jlig) {
    LigState<double> S;
    S.lq = R.dlam_q; S.lv = R.dlam_v; S.A = R.dsc_A; S.dA = R.dsc_dA;
    const bool dec = P.ligand_mode == 1;
    S.soft = !(jlig && dec);
    if (!jlig) { S.cs = S.lq; S.dcs = 1.0; }
    else if (!dec) { S.cs = S.lq * S.lq; S.dcs = 2.0 * S.lq; }
    else { S.cs = 1.0; S.dcs = 0.0; }
    return S;
}

// The entries of a ligand item, 32 at a time: lane l holds entry base + l (and
// its exclusion mask), so that the loop over entries takes them by shuffles and
// the j atoms of the next entry can be loaded ahead.
struct LigEntries {
    int2 e;
    unsigned long long m;
    __device__ __forceinline__ void load(const DevPtrs& P, const Item& I, int base, int lane) {
        const int t = base + lane;
        e = make_int2(0, 0);
        m = 0ull;
        if (t < I.e_cnt) {
            e = P.entries[I.e_begin + t];
        } else if (t < I.e_cnt + I.x_cnt) {
            const int k = I.x_begin + (t - I.e_cnt);
            e = P.xentries[k];
            m = P.xmasks[(size_t)k * GMAX];
        }
    }
};

// Latency bound (a few hundred pairs per window): a warp's first item is its own
// index (no claim), the entries are loaded together and the j atoms one entry
// ahead. In FP64 an item's entries are dealt to LIGD_SEG warps.
template <typename T, bool ENERGY>
__global__ void __launch_bounds__(128) k_lig(DevPtrs P) {
    const int lane = threadIdx.x & 31, jj = lane & 7, ii = lane >> 3;
    const KC<T> K = make_kc<T>(P);
    constexpr int SEG = sizeof(T) == 8 ? LIGD_SEG : 1;
    const int n_items = P.ilig_pref[P.R] * SEG;
    const int nw = (int)gridDim.x * 4;
    int it = (threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x;
    while (it < n_items) {
        const Item I = P.items_lig[region_index(P.ilig_pref, P.ilig_base, P.R, it / SEG)];
        const RepDev& R = P.reps[I.rep];
        const int a0 = I.c0 * CL + ii;
        // coordinates relative to the cluster's first atom (see rel_img)
        const float4 c = P.xq[I.c0 * CL];
        Atom<T> ai0 = load_atom<T>(P, a0, R, K);
        Atom<T> ai1 = load_atom<T>(P, a0 + 4, R, K);
        ai0.x -= (T)c.x; ai0.y -= (T)c.y; ai0.z -= (T)c.z;
        ai1.x -= (T)c.x; ai1.y -= (T)c.y; ai1.z -= (T)c.z;
        T3<T> fi0{(T)0, (T)0, (T)0}, fi1{(T)0, (T)0, (T)0};
        double acc[6] = {0, 0, 0, 0, 0, 0};
        const int ntot = I.e_cnt + I.x_cnt;
        LigEntries L;
        Atom<T> aj_n{};
        for (int t = it % SEG, b = -1; t < ntot; t += SEG) {
            if ((t & ~31) != b) {
                b = t & ~31;
                L.load(P, I, b, lane);
                aj_n = load_atom<T>(P, __shfl_sync(FULL, L.e.x, t & 31) * CL + jj, R, K);
            }
            const int2 e = make_int2(__shfl_sync(FULL, L.e.x, t & 31), __shfl_sync(FULL, L.e.y, t & 31));
            const unsigned long long m = __shfl_sync(FULL, L.m, t & 31);
            Atom<T> aj = aj_n;
            if (((t + SEG) & ~31) == b && t + SEG < ntot)
                aj_n = load_atom<T>(P, __shfl_sync(FULL, L.e.x, (t + SEG) & 31) * CL + jj, R, K);
            const int jlig = entry_jlig(e.y);
            const LigState<T> S = lig_state<T>(P, R, jlig);
            float sx, sy, sz;
            entry_shift(e.y, R.box[0], R.box[1], R.box[2], sx, sy, sz);
            const int ja = e.x * CL + jj;
            aj.x = rel_img<T>((float)aj.x, sx, c.x);
            aj.y = rel_img<T>((float)aj.y, sy, c.y);
            aj.z = rel_img<T>((float)aj.z, sz, c.z);
            const bool k0 = !((m >> (ii * 8 + jj)) & 1ull);
            const bool k1 = !((m >> ((ii + 4) * 8 + jj)) & 1ull);
            T3<T> fj{(T)0, (T)0, (T)0};
            T elj = 0, ec = 0, dv = 0, dq = 0;
            pair_lig<T>(ai0, aj, k0, S, fi0, fj, elj, ec, dv, dq, K);
            pair_lig<T>(ai1, aj, k1, S, fi1, fj, elj, ec, dv, dq, K);
            red_jforce<T>(P, ja, ii, fj);
            if (ENERGY) {
                acc[jlig ? 1 : 0] += (double)elj;
                acc[jlig ? 3 : 2] += (double)ec;
                acc[4] += (double)dv;
                acc[5] += (double)dq;
            }
        }
        red_iforce<T>(P, I.c0 * CL, ii, jj, fi0, fi1);
        if (ENERGY) {
            const int slot_map[6] = {EA_LIGENV_LJ, EA_LIGLIG_LJ, EA_LIGENV_C, EA_LIGLIG_C, EA_DUDLV,
                                     EA_DUDLQ};
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const double s = warp_sum<double>(acc[q]);
                if (lane == 0) {
                    if (!isfinite(s)) set_err(P.cnt, ERRB_NONFINITE, I.rep);
                    if (s != 0.0)
                        add_fixed(P.eacc + (size_t)I.rep * EA_N + slot_map[q], to_fixed_d(s));
                }
            }
        }
        if (nw >= n_items) break;
        if (lane == 0) it = nw + atomicAdd(&P.cnt->lig_next, 1);
        it = __shfl_sync(FULL, it, 0);
    }
}

// ------------------------------------------------------------------ u_kn
constexpr int UKN_WARPS = 2;

template <typename T>
__global__ void __launch_bounds__(UKN_WARPS * 32) k_lig_ukn(DevPtrs P) {
    __shared__ T s_acc[UKN_WARPS][KV_MAX][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, jj = lane & 7, ii = lane >> 3;
    const KC<T> K = make_kc<T>(P);
    const int n_items = P.ilig_pref[P.R];
    const bool dec = P.ligand_mode == 1;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(&P.cnt->lig_next, 1);
        it = __shfl_sync(FULL, it, 0);
        if (it >= n_items) break;
        const Item I = P.items_lig[region_index(P.ilig_pref, P.ilig_base, P.R, it)];
        const RepDev& R = P.reps[I.rep];
        const int kv = R.kv;
        const float* kvl = P.kv_lam + R.sched * KV_MAX;
        const float* kva = P.kv_A + R.sched * KV_MAX;
        const double* kvld = P.kv_dlam + R.sched * KV_MAX;
        const double* kvad = P.kv_dA + R.sched * KV_MAX;
        for (int k = 0; k < kv; ++k) s_acc[w][k][lane] = (T)0;
        const int a0 = I.c0 * CL + ii;
        // coordinates relative to the cluster's first atom (see rel_img)
        const float4 c = P.xq[I.c0 * CL];
        Atom<T> ai[2] = {load_atom<T>(P, a0, R, K), load_atom<T>(P, a0 + 4, R, K)};
        for (int h = 0; h < 2; ++h) {
            ai[h].x -= (T)c.x; ai[h].y -= (T)c.y; ai[h].z -= (T)c.z;
        }
        double c_le = 0.0, c_ll = 0.0;
        const int ntot = I.e_cnt + I.x_cnt;
        for (int t = 0; t < ntot; ++t) {
            const bool xm = t >= I.e_cnt;
            const int k = xm ? I.x_begin + (t - I.e_cnt) : I.e_begin + t;
            const int2 e = xm ? P.xentries[k] : P.entries[k];
            const unsigned long long m = xm ? P.xmasks[(size_t)k * GMAX] : 0ull;
            const int jlig = entry_jlig(e.y);
            float sx, sy, sz;
            entry_shift(e.y, R.box[0], R.box[1], R.box[2], sx, sy, sz);
            const int ja = e.x * CL + jj;
            Atom<T> aj = load_atom<T>(P, ja, R, K);
            aj.x = rel_img<T>((float)aj.x, sx, c.x);
            aj.y = rel_img<T>((float)aj.y, sy, c.y);
            aj.z = rel_img<T>((float)aj.z, sz, c.z);
            const bool soft = !(jlig && dec);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool keep0 = !((m >> ((ii + 4 * h) * 8 + jj)) & 1ull);
                const T dx = aj.x - ai[h].x, dy = aj.y - ai[h].y, dz = aj.z - ai[h].z;
                const T r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                const bool keep = keep0 && (r2 < K.rc2);
                if (keep) {
                    T r, rinv, rinv2;
                    root_acc(r2, r, rinv, rinv2);
                    T erfcv, ex;
                    ewald_acc(r, r2, K, erfcv, ex);
                    const double u1 = (double)(ai[h].q * aj.q * erfcv * rinv);
                    if (!jlig) c_le += u1;
                    else if (!dec) c_ll += u1;
                    if (soft) {
                        const T sig = ai[h].sh + aj.sh;
                        const T eps4 = ai[h].e2 * aj.e2;
                        const T sig2 = sig * sig;
                        const T sig6 = sig2 * sig2 * sig2;
                        const T r6 = r2 * r2 * r2;
                        for (int q = 0; q < kv; ++q) {
                            const T lam = (sizeof(T) == 4) ? (T)kvl[q] : (T)kvld[q];
                            const T A = (sizeof(T) == 4) ? (T)kva[q] : (T)kvad[q];
                            const T a = sig6 * t_rcp_acc(fma(A, sig6, r6));
                            s_acc[w][q][lane] += lam * eps4 * fma(a, a, -a);
                        }
                    }
                }
            }
        }
        __syncwarp();
        for (int q = lane; q < kv; q += 32) {
            double s = 0.0;
            for (int l = 0; l < 32; ++l) s += (double)s_acc[w][q][l];
            if (!isfinite(s)) set_err(P.cnt, ERRB_NONFINITE, I.rep);
            if (s != 0.0) add_fixed(P.ukn_lj + (size_t)I.rep * KV_MAX + q, to_fixed_d(s));
        }
        const double sle = warp_sum<double>(c_le), sll = warp_sum<double>(c_ll);
        if (lane == 0) {
            if (sle != 0.0) add_fixed(P.ukn_c + (size_t)I.rep * 2 + 0, to_fixed_d(sle));
            if (sll != 0.0) add_fixed(P.ukn_c + (size_t)I.rep * 2 + 1, to_fixed_d(sll));
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ pair counting
// Environment pairs through the inner rows (the list the force kernel walks), in the
// FP32 force kernel's lane layout (lane per row, 32 rows per round, plain then masked
// rows); the pairs that kernel evaluates for the item go to pair_cnt[2 R] in units of
// 32, for the lane efficiency: all eight i atoms for each lane of every round, half rows
// and the idle lanes of the last round included.
__global__ void __launch_bounds__(128) k_count_rows(DevPtrs P) {
    const int lane = threadIdx.x & 31;
    const int n_items = P.ritem_pref[P.R];
    const int stride = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += stride) {
        const RowItem I = row_item(P, it);
        const int rep = P.rep_of_cl[I.c];
        const RepDev& R = P.reps[rep];
        int cnt = 0;
        const int n_full = I.cnt & 0xFFFF, n_lo_end = n_full + I.n_lo;
        const int n_plain = n_lo_end + I.n_hi, n = n_plain + (I.cnt >> 16);
        for (int k0 = 0; k0 < n; k0 += 32) {
            const int k = k0 + lane;
            const bool valid = k < n, masked = k >= n_plain;
            const bool act_lo = valid && (masked || k < n_lo_end);
            const bool act_hi = valid && (masked || k < n_full || k >= n_lo_end);
            if (!valid) continue;
            unsigned int word, em = 0u;
            if (masked) {
                const int2 xr = P.xrows[I.x_begin + (k - n_plain)];
                word = (unsigned int)xr.x;
                em = (unsigned int)xr.y;
            } else {
                word = P.rows[I.r_begin + (unsigned int)k];
            }
            const int ja = (int)(word & ROW_SLOT_MASK), code = (int)(word >> ROW_SLOT_BITS);
            float4 xj = P.xq[ja];
            xj.x += (float)(code % 3 - 1) * R.box[0];
            xj.y += (float)((code / 3) % 3 - 1) * R.box[1];
            xj.z += (float)(code / 9 - 1) * R.box[2];
            const bool jreal = P.orig[ja] >= 0;
            for (int ii = 0; ii < CL; ++ii) {
                if (!(ii < 4 ? act_lo : act_hi) || ((em >> ii) & 1u)) continue;
                const int a = I.c * CL + ii;
                const float4 xi = P.xq[a];
                const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (r2 < P.rc2 && jreal && P.orig[a] >= 0) {
                    ++cnt;
                    if (P.atom_cnt) {
                        atomicAdd(&P.atom_cnt[a], 1);
                        atomicAdd(&P.atom_cnt[ja], 1);
                    }
                }
            }
        }
        const int tot = warp_sum<int>(cnt);
        if (lane == 0 && tot)
            atomicAdd(reinterpret_cast<unsigned long long*>(P.pair_cnt + (size_t)rep * 2),
                      (unsigned long long)tot);
        if (lane == 0)
            atomicAdd(reinterpret_cast<unsigned long long*>(P.pair_cnt + (size_t)P.R * 2),
                      (unsigned long long)(CL * ((n + 31) / 32)));
    }
}

// Ligand-involved pairs through the ligand list.
__global__ void __launch_bounds__(128) k_count_lig(DevPtrs P) {
    const int lane = threadIdx.x & 31, jj = lane & 7, ii = lane >> 3;
    const int n_items = P.ilig_pref[P.R];
    const int stride = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_items; it += stride) {
        const Item I = P.items_lig[region_index(P.ilig_pref, P.ilig_base, P.R, it)];
        const RepDev& R = P.reps[I.rep];
        int cnt = 0;
        const int ntot = I.e_cnt + I.x_cnt;
        for (int t = 0; t < ntot; ++t) {
            const bool xm = t >= I.e_cnt;
            const int k = xm ? I.x_begin + (t - I.e_cnt) : I.e_begin + t;
            const int2 e = xm ? P.xentries[k] : P.entries[k];
            float sx, sy, sz;
            entry_shift(e.y, R.box[0], R.box[1], R.box[2], sx, sy, sz);
            const int ja = e.x * CL + jj;
            float4 xj = P.xq[ja];
            xj.x += sx; xj.y += sy; xj.z += sz;
            const bool jreal = P.orig[ja] >= 0;
            for (int g = 0; g < I.ng; ++g) {
                const unsigned long long m = xm ? P.xmasks[(size_t)k * GMAX + g] : 0ull;
                for (int h = 0; h < 2; ++h) {
                    if (!entry_half(e.y, g, h)) continue;
                    const int a = (I.c0 + g) * CL + ii + 4 * h;
                    const float4 xi = P.xq[a];
                    const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
                    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                    const bool keep = !((m >> ((ii + 4 * h) * 8 + jj)) & 1ull) && r2 < P.rc2 &&
                                      jreal && P.orig[a] >= 0;
                    if (keep) {
                        ++cnt;
                        if (P.atom_cnt) {
                            atomicAdd(&P.atom_cnt[a], 1);
                            atomicAdd(&P.atom_cnt[ja], 1);
                        }
                    }
                }
            }
        }
        const int tot = warp_sum<int>(cnt);
        if (lane == 0 && tot)
            atomicAdd(reinterpret_cast<unsigned long long*>(P.pair_cnt + (size_t)I.rep * 2 + 1),
                      (unsigned long long)tot);
    }
}

}  // namespace

// Small systems: at most ENV_SMALL_ITEMS clusters per SM give each scheduler a
// warp or two, whatever the registers allow: there the kernel is bound by one
// warp's latency, and the variant with 255 registers interleaves the eight pairs
// of a row. Both variants add the same bits. Windows of 4,500 atoms (4.2 clusters per
// SM each), us of a step in the graph and of a whole energy pass with 64 | 255
// registers, for 256-thread blocks (items of up to 512 entries) and 128 (up to 64):
//   clusters per SM     4.2         8.3         17          33         66        265
//   step, 256       48.5|46.8   65.0|53.0   71.0|68.7   81.7|85.5   133|141   408|458
//   step, 128       52.4|54.0   58.0|61.5   70.3|74.5   93.5|101    142|155   465|522
//   energy, 256     84.5|80.0    121|89.0    124|105     130|125    206|196   574|592
//   energy, 128     77.2|78.1   97.3|85.4    112|101     144|131    210|192   666|610
// Steps with 256-thread blocks gain up to 17 clusters per SM, with 128 they lose 3 to
// 6%; energy passes gain at both, and on beyond the line.
constexpr int ENV_SMALL_ITEMS = 8;
static bool env_small(const DevPtrs& P, int n_sm) { return P.C <= ENV_SMALL_ITEMS * n_sm; }

static size_t envd_smem(int block) { return sizeof(EnvdWarp) * (size_t)(block / 32); }

cudaError_t env_prepare() {
    return cudaFuncSetAttribute(k_env_rows_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)envd_smem(ENV_WARPS_MAX * 32));
}

void launch_env_forces(const DevPtrs& P, cudaStream_t s, bool energy, int precision, int grid,
                       int block, int n_sm) {
    if (precision == 1) {
        k_env_rows_f64<<<grid, block, envd_smem(block), s>>>(P);
    } else if (env_small(P, n_sm)) {
        if (energy) k_env_rows<true, 1><<<grid, block, 0, s>>>(P);
        else k_env_rows<false, 1><<<grid, block, 0, s>>>(P);
    } else {
        if (energy) k_env_rows<true, 4><<<grid, block, 0, s>>>(P);
        else k_env_rows<false, 4><<<grid, block, 0, s>>>(P);
    }
}

int env_kernel_occupancy(int block, int precision, bool energy) {
    int nb = 0;
    if (precision == 1)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_env_rows_f64, block, envd_smem(block));
    else if (energy)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_env_rows<true, 4>, block, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_env_rows<false, 4>, block, 0);
    return nb;
}

void launch_lig_forces(const DevPtrs& P, cudaStream_t s, int precision, int grid, int block,
                       bool energy) {
    // force steps skip the energy sums (FP64 adds: the FP64 pipe bounds them)
    if (precision == 1) {
        if (energy) k_lig<double, true><<<grid, block, 0, s>>>(P);
        else k_lig<double, false><<<grid, block, 0, s>>>(P);
    } else {
        if (energy) k_lig<float, true><<<grid, block, 0, s>>>(P);
        else k_lig<float, false><<<grid, block, 0, s>>>(P);
    }
}

void launch_lig_ukn(const DevPtrs& P, cudaStream_t s, int grid, int precision) {
    if (precision == 1) k_lig_ukn<double><<<grid, UKN_WARPS * 32, 0, s>>>(P);
    else k_lig_ukn<float><<<grid, UKN_WARPS * 32, 0, s>>>(P);
}

void launch_count_pairs(const DevPtrs& P, cudaStream_t s, int grid, int block) {
    k_count_rows<<<grid, block, 0, s>>>(P);
    k_count_lig<<<grid, block, 0, s>>>(P);
}

}  // namespace abfe
