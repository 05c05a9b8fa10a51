// sources.cu -- Sec. 4 sources (Eq. 1 spectrum, isotropic emission) and arrival maps (Fig. 4:
// HEALPix maps of arrival directions). Compiled with --fmad=false: every expression is
// evaluated as written, so species, energies, directions and pixel indices are identical to
// the FP64 reading.
#include <cuda_runtime.h>

#include "crp.h"
#include "crp_internal.h"
#include "crp_math.cuh"
#include "crp_sky.cuh"

// Runs of this file's kernels (diagnostics: each launch adds one, from its first thread).
namespace {
__device__ unsigned long long g_kernel_runs = 0;
}

namespace crp {
namespace {

// U = (m + 1/2) 2^-52 from 52 random bits m, exactly, with integer instructions: (2m + 1) 2^-53.
__device__ __forceinline__ double uniform_words(uint32_t hi, uint32_t lo) {
    const unsigned long long G = 2ull * (((unsigned long long)hi << 20) | (unsigned long long)(lo >> 12)) + 1ull;
    const int z = __clzll((long long)G);               // 11 .. 63
    return __longlong_as_double(((long long)(1033 - z) << 52) | (long long)((G << (z - 11)) & 0xFFFFFFFFFFFFFull));
}
// The same to within 2^-23.
__device__ __forceinline__ float uniform_f32(uint32_t hi) { return __uint2float_rn(hi) * 0x1p-32f; }

__device__ __forceinline__ U4 words(unsigned long long seed, unsigned long long uid, uint32_t k,
                                    uint32_t tag) {
    return philox10((uint32_t)uid, (uint32_t)(uid >> 32), k, tag, (uint32_t)seed, (uint32_t)(seed >> 32));
}

// Constants of the spectrum, the same for every particle: formed once per block, one power per lane
// of its first warp. (Formed by every thread they were most of the kernel's FP64 work.)
struct SpectrumConsts {
    double cum[CRP_MAX_SPECIES];   // cumulative species weights x_i A_i^(alpha-1)
    double W, g, lo, hi, lr;       // inverse-CDF constants of E^-alpha
    // the same in FP32: hi / lo, 1 / g, lr log2 e, E_min / R_cut; flat: alpha is 1
    float cum_f[CRP_MAX_SPECIES], W_f, ratio, inv_g, lr2, q0;
    int flat;
};

__device__ __forceinline__ void spectrum_consts(const crp_spectrum& sp, SpectrumConsts& K) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const double g = 1.0 - sp.alpha;
        // exp(c log v): lanes 0 .. 7 A_i^(alpha-1), lanes 8 and 9 e_min^g and e_max^g
        const double v = lane < 8 ? (double)sp.A[lane < sp.n_species ? lane : 0] : (lane == 8 ? sp.e_min_ev : sp.e_max_ev);
        const double e = crp_exp((lane < 8 ? sp.alpha - 1.0 : g) * crp_log(v));
        const double w = lane < sp.n_species ? sp.x[lane] * e : 0.0;
        double acc = 0.0;
        for (int i = 0; i < sp.n_species; ++i) {
            acc = acc + __shfl_sync(0xffffffffu, w, i);
            if (lane == 0) {
                K.cum[i] = acc;
                K.cum_f[i] = (float)acc;
            }
        }
        const double lo = __shfl_sync(0xffffffffu, e, 8), hi = __shfl_sync(0xffffffffu, e, 9);
        if (lane == 0) {
            K.W = acc;
            K.g = g;
            K.lo = g != 0.0 ? lo : 0.0;
            K.hi = g != 0.0 ? hi : 0.0;
            K.lr = g != 0.0 ? 0.0 : crp_log(sp.e_max_ev / sp.e_min_ev);
            // below the normal FP32 numbers the sums' roundings are coarser than the margins: decided in FP64
            K.W_f = acc > 1e-30 ? (float)acc : __int_as_float(0x7fc00000);
            K.ratio = (float)(hi / lo);
            K.inv_g = (float)(1.0 / g);
            K.lr2 = (float)(K.lr * 1.4426950408889634);
            K.q0 = (float)(sp.e_min_ev / sp.rcut_v);
            K.flat = g == 0.0;
        }
    }
    __syncthreads();
}

// Energy of the uniform number u2 by the inverse CDF.
__device__ __forceinline__ double energy_of(const SpectrumConsts& K, const crp_spectrum& sp, double u2) {
    return !K.flat ? crp_exp(crp_log(K.lo + u2 * (K.hi - K.lo)) / K.g) : sp.e_min_ev * crp_exp(u2 * K.lr);
}

// Species of a draw's first number, and whether the draw is kept, u3 < exp(-E / (Z R_cut)): decided
// in FP32 where that is certain, by the FP64 expressions elsewhere, so that a draw that is rejected (or
// a warp that draws again for some of its lanes) costs no FP64 instructions. Bounds: the uniform
// numbers are off by at most 2^-23; t = 1 + u2 (hi/lo - 1) by dt, E = E_min t^(1/g) relatively by
// dt / t / |g| and the FP32 logarithm and power (2^-20 |y| for the exponent y); the margin is twice
// what follows for exp(-q). Anything not finite is uncertain.
__device__ __forceinline__ bool draw_kept(const SpectrumConsts& K, const crp_spectrum& sp, const U4& w, const U4& v, int& s) {
    const float target = uniform_f32(w.a) * K.W_f;
    s = sp.n_species - 1;
    bool sure = true;
    for (int i = sp.n_species - 1; i >= 0; --i) {
        const float c = K.cum_f[i];
        if (target < c) s = i;
        sure = sure && fabsf(target - c) > 1e-6f * K.W_f;
    }
    if (!sure) {
        const double t = uniform_words(w.a, w.b) * K.W;
        s = sp.n_species - 1;
        for (int i = 0; i < sp.n_species; ++i)
            if (t < K.cum[i]) { s = i; break; }
    }
    const float u2 = uniform_f32(w.c), u3 = uniform_f32(v.a);
    float y, dy;      // log2(E / E_min) and the bound of its error
    if (!K.flat) {
        const float t = fmaf(u2, K.ratio - 1.0f, 1.0f);
        const float dt = 4e-7f * (1.0f + K.ratio);
        y = __log2f(t) * K.inv_g;
        dy = 1.5f * (dt / t + 1e-6f) * fabsf(K.inv_g) + 2e-6f * (1.0f + fabsf(y));
        if (!(t > 4.0f * dt)) dy = __int_as_float(0x7f800000);
    } else {
        y = u2 * K.lr2;
        dy = 4e-7f * K.lr2 + 2e-6f * (1.0f + fabsf(y));
    }
    const float q = K.q0 / (float)sp.Z[s] * exp2f(y);                       // E / (Z R_cut)
    const float p = __expf(-q);
    const float margin = 2.0f * (p * (q * (dy + 4e-6f) + 1e-5f) + 4e-7f);
    const float d = u3 - p;
    if (dy < 0.1f && fabsf(d) > margin) return d < 0.0f;
    const double en = energy_of(K, sp, uniform_words(w.c, w.d));
    return uniform_words(v.a, v.b) < crp_exp(-en / ((double)sp.Z[s] * sp.rcut_v));
}

// One draw per particle and thread. Per particle: species and energy from Eq. 1 by rejection
// from the cutoff-free joint law, then an isotropic direction (Marsaglia 1972). The draws are tried in
// FP32 and only the one that is kept is evaluated in FP64, whose issue bounds the kernel: 10^6
// particles of the Sec. 4 spectrum 1286 us with everything in FP64 and the spectrum's constants
// formed by every thread, 201 us so.
__global__ void __launch_bounds__(128) k_source_sample(SimState S, long long first, long long n,
                                                       unsigned long long uid_base, crp_spectrum sp,
                                                       unsigned long long seed) {
    CRP_COUNT_RUN();
    __shared__ SpectrumConsts K;
    spectrum_consts(sp, K);
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const long long slot = first + p;
        const unsigned long long uid = uid_base + (unsigned long long)p;
        int a = 0, z = 0;
        double e = 0.0;
        U4 kept{0, 0, 0, 0};
        int s = -1;
        for (uint32_t k = 0; k < CRP_SOURCE_DRAWS; ++k) {
            const U4 w = words(seed, uid, k, 2u);
            int sk;
            if (draw_kept(K, sp, w, words(seed, uid, k, 3u), sk)) {
                kept = w;
                s = sk;
                break;
            }
        }
        bool have_dir = false;
        U4 dir{0, 0, 0, 0};
        for (uint32_t k = 0; k < CRP_SOURCE_DRAWS; ++k) {
            dir = words(seed, uid, k, 4u);
            // inside the unit circle? v1^2 + v2^2 in FP32 is off by less than 2e-6
            const float f1 = 2.0f * uniform_f32(dir.a) - 1.0f, f2 = 2.0f * uniform_f32(dir.c) - 1.0f;
            const float r2 = fmaf(f1, f1, f2 * f2);
            if (fabsf(r2 - 1.0f) > 4e-6f) {
                have_dir = r2 < 1.0f;
            } else {
                const double v1 = 2.0 * uniform_words(dir.a, dir.b) - 1.0, v2 = 2.0 * uniform_words(dir.c, dir.d) - 1.0;
                have_dir = v1 * v1 + v2 * v2 < 1.0;
            }
            if (have_dir) break;
        }
        if (s >= 0) {
            a = sp.A[s];
            z = sp.Z[s];
            e = energy_of(K, sp, uniform_words(kept.c, kept.d));
        }
        double dx = 0.0, dy = 0.0, dz = 0.0;
        if (have_dir) {
            const double v1 = 2.0 * uniform_words(dir.a, dir.b) - 1.0, v2 = 2.0 * uniform_words(dir.c, dir.d) - 1.0;
            const double s2 = v1 * v1 + v2 * v2;
            const double r = 2.0 * sqrt(1.0 - s2);
            dx = v1 * r;
            dy = v2 * r;
            dz = 1.0 - 2.0 * s2;
        } else {
            a = 0;
            z = 0;      // A = 0: flagged invalid by the injection kernel
        }
        S.uid[slot] = (long long)uid;
        S.A[slot] = a;
        S.Z[slot] = z;
        S.E[slot] = e;
        S.ux[slot] = dx;
        S.uy[slot] = dy;
        S.uz[slot] = dz;
    }
}

__global__ void k_healpix(int nside, const double* __restrict__ u, long long n, long long* __restrict__ pix) {
    CRP_COUNT_RUN();
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x)
        pix[k] = sky::healpix_pixel(nside, u[3 * k], u[3 * k + 1], u[3 * k + 2]);
}

// Arrival map over the used slots. With `shared`, each block counts into a shared copy of
// the map (12 nside^2 32-bit counters) and adds its non-zero pixels to the global map once.
__global__ void k_arrival_map(SimState S, const Counters* C, int nside, double e_min, int shared,
                              unsigned long long* __restrict__ map) {
    CRP_COUNT_RUN();
    extern __shared__ unsigned int smap[];
    const long long npix = 12ll * nside * nside;
    if (shared) {
        for (long long q = threadIdx.x; q < npix; q += blockDim.x) smap[q] = 0u;
        __syncthreads();
    }
    const long long n = (long long)C->n_used;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        if (S.status[i] != CRP_STATUS_DONE_ || !(S.E[i] > e_min)) continue;
        const long long p = sky::healpix_pixel(nside, -S.ux[i], -S.uy[i], -S.uz[i]);
        if (p < 0 || p >= npix) continue;
        if (shared) atomicAdd(&smap[p], 1u);
        else atomicAdd(&map[p], 1ull);
    }
    if (shared) {
        __syncthreads();
        for (long long q = threadIdx.x; q < npix; q += blockDim.x)
            if (smap[q]) atomicAdd(&map[q], (unsigned long long)smap[q]);
    }
}

}  // namespace

int launch_source_sample(const SimState& S, long long first, long long n, unsigned long long uid_base,
                         const crp_spectrum& sp, unsigned long long seed, int grid, void* stream) {
    k_source_sample<<<grid, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(S, first, n, uid_base, sp, seed);
    return (int)cudaGetLastError();
}

int launch_healpix(int nside, const double* u, long long n, long long* pix, int grid, void* stream) {
    k_healpix<<<grid, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(nside, u, n, pix);
    return (int)cudaGetLastError();
}

int launch_arrival_map(const SimState& S, const Counters* C, int nside, double e_min,
                       unsigned long long* map, int grid, void* stream) {
    const long long npix = 12ll * nside * nside;
    const bool shared = npix * 4 <= 48 * 1024;
    k_arrival_map<<<grid, 256, shared ? (size_t)npix * 4 : 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        S, C, nside, e_min, shared ? 1 : 0, map);
    return (int)cudaGetLastError();
}

}  // namespace crp

namespace crp {
unsigned long long kernel_runs_sources() {
    unsigned long long v = 0;
    if (cudaMemcpyFromSymbol(&v, g_kernel_runs, sizeof v) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}
}  // namespace crp
