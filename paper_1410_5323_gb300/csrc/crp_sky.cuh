// crp_sky.cuh -- directions on the sky: atan2 by one stated algorithm and the HEALPix RING
// pixelization (Gorski et al. 2005), shared by the arrival-map and lens kernels. Translation
// units including it are compiled with --fmad=false, so pixel indices are those of the FP64
// reading.
#pragma once
#include <cuda_runtime.h>

namespace crp {
namespace sky {

constexpr double kPi = 3.141592653589793;
constexpr double kHalfPi = 1.5707963267948966;
constexpr double kQuarterPi = 0.7853981633974483;
constexpr double kTanPi8 = 0.41421356237309503;
constexpr int kFastNside = 512;

// atan2 by the stated reduction: octant, tan(pi/8) split, half-angle step, Taylor series.
__device__ __forceinline__ double atan2_stated(double y, double x) {
    if (x != x || y != y) return __longlong_as_double(0x7ff8000000000000LL);
    const double ax = fabs(x), ay = fabs(y);
    if (ax == 0.0 && ay == 0.0) return 0.0;
    const bool swap = ay > ax;
    const double a = swap ? ax / ay : ay / ax;
    double base = 0.0, b = a;
    if (a > kTanPi8) {
        b = (a - 1.0) / (a + 1.0);
        base = kQuarterPi;
    }
    const double c = b / (1.0 + sqrt(1.0 + b * b));
    const double s = c * c;
    double p = -1.0 / 27.0;
    p = p * s + 1.0 / 25.0;
    p = p * s - 1.0 / 23.0;
    p = p * s + 1.0 / 21.0;
    p = p * s - 1.0 / 19.0;
    p = p * s + 1.0 / 17.0;
    p = p * s - 1.0 / 15.0;
    p = p * s + 1.0 / 13.0;
    p = p * s - 1.0 / 11.0;
    p = p * s + 1.0 / 9.0;
    p = p * s - 1.0 / 7.0;
    p = p * s + 1.0 / 5.0;
    p = p * s - 1.0 / 3.0;
    p = p * s + 1.0;
    double r = base + 2.0 * (c * p);
    if (swap) r = kHalfPi - r;
    if (x < 0.0) r = kPi - r;
    if (y < 0.0) r = -r;
    return r;
}

// HEALPix RING pixel (Gorski et al. 2005): belt |z| <= 2/3 from the edge-line indices
// jp = floor(nside (t - 3z/4 + 1/2)), jm = floor(nside (t + 3z/4 + 1/2)); caps from the
// equal-area radius sigma = nside sqrt(3 (1 - |z|)). t = phi / (pi/2) in [0, 4).
__device__ __forceinline__ long long healpix_ring(int nside, double x, double y, double z) {
    const double r = sqrt(x * x + y * y + z * z);
    if (!(r > 0.0) || !isfinite(r)) return -1;
    const double zz = z / r;
    double phi = atan2_stated(y, x);
    if (phi < 0.0) phi = phi + 2.0 * kPi;
    double t = phi / kHalfPi;
    if (t >= 4.0) t = t - 4.0;
    const long long ns = nside;
    const double dn = (double)nside;
    const double az = fabs(zz);
    if (az <= 2.0 / 3.0) {
        const double sg = 0.75 * zz;
        const long long jp = (long long)floor(dn * (t - sg + 0.5));
        const long long jm = (long long)floor(dn * (t + sg + 0.5));
        long long i = 2 * ns - (jm - jp);
        if (i < ns) i = ns;
        if (i > 3 * ns) i = 3 * ns;
        const long long s = (i - ns + 1) & 1;
        long long j = (jp + jm + 1 - ns - s) / 2;
        const long long m = 4 * ns;
        j = ((j % m) + m) % m;
        return 2 * ns * (ns - 1) + m * (i - ns) + j;
    }
    const double tp = t - floor(t);
    const double sigma = dn * sqrt(3.0 * (1.0 - az));
    long long i = (long long)floor(tp * sigma) + (long long)floor((1.0 - tp) * sigma) + 1;
    if (i > ns) i = ns;
    long long j = (long long)floor(t * (double)i);
    if (j >= 4 * i) j = 4 * i - 1;
    if (zz > 0.0) return 2 * i * (i - 1) + j;
    return 12 * ns * ns - 2 * i * (i + 1) + j;
}

// Leading 24 bits of a double whose exponent a normal float holds, by integer instructions; 0 below
// that range, NaN above it.
__device__ __forceinline__ float head_f32(double v) {
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    const int e = (hi >> 20) & 0x7FF;
    if (e > 1150) return __int_as_float(0x7fc00000);
    return e < 897 ? 0.0f
                   : __int_as_float((hi & (int)0x80000000) | ((e - 896) << 23) | ((hi & 0xFFFFF) << 3) | (int)(lo >> 29));
}

// floor(v) if v is at least `eps` away from the integers.
__device__ __forceinline__ bool sure_floor(float v, float eps, int& i) {
    const float f = floorf(v);
    i = (int)f;
    const float d = v - f;
    return d > eps && d < 1.0f - eps;
}

// healpix_ring decided in FP32, or -2 where that is not certain: within the error of a pixel border, a
// ring border, a meridian k pi/2 or the belt's edge, near a pole, or for directions that are not
// ordinary numbers. Bounds: z/r and phi / (pi/2) are off by less than 1e-6 (inputs 2^-23 relative,
// atan2f 3 ulp of pi, rsqrtf 2 ulp); twice that is used, and the sums' own roundings.
__device__ __forceinline__ int healpix_ring_f32(int ns, double dx, double dy, double dz) {
    if (ns > kFastNside) return -2;
    const float x = head_f32(dx), y = head_f32(dy), z = head_f32(dz);
    const float r2 = fmaf(x, x, fmaf(y, y, z * z));
    if (!(r2 > 1e-20f && r2 < 1e20f)) return -2;
    const float zz = z * rsqrtf(r2);
    float t = atan2f(y, x) * 0.63661977f;
    if (t < 0.0f) t += 4.0f;
    constexpr float e = 2e-6f;
    const float az = fabsf(zz), dn = (float)ns;
    int q;
    if (!sure_floor(t, 4.0f * e, q) || fabsf(az - 0.6666667f) < 4.0f * e) return -2;
    if (az < 0.6666667f) {
        const float sg = 0.75f * zz, eps = dn * 6e-6f;
        int jp, jm;
        if (!sure_floor(dn * (t - sg + 0.5f), eps, jp) || !sure_floor(dn * (t + sg + 0.5f), eps, jm)) return -2;
        int i = 2 * ns - (jm - jp);
        i = max(ns, min(3 * ns, i));
        const int s = (i - ns + 1) & 1, m = 4 * ns;
        int j = (jp + jm + 1 - ns - s) / 2;
        j = j < 0 ? j + m : (j >= m ? j - m : j);
        return 2 * ns * (ns - 1) + m * (i - ns) + j;
    }
    const float h = 1.0f - az;
    if (!(h > 1e-3f)) return -2;
    const float sigma = dn * sqrtf(3.0f * h), tp = t - (float)q;
    const float eps = sigma * 2.0f * e + dn * (2.0f * e / sqrtf(h)) + dn * 1e-6f;
    int i0, i1, j;
    if (!sure_floor(tp * sigma, eps, i0) || !sure_floor((1.0f - tp) * sigma, eps, i1)) return -2;
    const int i = min(i0 + i1 + 1, ns);
    if (!sure_floor(t * (float)i, (float)i * 3.0f * e, j)) return -2;
    if (zz > 0.0f) return 2 * i * (i - 1) + j;
    return 12 * ns * ns - 2 * i * (i + 1) + j;
}

// The pixel, in FP32 where that decides it: the FP64 pixelization is ~130 FP64 instructions at 64
// cycles a warp; one direction in 500 needs it at nside 64 (arrival map of 10^6 particles 308 -> 41 us,
// rigidity-binned maps 343 -> 56 us).
// Its share grows with nside; above kFastNside nearly every warp would have one.
__device__ __forceinline__ long long healpix_pixel(int nside, double x, double y, double z) {
    const int p = healpix_ring_f32(nside, x, y, z);
    return p != -2 ? (long long)p : healpix_ring(nside, x, y, z);
}

}  // namespace sky
}  // namespace crp
