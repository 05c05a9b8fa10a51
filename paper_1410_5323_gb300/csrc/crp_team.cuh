// crp_team.cuh -- three lanes per particle: the FP64 arithmetic of crp_fp64.cuh split over a team.
//
// GB300 issues one FP64 warp instruction per 64 cycles per SM sub-partition, however many of its
// lanes are active, so a trajectory's time is the number of FP64 instructions that its lane
// issues. A team of three lanes (lanes 3t, 3t + 1, 3t + 2; ten teams per warp) shares one
// particle: lane c owns component c of the position and direction, of every stage state and of
// every stage derivative, forms axis c of each lookup, a share of the corner weights, B_c and the
// c-th Lorentz component. Every value is formed by the operations of the one-lane form in their
// order, so the results are the same bits. All lanes of a warp run these functions together
// (shuffles over the whole warp); lanes without a particle compute on whatever they hold.
#pragma once
#include "crp_fp64.cuh"

namespace crp {
namespace team {

using namespace fp64;

constexpr int kTeams = kTeamsPerWarp;   // ten; lanes 30 and 31 belong to none

struct Lane {
    int l0, c, l2;                  // the team's first lane, this lane's component, the team's last lane
    __device__ __forceinline__ double get(double v, int k) const { return __shfl_sync(kFull, v, k == 2 ? l2 : l0 + k); }
    __device__ __forceinline__ int get(int v, int k) const { return __shfl_sync(kFull, v, k == 2 ? l2 : l0 + k); }
    __device__ __forceinline__ int nx1() const { return c == 2 ? 0 : c + 1; }
    __device__ __forceinline__ int nx2() const { return c == 0 ? 2 : c - 1; }
};

__device__ __forceinline__ Lane lane_of_team() {
    const int lane = threadIdx.x & 31, t = lane / 3;
    return {3 * t, lane - 3 * t, min(3 * t + 2, 31)};
}

// Axis c of one periodic grid (FP64 vector node copy, or the FP32 modulation grid).
struct Axis {
    double inv, oi;                 // 1/spacing, origin (1/spacing) rounded once
    int n, stride, pow2;            // nodes along the axis, distance of neighbours in nodes
};

__device__ __forceinline__ Axis vector_axis(const FieldDev& F, int c) {
    return {F.inv_spacing, c == 0 ? F.oix : (c == 1 ? F.oiy : F.oiz), c == 0 ? F.nx : (c == 1 ? F.ny : F.nz),
            c == 0 ? F.ny * F.nz : (c == 1 ? F.nz : 1), F.pow2};
}
__device__ __forceinline__ Axis modulation_axis(const FieldDev& F, int c) {
    return {F.m_inv_spacing, c == 0 ? F.moix : (c == 1 ? F.moiy : F.moiz), c == 0 ? F.mnx : (c == 1 ? F.mny : F.mnz),
            c == 0 ? F.mny * F.mnz : (c == 1 ? F.mnz : 1), F.mpow2};
}
// The axis of lanes without a particle (lanes 30 and 31 exchange values with each other alone): node 0
// whatever the position, and a grid coordinate of 1, which takes the common path of the lookup.
__device__ __forceinline__ Axis parked_axis() { return {0.0, -1.0, 1, 0, 1}; }

// Nodes and weights of the 8 corners (000, 001, ..., 111) around the team's position, whose
// coordinate c this lane holds.
struct Corners {
    int node[8];
    double w[8];
};

template <bool P2>
__device__ __forceinline__ Corners corners(const Axis& A, const Lane& T, double xc) {
    const double r = __fma_rn(xc, A.inv, -A.oi);
    long long i;
    double w0, w1;
    floor_weights(r, i, w0, w1);
    int i0;
    if (P2 || A.pow2) {
        i0 = (int)i & (A.n - 1);
    } else if (i == (long long)(int)i) {      // the 32-bit remainder is a third of the 64-bit one
        i0 = (int)i % A.n;
        if (i0 < 0) i0 += A.n;
    } else {
        i0 = (int)(i % A.n);
        if (i0 < 0) i0 += A.n;
    }
    const int o0 = i0 * A.stride, o1 = (i0 + 1 == A.n ? 0 : i0 + 1) * A.stride;
    const int x0 = T.get(o0, 0), x1 = T.get(o1, 0), y0 = T.get(o0, 1), y1 = T.get(o1, 1), z0 = T.get(o0, 2),
              z1 = T.get(o1, 2);
    const double wx1 = T.get(w1, 0), wy0 = T.get(w0, 1), wy1 = T.get(w1, 1), wz0 = T.get(w0, 2), wz1 = T.get(w1, 2);
    // lane 0 forms w00, w01 and corners 0..3, lane 1 w10, w11 and corners 4..7 (lane 2 repeats lane 1)
    const double wx = T.c == 0 ? w0 : wx1;
    const double a = wx * wy0, b = wx * wy1;
    const double a0 = a * wz0, a1 = a * wz1, b0 = b * wz0, b1 = b * wz1;
    return {{x0 + y0 + z0, x0 + y0 + z1, x0 + y1 + z0, x0 + y1 + z1, x1 + y0 + z0, x1 + y0 + z1, x1 + y1 + z0,
             x1 + y1 + z1},
            {T.get(a0, 0), T.get(a1, 0), T.get(b0, 0), T.get(b1, 0), T.get(a0, 1), T.get(a1, 1), T.get(b0, 1),
             T.get(b1, 1)}};
}

// The corner sum in the stated order, each corner added with one rounding from 0.
__device__ __forceinline__ double corner_sum(const double (&w)[8], const double (&g)[8]) {
    double B = __fma_rn(w[0], g[0], 0.0);
#pragma unroll
    for (int k = 1; k < 8; ++k) B = __fma_rn(w[k], g[k], B);
    return B;
}

// B_c at the team's position: data is the node copy shifted to component c (node k at 4k).
template <bool P2>
__device__ __forceinline__ double field_c(const double* data, const Axis& A, const Lane& T, double xc) {
    const Corners q = corners<P2>(A, T, xc);
    double g[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = __ldg(data + 4ll * q.node[k]);
    return corner_sum(q.w, g);
}

// The modulation value at the team's position (the same in its three lanes).
__device__ __forceinline__ double modulation_t(const float* mod, const Axis& A, const Lane& T, double xc) {
    const Corners q = corners<false>(A, T, xc);
    double g[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) g[k] = widen_f32(__ldg(mod + q.node[k]));
    return corner_sum(q.w, g);
}

// Component c of kappa u x B: kappa fma(u_{c+1}, B_{c+2}, -(u_{c+2} B_{c+1})).
__device__ __forceinline__ double force_c(const Lane& T, double kappa, double yu, double B) {
    const double u1 = T.get(yu, T.nx1()), u2 = T.get(yu, T.nx2());
    const double B1 = T.get(B, T.nx1()), B2 = T.get(B, T.nx2());
    return kappa * __fma_rn(u1, B2, -(u2 * B1));
}

// One Cash-Karp attempt of size h from (yx, yu) with the direction derivative k1u at the start;
// deriv(x, u) gives the direction derivative at a stage state.
template <typename Deriv>
__device__ __forceinline__ void attempt_c(double h, double yx, double yu, double k1u, const Deriv& deriv, double& y5x,
                                          double& y5u, double& ex, double& eu) {
    const double k1x = yu;
    double tx, tu;
    tx = __fma_rn(h, A21 * k1x, yx); tu = __fma_rn(h, A21 * k1u, yu);
    const double k2x = tu, k2u = deriv(tx, tu);
#define T3(k) __fma_rn(A32, k2##k, A31 * k1##k)
    tx = __fma_rn(h, T3(x), yx); tu = __fma_rn(h, T3(u), yu);
    const double k3x = tu, k3u = deriv(tx, tu);
#define T4(k) __fma_rn(A43, k3##k, __fma_rn(A42, k2##k, A41 * k1##k))
    tx = __fma_rn(h, T4(x), yx); tu = __fma_rn(h, T4(u), yu);
    const double k4x = tu, k4u = deriv(tx, tu);
#define T5(k) __fma_rn(A54, k4##k, __fma_rn(A53, k3##k, __fma_rn(A52, k2##k, A51 * k1##k)))
    tx = __fma_rn(h, T5(x), yx); tu = __fma_rn(h, T5(u), yu);
    const double k5x = tu, k5u = deriv(tx, tu);
#define T6(k) __fma_rn(A65, k5##k, __fma_rn(A64, k4##k, __fma_rn(A63, k3##k, __fma_rn(A62, k2##k, A61 * k1##k))))
    tx = __fma_rn(h, T6(x), yx); tu = __fma_rn(h, T6(u), yu);
    const double k6x = tu, k6u = deriv(tx, tu);
#define TB(k) __fma_rn(B6, k6##k, __fma_rn(B4, k4##k, __fma_rn(B3, k3##k, B1 * k1##k)))
#define TE(k) (h * __fma_rn(E6, k6##k, __fma_rn(E5, k5##k, __fma_rn(E4, k4##k, __fma_rn(E3, k3##k, E1 * k1##k)))))
    y5x = __fma_rn(h, TB(x), yx); y5u = __fma_rn(h, TB(u), yu);
    ex = TE(x); eu = TE(u);
#undef T3
#undef T4
#undef T5
#undef T6
#undef TB
#undef TE
}

// Squared norms ((e0^2 + e1^2) + e2^2) of the error with fused products, as error_sums.
__device__ __forceinline__ void error_sums_t(const Lane& T, double ex, double eu, double& sx, double& su) {
    const double x0 = T.get(ex, 0), x1 = T.get(ex, 1), x2 = T.get(ex, 2);
    const double u0 = T.get(eu, 0), u1 = T.get(eu, 1), u2 = T.get(eu, 2);
    sx = __fma_rn(x2, x2, __fma_rn(x1, x1, x0 * x0));
    su = __fma_rn(u2, u2, __fma_rn(u1, u1, u0 * u0));
}

}  // namespace team
}  // namespace crp
