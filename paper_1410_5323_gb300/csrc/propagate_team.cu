// propagate_team.cu -- FP64 form of the propagation in teams of three lanes per particle
// (arXiv:1410.5323, Sec. 3.1 module sequence): the module sequence of propagate_fp64.cu, value for
// value, for batches and remainders of batches that do not fill the one-lane kernel.
//
// Why: the FP64 unit takes a warp instruction per 64 cycles per sub-partition whatever its active
// lanes, so one lane per particle spends ~600 of them on an attempt (23 us measured, alone on its
// sub-partition) however few particles there are; a team issues ~185 (9 us). What belongs to the whole
// particle (rates, bids, step size, energy loss) is formed by the same operations in all three
// lanes, which costs large batches with tables a fifth, so those start in the one-lane kernel.
// Measured (times per call, start of the comparison in the one-lane kernel alone): 1024 protons over
// 100 Mpc 8.4 -> 3.9 ms; 20 000 protons 13.6 -> 9.7 ms; 3000 nuclei with tables 153 -> 48 ms; as the
// last launches of 200 000 nuclei 363 -> 244 ms.
//
// A call runs the one-lane kernel on work lists of more entries than it has lanes (38 912 here); when
// its list has run out and half of its lanes are empty it hands its particles on. Lists of more than three
// particles for each team of one block per SM (18 240) go to this kernel with several blocks per SM, which
// hands on once one block per SM can hold what is left, and the rest runs with one block per SM to the end:
// warps that share a sub-partition share its FP64 unit.
#include <cuda_runtime.h>

#include "crp_internal.h"
#include "crp_math.cuh"
#include "crp_sched.cuh"
#include "crp_team.cuh"

// Runs of this file's kernels (diagnostics: each launch adds one, from its first thread).
namespace {
__device__ unsigned long long g_kernel_runs = 0;
}

namespace crp {
namespace {

using namespace team;

template <bool M, bool P2>
__global__ void __launch_bounds__(256, M ? 1 : 2) k_propagate_fp64_team(const PropArgs a) {
    CRP_COUNT_RUN();
    const int lane = threadIdx.x & 31;
    const Lane T = lane_of_team();
    const bool mine = lane < 3 * kTeams, first = mine && T.c == 0;
    Counters* C = a.ctr;
    const WorkList work = work_list(a);
    const int pushes = 1 - work.L;
    if (!work.fits(a)) return;
    // fewer particles than teams: evenly over the warps
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    const int quota = (int)min((unsigned long long)kTeams, (work.n_work - work.head0 + warps - 1) / warps);
    const double INF = __longlong_as_double(0x7ff0000000000000LL);
    const SimState& S = a.st;

    int slot = -1, gid = 0;
    double yx = 0.0, yu = 0.0, k1u = 0.0;
    double E = 0, s = 0, hprop = 0, tau = 0;
    int A = 0, Z = 0, n_int = 0;
    unsigned long long uid = 0;
    long long taken = 0, taken0 = 0;          // accepted steps of this call, and of this launch's start
    unsigned n_att = 0;
    const double* data = nullptr;             // node copy of the particle's field, shifted to component c
    Axis V = parked_axis(), W = parked_axis();
    const float* mod = nullptr;
    bool new_step = true, dry = false;
    double h = 0, h_first = 0, h_propc = 0, h_int = 0, h_dist = 0, rl = 0, rpd = 0, kappa = 0;
    const double tol2 = a.tol * a.tol;
    const float lg_tol = ctrl_log2(a.tol);
    int rejected = 0;
    unsigned att_step = 0;
    unsigned long long acc_tot = 0, att_tot = 0, sec_tot = 0;
    unsigned bits = 0;

    auto col3 = [&](double* x, double* y, double* z) { return T.c == 0 ? x : (T.c == 1 ? y : z); };
    auto set_field = [&](int g) {
        const FieldDev& F = a.fields[g];
        data = static_cast<const double*>(F.data) + T.c;
        V = vector_axis(F, T.c);
        if constexpr (M) {
            mod = F.mod;
            W = modulation_axis(F, T.c);
        }
    };
    auto deriv = [&](double x, double u) {
        double B = field_c<P2>(data, V, T, x);
        if constexpr (M) B = modulation_t(mod, W, T, x) * B;
        return force_c(T, kappa, u, B);
    };
    auto store = [&](int status) {
        col3(S.x, S.y, S.z)[slot] = yx;
        col3(S.ux, S.uy, S.uz)[slot] = yu;
        if (T.c == 0) {
            S.E[slot] = E; S.s[slot] = s; S.hprop[slot] = hprop; S.tau[slot] = tau;
            S.A[slot] = A; S.Z[slot] = Z; S.n_int[slot] = n_int; S.status[slot] = status;
            S.n_steps[slot] = __ldcg(&S.n_steps[slot]) + (taken - taken0);
            S.n_att[slot] = __ldcg(&S.n_att[slot]) + n_att;
            if (status != CRP_STATUS_ACTIVE_) {
                const unsigned long long d = atomicAdd(&C->n_done, 1ull);
                a.done_list[d] = slot;
            }
            if (a.drain) atomicAdd(&C->left, 1ull);
        }
        slot = -1;
    };

    data = static_cast<const double*>(a.fields[0].data);   // lanes without a particle look up its first node
    if constexpr (M) mod = a.fields[0].mod;
    bool drain = false;
    for (unsigned turn = 0;; ++turn) {
        // ---- refill idle teams from the work list, then with secondaries pushed by this launch ----
        const bool pick = a.pickup && !drain && turn % 4 == 0;
        if ((!dry && !drain) || pick) {
            int p0 = -1, resumed = 0;
            if (pick) p0 = sched_pick_secondaries(a, pushes, warps * kTeams, first && slot < 0, lane, bits);
            if (!dry && !drain) {
                const int p = sched_pop<true>(a, work, first && slot < 0 && p0 < 0 && lane < 3 * quota, lane, bits, dry, resumed);
                if (p >= 0) p0 = p;
            }
            const int popped = T.get(p0, 0);
            resumed = T.get(resumed, 0);
            __syncwarp();   // what lane 0 acquired is visible to its team
            if (mine && slot < 0 && popped >= 0) {
                slot = popped;
                yx = __ldcg(col3(S.x, S.y, S.z) + slot); yu = __ldcg(col3(S.ux, S.uy, S.uz) + slot);
                E = __ldcg(&S.E[slot]); s = __ldcg(&S.s[slot]); hprop = __ldcg(&S.hprop[slot]); tau = __ldcg(&S.tau[slot]);
                A = __ldcg(&S.A[slot]); Z = __ldcg(&S.Z[slot]); n_int = __ldcg(&S.n_int[slot]); gid = __ldcg(&S.grid_id[slot]);
                uid = (unsigned long long)__ldcg(&S.uid[slot]);
                taken0 = taken = resumed ? __ldcg(&a.taken[slot]) : 0;
                n_att = 0;
                new_step = true;
                if (gid < 0 || gid >= a.n_fields) {
                    bits |= BIT_BOUNDS;
                    gid = 0;
                    slot = -1;
                } else {
                    set_field(gid);
                    kappa = (double)Z * kC / E;
                }
            }
            __syncwarp();
        }
        if (a.drain && dry && !drain && turn % 8 == 7) {   // few enough for one warp per sub-partition?
            long long left = lane == 0 ? (long long)(work.n_work - work.head0 + ld_volatile(&C->head[pushes]) -
                                                     ld_volatile(&C->left)) : 0ll;
            left = __shfl_sync(kFull, left, 0);
            drain = left <= a.drain_at;
        }
        if (drain) {
            if (slot >= 0 && new_step) {      // the next launch resumes it here
                const int32_t q = slot;
                if (T.c == 0) a.taken[q] = (int32_t)taken;
                store(CRP_STATUS_ACTIVE_);
                if (T.c == 0) sched_hand_on(a, pushes, q);
            }
            __syncwarp();
        }
        if (!__any_sync(kFull, slot >= 0)) break;

        // ---- bids (Sec. 3.1): lowest of propagation, loss, interaction, distance ----
        if (slot >= 0 && new_step) {
            float rl_f = 0.0f, rpd_f = 0.0f;
            if (a.has_tables && !table_rates_f32(a.tab, A, Z, E, rl_f, rpd_f)) {
                bits |= BIT_RANGE;
                store(CRP_STATUS_RANGE_);
            } else {
                rl = rl_f > 0.0f ? widen_normal(rl_f) : 0.0;
                rpd = rpd_f > 0.0f ? widen_normal(rpd_f) : 0.0;
                h_propc = clampd(hprop, a.hmin, a.hmax);
                const double h_loss = rl_f > 0.0f ? widen_f32(__fdiv_rn(0.1f, rl_f)) : INF;
                h_int = rpd_f > 0.0f ? widen_f32(__fdiv_rn(__double2float_rn(fmax(tau, 0.0)), rpd_f)) : INF;
                h_dist = a.dmax - s;
                h = h_propc;
                if (lt_pos(h_loss, h)) h = h_loss;
                if (lt_pos(h_int, h)) h = h_int;
                if (dbits(h_dist) < dbits(h)) h = h_dist;   // h_dist is never -0
                h_first = h;
                rejected = 0;
                att_step = 0;
            }
        }
        __syncwarp();

        // ---- propagation: one Cash-Karp attempt, all teams together ----
        if (__any_sync(kFull, slot >= 0 && new_step)) {
            const double k1n = deriv(yx, yu);
            if (new_step) {          // rejected attempts reuse k1
                k1u = k1n;
                new_step = false;
            }
        }
        double y5x, y5u, ex, eu, sx, su;
        attempt_c(h, yx, yu, k1u, deriv, y5x, y5u, ex, eu);
        error_sums_t(T, ex, eu, sx, su);
        auto fin = [](double v) { return ((unsigned long long)dbits(v) >> 52 & 0x7FFu) != 0x7FFu; };
        const unsigned finite = __ballot_sync(kFull, fin(y5x) && fin(y5u)) >> T.l0;
        if (slot < 0) continue;
        att_step += 1;
        const bool accept = error_accept(sx, su, h, a.tol, tol2) || le_pos(h, a.hmin);
        const double hnew = h * widen_normal(step_factor(accept, sx, su, h, lg_tol));
        if (!accept) {
            h = max_pos(hnew, a.hmin);
            rejected = 1;
            continue;
        }
        if ((finite & 7u) != 7u) {
            n_att += att_step;
            att_tot += att_step;
            bits |= BIT_NAN;
            store(CRP_STATUS_NAN_);
            continue;
        }
        const bool fires = (dbits(rpd) > 0 && eq_num(h, h_int));
        unsigned long long q = 0;
        if (fires) {
            if (T.c == 0) q = atomicAdd(&C->reserve, 1ull);
            q = __shfl_sync(7u << T.l0, q, T.l0);
            if (q >= (unsigned long long)a.capacity) {
                bits |= BIT_QUEUE_FULL;      // parked at the start of this step
                store(CRP_STATUS_ACTIVE_);
                continue;
            }
        }
        // ---- accept ----
        n_att += att_step;
        att_tot += att_step;
        yx = y5x;
        yu = y5u;
        if (a.boundary) {   // reflective box: fold this axis, flip u (and u0) if odd
            const double lo = T.c == 0 ? a.box_lo[0] : (T.c == 1 ? a.box_lo[1] : a.box_lo[2]);
            const double hi = T.c == 0 ? a.box_hi[0] : (T.c == 1 ? a.box_hi[1] : a.box_hi[2]);
            const double len = T.c == 0 ? a.box_len[0] : (T.c == 1 ? a.box_len[1] : a.box_len[2]);
            const double inv = T.c == 0 ? a.box_inv[0] : (T.c == 1 ? a.box_inv[1] : a.box_inv[2]);
            if (reflect_axis(yx, lo, hi, len, inv)) {
                double* u0 = col3(S.u0x, S.u0y, S.u0z) + slot;
                yu = -yu;
                *u0 = -*u0;
            }
        }
        const bool done = eq_num(h, h_dist);
        s = done ? a.dmax : s + h;
        acc_tot += 1;
        taken += 1;
        double hnext = hnew;
        if (!rejected && lt_pos(h_first, h_propc)) hnext = max_pos(hnext, h_propc);
        hprop = clampd(hnext, a.hmin, a.hmax);
        // ---- continuous loss at gamma0 ----
        if (dbits(rl) > 0) E = E * crp_exp(-h * rl);
        // ---- photo-disintegration ----
        if (dbits(rpd) > 0) {
            if (fires) {
                const unsigned kk = (unsigned)(n_int + 1);
                const int dz = nucleon_proton(a.seed, uid, kk, A, Z) ? 1 : 0;
                const double E_sec = E / (double)A;
                const double E_par = E * (double)(A - 1) / (double)A;
                const long long qs = (long long)q;
                const unsigned long long uid2 = (1ull << 32) + uid * 64ull + kk;
                col3(S.x, S.y, S.z)[qs] = yx;
                col3(S.ux, S.uy, S.uz)[qs] = yu;
                double* u0 = col3(S.u0x, S.u0y, S.u0z);
                u0[qs] = u0[slot];
                __syncwarp(7u << T.l0);      // the secondary's columns are written before it is listed
                if (T.c == 0) {
                    S.E[qs] = E_sec; S.s[qs] = s;
                    S.hprop[qs] = INF;
                    S.tau[qs] = -crp_log(uniform01(a.seed, uid2, 0u, 0u));
                    S.A[qs] = 1; S.Z[qs] = dz; S.n_int[qs] = 0; S.grid_id[qs] = gid;
                    S.uid[qs] = (long long)uid2;
                    S.n_steps[qs] = 0; S.n_att[qs] = 0;
                    S.status[qs] = done ? CRP_STATUS_DONE_ : CRP_STATUS_ACTIVE_;
                    if (done) {
                        const unsigned long long d = atomicAdd(&C->n_done, 1ull);
                        a.done_list[d] = (int32_t)qs;
                    } else {
                        sched_push(a, pushes, (int32_t)qs);
                    }
                    sec_tot += 1;
                }
                A = A - 1;
                Z = Z - dz;
                E = E_par;
                n_int = (int)kk;
                tau = -crp_log(uniform01(a.seed, uid, kk, 0u));
            } else {
                tau = tau - h * rpd;
            }
        }
        new_step = true;
        if (dbits(rl) > 0 || fires) kappa = (double)Z * kC / E;   // else neither E nor Z changed
        // ---- observer ----
        if (done) {
            store(CRP_STATUS_DONE_);
        } else if (a.max_steps > 0 && taken >= a.max_steps) {
            store(CRP_STATUS_ACTIVE_);
        }
    }

    // ---- statistics: one lane per team counts, warp reduction, one atomic per warp ----
    if (!first) acc_tot = att_tot = sec_tot = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc_tot += __shfl_xor_sync(kFull, acc_tot, o);
        att_tot += __shfl_xor_sync(kFull, att_tot, o);
        sec_tot += __shfl_xor_sync(kFull, sec_tot, o);
        bits |= __shfl_xor_sync(kFull, bits, o);
    }
    if (lane == 0) {
        if (acc_tot) atomicAdd(&C->accepted, acc_tot);
        if (att_tot) atomicAdd(&C->attempted, att_tot);
        if (sec_tot) atomicAdd(&C->secondaries, sec_tot);
        if (bits) atomicOr(&C->status_bits, bits);
    }
}

template <typename Fn>
int with_team_kernel(int mod, int p2, Fn&& fn) {
    if (mod) return p2 ? fn(k_propagate_fp64_team<true, true>) : fn(k_propagate_fp64_team<true, false>);
    return p2 ? fn(k_propagate_fp64_team<false, true>) : fn(k_propagate_fp64_team<false, false>);
}

}  // namespace

// one_per_sm: shared memory that only one block of an SM finds room for. Warps that share a
// sub-partition share its FP64 unit, and blocks are not dealt out evenly over SMs that have room for
// several: 1024 protons over 100 Mpc took 4.5 ms with up to four blocks on some SMs and none on others.
int launch_propagate_team(const PropArgs& a, int mod, int p2, int grid, int block, int one_per_sm, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int shm = one_per_sm ? kOnePerSmBytes : 0;
    return with_team_kernel(mod, p2, [&](void (*k)(const PropArgs)) {
        if (shm) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, shm);
            if (e != cudaSuccess) return (int)e;
        }
        k<<<grid, block, shm, st>>>(a);
        return (int)cudaGetLastError();
    });
}

int propagate_team_occupancy(int mod, int p2, int block, int* blocks_per_sm) {
    return with_team_kernel(mod, p2, [&](void (*k)(const PropArgs)) {
        return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, block, 0);
    });
}

unsigned long long kernel_runs_team() {
    unsigned long long v = 0;
    if (cudaMemcpyFromSymbol(&v, g_kernel_runs, sizeof v) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}

}  // namespace crp
