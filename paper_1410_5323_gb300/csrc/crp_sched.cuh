// crp_sched.cuh -- work distribution for the persistent propagate kernels: a warp refills
// its idle lanes with one claim on a global counter (ballot + popc), first from the fixed
// work list of the launch, then from the list of secondaries pushed during this launch.
// A pushed entry is published with a release store after the particle's state is written;
// a reader claims entries below the push count and waits, bounded, for each to
// appear with an acquire load. A wait that runs out sets a status bit instead of hanging;
// nothing here traps.
#pragma once
#include <cuda/atomic>

#include "crp_internal.h"

namespace crp {

constexpr unsigned kSchedFull = 0xffffffffu;
constexpr int kPublishWaitLimit = 1 << 22;     // iterations of 64 ns sleeps (~0.3 s)
constexpr int kClaimRetryLimit = 64;

__device__ __forceinline__ unsigned long long ld_volatile(const unsigned long long* p) {
    return *(volatile const unsigned long long*)p;
}

// Waits, at most `limit` times 64 ns, for a value other than -1 to be published at p (acquire
// loads). Returns false if it never appeared; the caller turns that into a status bit.
__device__ __forceinline__ bool bounded_acquire_wait(int32_t* p, int limit, int32_t& v) {
    cuda::atomic_ref<int32_t, cuda::thread_scope_device> e(*p);
#pragma unroll 1
    for (int t = 0; t < limit; ++t) {
        v = e.load(cuda::memory_order_acquire);
        if (v != -1) return true;
        __nanosleep(64);
    }
    return false;
}

// Append entry q to work list L.
__device__ __forceinline__ void sched_push(const PropArgs& a, int L, int32_t q) {
    const unsigned long long p = atomicAdd(&a.ctr->count[L], 1ull);
    cuda::atomic_ref<int32_t, cuda::thread_scope_device> e(a.lists[L][p]);
    e.store(q, cuda::memory_order_release);
}

// Entries of a work list: the slot of a particle, or kResumed - slot for one that the previous launch
// of the call handed on; -1: not yet published (the bookkeeping after each launch puts it back).
constexpr int32_t kResumed = -2;

__device__ __forceinline__ void sched_hand_on(const PropArgs& a, int L, int32_t slot) {
    atomicAdd(&a.ctr->handed, 1ull);
    sched_push(a, L, kResumed - slot);
}

template <bool HandedOn>
__device__ __forceinline__ int sched_slot(const PropArgs& a, int32_t v, unsigned& bits, int& resumed) {
    if (HandedOn && v <= kResumed && a.taken) {
        v = kResumed - v;
        resumed = 1;
    }
    if (v < 0 || v >= a.capacity) { bits |= BIT_BOUNDS; return -1; }
    return v;
}

// What a launch works through: list L from position head0 (entries before it were taken by the
// previous launch) to n_work. A list that a launch filled ends with the particles it handed on, which are
// in mid-flight: as many entries as those, from the end, come first, then the secondaries in the order in
// which they were released, lowest rigidities first. (All from the end, with the longest secondaries
// last, 10^6 nuclei over 500 Mpc took 7.50 s instead of 7.04.)
struct WorkList {
    int L;
    unsigned long long from_end, n_work, head0;
    __device__ __forceinline__ bool fits(const PropArgs& a) const {
        const long long n = (long long)(n_work - head0);
        return n > a.min_work && n <= a.max_work;
    }
};
__device__ __forceinline__ WorkList work_list(const PropArgs& a) {
    const Counters* C = a.ctr;
    const int L = *(volatile const int*)&C->cur;
    return {L, ld_volatile(&C->handed0), ld_volatile(&C->count[L]), ld_volatile(&C->head0)};
}

// Returns the slot this lane should load next from the work list, or -1. Lanes with idle == false
// get -1. dry (the same in all lanes) turns true once the list has run out for good. HandedOn: the list may
// hold particles handed on (FP64 form; the precision kernels have no registers to spare for them).
template <bool HandedOn>
__device__ __forceinline__ int sched_pop(const PropArgs& a, const WorkList& W, bool idle, int lane, unsigned& bits,
                                        bool& dry, int& resumed) {
    const unsigned im = __ballot_sync(kSchedFull, idle);
    if (!im) return -1;
    Counters* C = a.ctr;
    unsigned long long base = 0;
    unsigned got = 0, out = 0;
    if (lane == 0) {
        const unsigned need = (unsigned)__popc(im);
        if (ld_volatile(&C->head[W.L]) < W.n_work) {
            base = atomicAdd(&C->head[W.L], (unsigned long long)need);
            if (base < W.n_work) got = (unsigned)min((unsigned long long)need, W.n_work - base);
        }
        out = got < need;
    }
    base = __shfl_sync(kSchedFull, base, 0);
    got = __shfl_sync(kSchedFull, got, 0);
    dry = __shfl_sync(kSchedFull, out, 0);
    if (!idle) return -1;
    const unsigned rank = (unsigned)__popc(im & ((1u << lane) - 1u));
    if (rank >= got) return -1;
    unsigned long long pos = base + rank;
    if constexpr (HandedOn) {
        const unsigned long long k = pos - W.head0;
        pos = k < W.from_end ? W.n_work - 1 - k : pos - W.from_end;
    }
    return sched_slot<HandedOn>(a, a.lists[W.L][pos], bits, resumed);
}

// Whether idle lanes look for pushed secondaries in this turn of the one-lane kernels: every few turns,
// with CRP_PICKUP_ON once the list has run out. The look is a round trip to L2, and with thousands of warps
// asking it is the counters' line that everyone waits for (10^6 nuclei in the precision form: 73 ms without
// pick-ups; 265, 114, 81, 66 ms looking every 1, 4, 16, 64 turns. 10^5 nuclei in the modulated scenario: 65 ms
// without, 44 to 47 ms with). So that form's warps look every 32 turns, each in a turn of its own (20 000
// nuclei over at most 200 steps 4.4 ms all at once, 2.7 so), and every 4 once the list has run out, where
// lanes without a particle have nothing else to do (200 000 nuclei, 2 Mpc between interactions, over 6 Mpc:
// 9.2 ms every 128 turns, 4.5 every 32, 3.8 every 4).
// The FP64 form, whose turns take ten times as long, looks every 4 (200 000 nuclei: 284 ms without,
// 247 ms, 267 ms looking every 32).
//
// Where too many secondaries wait, the next launch takes them: it fills its lanes without asking for each.
// In the precision form that is three times the lanes for lists that don't fill the lanes (30 000 iron
// nuclei 3.4 ms without a limit, 2.4 with it; 19 000 in one block per SM 5.3 and 1.5), and no limit for longer
// lists, whose tail the secondaries fill (10^6 nuclei over 500 Mpc 396 ms; 420 with the limit, the secondaries'
// own tail behind the nuclei's); in the FP64 form, whose tail other launches take, the lanes or teams.
template <unsigned Every, unsigned Dry>
__device__ __forceinline__ bool sched_look(const PropArgs& a, bool dry, unsigned turn) {
    return a.pickup && (dry ? turn % Dry == 0 : (a.pickup == 2 && turn % Every == 0));
}

// The same from list P, into which this launch pushes secondaries only: claims positions below the push
// count, then waits, bounded, for the entries to be published. The claim is a semaphore (Counters::claimed):
// add what is wanted, keep what the count covers, give the rest back, and take that many positions at the
// head, which so never passes the count. No claim fails because another one came first: with a CAS on the
// head one warp won per round trip, 30 entries a microsecond (100 000 nuclei as above, looking every 32 turns,
// 4.6 -> 2.6 ms).
__device__ __forceinline__ int sched_pick(const PropArgs& a, int P, unsigned long long n_work, bool idle, int lane,
                                         unsigned& bits) {
    const unsigned im = __ballot_sync(kSchedFull, idle);
    if (!im) return -1;
    Counters* C = a.ctr;
    unsigned long long base = 0;
    unsigned got = 0;
    if (lane == 0) {
        const unsigned long long c = ld_volatile(&C->count[P]), lanes = (unsigned long long)gridDim.x * blockDim.x;
        const bool fills = n_work - ld_volatile(&C->head0) > lanes;
        unsigned long long taken = ld_volatile(&C->claimed);
        if (taken < c && (fills || c - taken <= 3 * lanes)) {
            const unsigned long long want = min((unsigned long long)__popc(im), c - taken);
            taken = atomicAdd(&C->claimed, want);
            got = taken < c ? (unsigned)min(want, c - taken) : 0u;
            if (got < want) atomicAdd(&C->claimed, got - want);
            if (got) base = atomicAdd(&C->head[P], (unsigned long long)got);
        }
    }
    base = __shfl_sync(kSchedFull, base, 0);
    got = __shfl_sync(kSchedFull, got, 0);
    if (!idle) return -1;
    const unsigned rank = (unsigned)__popc(im & ((1u << lane) - 1u));
    if (rank >= got) return -1;
    int32_t v = -1;
    if (!bounded_acquire_wait(a.lists[P] + base + rank, kPublishWaitLimit, v)) {
        bits |= BIT_TIMEOUT;   // the entry never appeared: reported by crp_sync
        return -1;
    }
    int resumed = 0;
    return sched_slot<false>(a, v, bits, resumed);
}

// The same where the list also receives particles handed on to the next launch (FP64 form). The warp
// reads the entries at the head, waiting (bounded) for each to be published, and claims the secondaries
// before the first particle handed on. So no particle is handed on twice in one launch, which bounds the
// length of the list (list_length). In the precision form, where all warps ask the same counters, this
// costs 5 % (10^6 nuclei 65.4 ms claiming first, 68.8 ms reading first); the FP64 form shows no difference.
__device__ __forceinline__ int sched_pick_secondaries(const PropArgs& a, int P, unsigned long long room, bool idle, int lane,
                                                     unsigned& bits) {
    const unsigned im = __ballot_sync(kSchedFull, idle);
    if (!im) return -1;
    Counters* C = a.ctr;
#pragma unroll 1
    for (int t = 0; t < kClaimRetryLimit; ++t) {
        unsigned long long h = 0;
        unsigned n = 0;
        if (lane == 0) {
            h = ld_volatile(&C->head[P]);
            const unsigned long long c = ld_volatile(&C->count[P]);
            if (h < c && c - h <= room) n = (unsigned)min((unsigned long long)__popc(im), c - h);
        }
        n = __shfl_sync(kSchedFull, n, 0);
        if (n == 0) return -1;
        h = __shfl_sync(kSchedFull, h, 0);
        int32_t v = -1;
        if ((unsigned)lane < n && !bounded_acquire_wait(a.lists[P] + h + lane, kPublishWaitLimit, v))
            bits |= BIT_TIMEOUT;   // the entry never appeared: reported by crp_sync
        const unsigned stop = __ballot_sync(kSchedFull, (unsigned)lane >= n || v < 0);
        const unsigned take = stop ? (unsigned)__ffs((int)stop) - 1u : 32u;
        if (take == 0) return -1;
        unsigned won = 0;
        if (lane == 0) won = atomicCAS(&C->head[P], h, h + take) == h;
        if (!__shfl_sync(kSchedFull, won, 0)) continue;
        __syncwarp();              // what a lane acquired is visible to the one that takes the entry
        const unsigned rank = (unsigned)__popc(im & ((1u << lane) - 1u));
        v = __shfl_sync(kSchedFull, v, (int)(rank & 31u));
        if (!idle || rank >= take) return -1;
        if (v >= a.capacity) { bits |= BIT_BOUNDS; return -1; }
        return v;
    }
    return -1;
}

}  // namespace crp
