// Pieces shared by the warp-specialised FP64 kernels (redo.cu, quad.cu): the hand-off
// rings between the warps of a block, the view of a planar state that the
// recombination terms take, the root of det Z, where a block's groups come from and
// where a group ends.
#pragma once

#include "traj_block.cuh"

namespace sfhk {
namespace {

// read-only view of the planar state for the recombination terms (q_y = p_y = 0)
struct PView {
    double q[3], p[3];
    struct {
        double s;
        __device__ double reduced() const { return s; }
    } S;
    __device__ PView(double q0, double q2, double p0, double p2, double s) : q{q0, 0.0, q2}, p{p0, 0.0, p2}, S{s} {}
};

// The principal root of D = det Z, m2 = |D|^2, with |D| = sqrt(m2): an eighth of hypot's
// FP64 instructions.  Calls with d_t up to kWarpsDt come here, so |D| of a trajectory that
// stays is at most that and m2 is in range (as are the products of 8 det Z that follow the
// branch).
__device__ __forceinline__ cd root_det(cd D, double m2) {
    const double r = sqrt(m2);
    const double q = sqrt(0.5 * (r + fabs(D.re))), o = positive(q) ? D.im / (2.0 * q) : 0.0;
    return D.re >= 0.0 ? mk(q, o) : mk(fabs(o), copysign(q, D.im));
}

// Hand-offs of N slots between consecutive roles on named barriers (0 is left to
// __syncthreads): barrier base + d is "slot d full", arrived at by the producer and
// waited on by the consumer, base + N + d "slot d empty", the other way round, 64 threads
// each (the two warps).  A role runs ahead of the next by at most N grid points, so
// uneven work per grid point evens out across the pipeline.
// The barrier instructions want the warp converged.
__device__ __forceinline__ void bar_sync64(int id) {
    __syncwarp();
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void bar_arrive64(int id) {
    __syncwarp();
    asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}
template <int N>
struct Producer {
    int base, d;
    bool wrapped;
    int64_t k;
    __device__ explicit Producer(int base_) : base(base_), d(0), wrapped(false), k(0) {}
    __device__ int acquire() {                     // slot for item k, once its item k - N is consumed
        if (wrapped) bar_sync64(base + N + d);
        return d;
    }
    __device__ void publish(int slot) {
        bar_arrive64(base + slot);
        ++k;
        if (++d == N) {
            d = 0;
            wrapped = true;
        }
    }
    __device__ void drain() {                      // the consumer's releases of the last items
        for (int64_t j = (k >= N ? k - N : 0); j < k; ++j) bar_sync64(base + N + (int)(j % N));
    }
};
template <int N>
struct Consumer {
    int base, d;
    __device__ explicit Consumer(int base_) : base(base_), d(0) {}
    __device__ int wait() {
        bar_sync64(base + d);
        return d;
    }
    __device__ void release(int slot) {
        bar_arrive64(base + N + slot);
        if (++d == N) d = 0;
    }
};

// A group runs in stretches of 8 grid points and ends early, at the end of a stretch, when
// the bins warp has removed every trajectory.  The dynamics warp, the first of the chain,
// learns of it from the labels: at the start of a stretch, before it publishes an item of
// it, it marks that stretch as the last one.  The hand-offs order the mark before the items,
// so each warp behind finds it when it is done with the stretch, and all four end on the
// same one.  (Looking at every grid point costs a short list 2 %, nothing this way.)
struct GroupEnd {
    static constexpr int kStretch = 8;
    // grid points of the stretch that starts at n
    static __device__ int stretch(int64_t n, int64_t n_last) {
        return n_last - n + 1 < kStretch ? (int)(n_last - n + 1) : kStretch;
    }
    // by the dynamics warp, converged
    static __device__ void decide(long long& mark, int64_t hi, bool alive) {
        if (!__any_sync(0xffffffffu, alive) && (threadIdx.x & 31) == 0) *(volatile long long*)&mark = hi;
    }
    static __device__ bool here(const long long& mark, int64_t hi) { return *(const volatile long long*)&mark == hi; }
};

__device__ __forceinline__ unsigned sm_id() {
    unsigned r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return r;
}

// Where a block's next group of list entries comes from.  With a plan (redo_plan_kernel):
// the groups of its own SM's list, longest first, then those left on the other lists,
// one atomic counter per list.  A block that finds its own list empty waits 20 us before
// it turns to the others: the blocks of a launch start some microseconds apart, and a
// second block on one SM would take the groups of SMs whose blocks are about to start
// (groups of a short list then piled up on a few SMs: 166 to 220 ms for the same call).
// SM s serves list (s + redo_shift) mod L: launches that run side by side (batches)
// shift their lists, or the longest groups of all of them would meet on the first SMs.
// Without one (a call that must not touch the shared
// scratch): one group per block, rows of L blocks taken in alternating direction so
// that a column of blocks (about one SM's) gets long and short groups.
struct GroupSource {
    int probe, home;
    bool waited;
    int64_t g_static;
    __device__ GroupSource(const TrajArgs& a, int64_t n_groups) : probe(0), home(0), waited(false), g_static(-1) {
        const int L = a.redo_lists;
        if (a.redo_ctr) {
            home = (int)((sm_id() + (unsigned)a.redo_shift) % (unsigned)L);
        } else {
            const int64_t b = blockIdx.x, row = b / L, pos = b - row * L;
            const int64_t len = n_groups - row * L < L ? n_groups - row * L : L;
            if (pos < len) g_static = row * L + ((row & 1) ? len - 1 - pos : pos);
        }
    }
    // the next group, -1 when none is left; called by every thread of the block
    __device__ int64_t next(const TrajArgs& a, long long& s_g) {
        if (!a.redo_ctr) {
            const int64_t g = g_static;
            g_static = -1;
            return g;
        }
        const int L = a.redo_lists;
        const int* const len = a.redo_ctr + kRedoLists;
        const int* const start = a.redo_ctr + 2 * kRedoLists;
        const int* const grp = a.redo_ctr + 3 * kRedoLists;
        for (; probe < L; ++probe) {
            if (probe == 1 && !waited) {
                waited = true;
                __nanosleep(20000);
            }
            const int l = (home + probe) % L;
            if (threadIdx.x == 0) {
                const int k = atomicAdd(&a.redo_ctr[l], 1);
                s_g = k < len[l] ? (long long)grp[start[l] + k] : -1;
            }
            __syncthreads();
            const long long g = s_g;
            __syncthreads();   // every thread has read s_g before thread 0 writes the next
            if (g >= 0) return g;
        }
        return -1;
    }
};

}  // namespace
}  // namespace sfhk
