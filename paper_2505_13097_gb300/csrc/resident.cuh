// Resident launches: cooperative grids whose blocks stay on the GPU for many
// steps and meet at barriers in global memory (the D2Q9 / D2Q5 steps in
// step_resident.cu, the 2D ILFBM steps in ilfbm.cu).  The barrier, the sums of
// a step and the block that adds them up.
#pragma once

#include "step_common.cuh"

namespace lbm {

// A warp's, and a block's, sums of one step.
struct alignas(16) ResidentSlot {
    Fx e, f;                    // energy terms, boundary flux
    unsigned liquid, shifted;   // saturated liquid nodes; energy terms added less the shift
    unsigned dir[4];            // Dirichlet nodes per wall
    unsigned newton, iters;     // nodes solved, their iterations
    int maxit;
    unsigned lost;              // kLostEnergy, kLostFlux (FP64 forms)
    unsigned pad[2];
};

struct ResidentCommon {
    int nsteps;
    DevStats* stats;
    ResidentSlot* slots;        // kResidentRing sets of one per computing block
    ResidentBar* bar;
    long long wait_ns;          // bound of a wait
    int withhold;               // test hook: block 0 does not arrive at this barrier of the launch (-1: off)
};

// ---------------------------------------------------------------- grid barrier
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// One thread: an arrival for its block (the block has synchronized).
__device__ __forceinline__ void bar_arrive(unsigned* count)
{
    fence_gpu();
    atomicAdd(count, 1u);
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// The bound of a wait: limit_ns without an arrival at any barrier of the launch.
// Counted from the wait's start it would end correct runs: a warp of the
// statistics block waits for as many steps as the block has warps, each of up to
// newton_max_iter barriers in the 2D ILFBM launch.
struct WaitClock {
    unsigned long long t0 = 0, seen = 0;
};

// Now and then during a wait for *word: whether it has run out (arrivals are looked
// at once per limit, so that it runs out after one to two limits).
__device__ __forceinline__ bool wait_over(ResidentBar* b, unsigned long long word, WaitClock& c, long long limit_ns)
{
    const unsigned long long now = global_ns();
    if (c.t0 != 0 && (long long)(now - c.t0) <= limit_ns) return false;
    // counters that only grow during a launch
    const unsigned long long seen = word + ld_relaxed(&b->count) + ld_relaxed(&b->inner[0]) + ld_relaxed(&b->inner[1]);
    const bool over = c.t0 != 0 && seen == c.seen;
    c.t0 = now;
    c.seen = seen;
    return over;
}

// One thread: waits until *count has reached `target`; false when the wait ran out
// here or in another block.  The polls are relaxed (an acquiring load drops the
// SM's L1 lines each time); one fence follows.
__device__ __forceinline__ bool bar_wait(ResidentBar* b, const unsigned* count, unsigned target, long long limit_ns)
{
    WaitClock clock;
    for (unsigned i = 0;; ++i) {
        const unsigned v = ld_relaxed(count);
        if ((int)(v - target) >= 0) break;
        if ((i & 63u) == 63u) {
            if (ld_relaxed(&b->abort)) return false;
            if (wait_over(b, v, clock, limit_ns)) {
                atomicExch(&b->abort, 1u);
                return false;
            }
        }
    }
    fence_gpu();
    return true;
}

// Every block at its end: the last one resets the barrier for the next launch.
// Returns whether this is that block and a wait of the launch ran out.
__device__ __forceinline__ bool bar_leave(ResidentBar* bar)
{
    __shared__ bool last, failed;
    __syncthreads();
    if (threadIdx.x == 0) {
        fence_gpu();
        last = atomicAdd(&bar->done, 1u) == gridDim.x - 1;
        failed = last && ld_acquire(&bar->abort) != 0u;
    }
    __syncthreads();
    if (last) {
        unsigned* b = reinterpret_cast<unsigned*>(bar);
        for (int k = threadIdx.x; k < (int)(sizeof(ResidentBar) / 4); k += blockDim.x) b[k] = 0u;
    }
    return failed;
}

// ---------------------------------------------------------------- a block's sums
// One warp: adds up the block's warps' sums of step s, clears them for step
// s + 2, and hands the total to the statistics block: the block's next arrival
// at the barrier releases it.
static __device__ __noinline__ void resident_emit(const ResidentCommon& a, int s, int nb, int lane, int nwb, ResidentSlot* w)
{
    ResidentSlot t = {};
    if (lane < nwb) {
        t = w[lane];
        w[lane] = ResidentSlot{};
    }
    t.e = fx_tree(t.e);
    t.f = fx_tree(t.f);
    t.liquid = __reduce_add_sync(kFull, t.liquid);
    t.shifted = __reduce_add_sync(kFull, t.shifted);
#pragma unroll
    for (int k = 0; k < 4; ++k) t.dir[k] = __reduce_add_sync(kFull, t.dir[k]);
    t.newton = __reduce_add_sync(kFull, t.newton);
    t.iters = __reduce_add_sync(kFull, t.iters);
    t.maxit = __reduce_max_sync(kFull, t.maxit);
    t.lost = __reduce_or_sync(kFull, t.lost);
    // The sets of the next steps have been read (a ring ago: no wait in practice); looked
    // at for half a ring at once, one lane per set.
    constexpr int kHalf = kResidentRing / 2;
    if (s >= kResidentRing && s % kHalf == 0 && lane < kHalf)
        bar_wait(a.bar, &a.bar->read[(s + lane) % kResidentRing], (unsigned)(s / kResidentRing), a.wait_ns);
    __syncwarp();
    if (lane == 0) a.slots[(size_t)(s % kResidentRing) * nb + blockIdx.x] = t;
}

// ---------------------------------------------------------------- statistics block
// Adds up the computing blocks' sums of every step while later steps run: warp
// w takes the steps w, w + W, ... (W warps), each once the arrivals of the step
// after it are in (those of the last step: the blocks' arrivals at their end).
// A set of slots is written again kResidentRing steps later, after `read` says
// that it has been read.
static __device__ __noinline__ void resident_stats(const ResidentCommon& a, const Problem& pb, unsigned nb)
{
    __shared__ volatile double ring_e[kResidentRing];
    __shared__ volatile int ring_step[kResidentRing];
    __shared__ double imax_s[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    DevStats* st = a.stats;
    ResidentBar* bar = a.bar;
    const double e0 = st->energy;   // of the state before the first step
    const int have0 = st->have_energy;
    double imax = 0.0;
    if (threadIdx.x < kResidentRing) ring_step[threadIdx.x] = -1;
    __syncthreads();
    bool ok = true;
    for (int s = warp; ok && s < a.nsteps; s += nwb) {
        const int at = s % kResidentRing;
        int good = 0;
        if (lane == 0) good = bar_wait(bar, &bar->count, (unsigned)(s + 2) * nb, a.wait_ns);
        ok = __shfl_sync(kFull, good, 0) != 0;
        if (!ok) break;
        const ResidentSlot* set = a.slots + (size_t)at * nb;
        unsigned long long v[16] = {};   // e 4 limbs, f 4 limbs, dir 4, newton, iters, liquid, shifted
        int mx = 0;
        unsigned lost = 0;
        for (unsigned k = lane; k < nb; k += 32) {
            const uint4* p = reinterpret_cast<const uint4*>(set + k);
            const uint4 x0 = __ldcg(p), x1 = __ldcg(p + 1), x2 = __ldcg(p + 2), x3 = __ldcg(p + 3), x4 = __ldcg(p + 4);
            // Fx is {hi, lo}, 8 bytes each
            v[0] += x0.z; v[1] += x0.w; v[2] += x0.x; v[3] += x0.y;
            v[4] += x1.z; v[5] += x1.w; v[6] += x1.x; v[7] += x1.y;
            v[14] += x2.x; v[15] += x2.y;
            v[8] += x2.z; v[9] += x2.w; v[10] += x3.x; v[11] += x3.y;
            v[12] += x3.z; v[13] += x3.w;
            mx = max(mx, (int)x4.x);
            lost |= x4.y;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
        mx = __reduce_max_sync(kFull, mx);
        lost = __reduce_or_sync(kFull, lost);
        if (lane == 0) {
            fence_gpu();
            atomicAdd(&bar->read[at], 1u);   // the set is read
            AccSum es, fs;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                es.limb[j] = v[j];
                fs.limb[j] = v[4 + j];
            }
            double e = lost & kLostEnergy ? nan_d() : acc_read(&es);
            const double f = lost & kLostFlux ? nan_d() : acc_read(&fs);
            double c = (double)v[14];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v[8 + k]) c += (double)v[8 + k] * pb.wall_phi[k];
            e += c * pb.inv_ste;
            if (v[15]) e += (double)v[15] * (double)state_shift(pb, 0);
            // the previous step's energy, from the warp that has that step
            double ep = e0;
            bool have = have0 != 0;
            if (s > 0) {
                const int prev = (s - 1) % kResidentRing;
                unsigned i = 0;
                while (ring_step[prev] != s - 1) {
                    if ((++i & 255u) == 0u && ld_acquire(&bar->abort)) {
                        good = 0;
                        break;
                    }
                }
                __threadfence_block();
                ep = ring_e[prev];
                have = true;
            }
            ring_e[at] = e;
            __threadfence_block();
            ring_step[at] = s;
            const double imb = have ? e - ep - f : 0.0;
            imax = fmax(imax, fabs(imb));
            if (s + 1 == a.nsteps) {
                st->energy = e;
                st->energy_prev = ep;
                st->imbalance = imb;
                st->flux = f;
                st->have_energy = 1;
                st->newton_nodes = (long long)v[12];
                st->newton_iters = (long long)v[13];
                st->newton_max_iter = mx;
            }
        }
        ok = __shfl_sync(kFull, good, 0) != 0;
    }
    if (lane == 0) imax_s[warp] = imax;
    const int all_ok = __syncthreads_and(ok ? 1 : 0);
    if (threadIdx.x == 0) {
        for (int w = 1; w < nwb; ++w) imax = fmax(imax, imax_s[w]);
        if (imax > st->imbalance_max) st->imbalance_max = imax;
        st->steps += a.nsteps;
        if (!all_ok) atomicExch(&st->error, 4);   // LBM_ERR_TIMEOUT
    }
}

}  // namespace lbm
