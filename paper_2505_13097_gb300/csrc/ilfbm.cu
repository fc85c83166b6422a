// ILFBM step (Algorithm 1, the implicit liquid fraction based method of
// Sec. 3.3), the paper's second comparison scheme, in FP64: D1Q3 in one
// block (below), D2Q9 and D2Q5 in one cooperative launch (at the end).
//
// State: f_i (planes 0..q-1, theta = M0(f)) and the liquid fraction l (plane
// q of the same buffer).  One step:
//   theta = M0(f); l^(0) = l; for k = 1, 2, ...:
//     Omega_i = f_i - (f_i - w_i theta)/tau + (w_i/Ste)(l - l^(k-1))
//     f^(k)_i(y) = Omega_i(y - e_i), closures on the unknown one at a wall
//     H^(k) = M0(f^(k)) + l^(k-1)/Ste,  l^(k) = l(H^(k))  (lever rule)
//   until max_y |l^(k) - l^(k-1)| <= tol (at most maxit iterations; the
//   limit sets LBM_ERR_NEWTON); f~ = f^(k), l~ = l^(k).
// Closures: Dirichlet makes M0(f^(k)) = theta_D through the one unknown,
// bounce-back as for IREBM; a Dirichlet node's liquid fraction is that of its
// wall value, [theta_D > 0].
//
// Every inner iteration streams the whole lattice, and the loop's test is a
// maximum over the lattice, so the iterations of a step are separated by
// lattice-wide barriers.  D1Q3: a lattice of the paper's sizes (N <= 1601) fits
// in one thread block's shared memory (72 bytes per node): one block runs
// all steps of a call, its barriers are __syncthreads, and HBM is touched
// only at the start and the end of the call.  The inner loop is bound by the
// block's FP64 issue rate (FP64 is scarce on this GPU), so it is cut to what
// changes between iterations: the source-free part of the collision is formed
// once per step, an iteration forms only H^(k) and l^(k) (the populations
// f^(k) are streamed once, after the loop), and the loop's test is one flag
// per iteration behind a single barrier (three flags in rotation: the one
// cleared for the next iteration was last read two iterations earlier).
#include "resident.cuh"

namespace lbm {

constexpr int kIlfThreads = 512;
constexpr int kIlfWarps = kIlfThreads / 32;

__device__ __forceinline__ double ilf_lever(double H, double ste, double inv_ste)
{
    return H < 0.0 ? 0.0 : (H > inv_ste ? 1.0 : ste * H);
}

__global__ void __launch_bounds__(kIlfThreads) ilfbm_d1q3_kernel(StepArgs a, int nsteps)
{
    extern __shared__ double sm[];
    __shared__ double red_e[2][kIlfWarps], red_f[2][kIlfWarps];   // per-step partial sums, step parity
    __shared__ int s_more[3];   // "some node changed by more than tol", iteration gk uses gk % 3
    const Problem& pb = a.probs[0];
    DevStats* st = &a.stats[pb.stats];
    const int n = pb.nx;
    double* o = sm;              // f_i at time t, then Omega_i without the source: f_i - (f_i - w_i theta)/tau
    double* fn = sm + 3 * n;     // f~ of the step (the buffers swap roles every step)
    double* el = sm + 6 * n;     // l at time t
    double* lb[2] = {el + n, el + 2 * n};   // l^(k-1) and l^(k), alternating
    const long long pl = pb.plane, row = pb.pitch;
    const double* src = static_cast<const double*>(pb.state[a.parity]);
    // the state at time t: f_i and l
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        for (int i = 0; i < 3; ++i) o[i * n + x] = src[i * pl + row + x];
        el[x] = src[3 * pl + row + x];
    }
    const double om = pb.omega, ste = pb.ste, inv_ste = pb.inv_ste, tol = pb.tol;
    const double w0 = d1_w(0), w1 = d1_w(1), w2 = d1_w(2);
    const double c0 = w0 * inv_ste, c1 = w1 * inv_ste, c2 = w2 * inv_ste;
    const bool dirW = pb.wall_kind[0] == 1, dirE = pb.wall_kind[1] == 1;
    const double thW = pb.wall_theta[0], thE = pb.wall_theta[1];
    const bool mirror = pb.bb_mode == 0;
    bool failed = false;
    unsigned gk = 0;   // inner iterations so far in this launch: selects the flag
    // thread 0: the statistics carried across the steps of this launch
    double E = 0.0, E_prev = 0.0, imb = 0.0, imb_max = 0.0, flux = 0.0;
    int have = 0, last_it = 0;
    if (threadIdx.x == 0) {
        E = st->energy;
        E_prev = st->energy_prev;
        imb = st->imbalance;
        imb_max = st->imbalance_max;
        flux = st->flux;
        have = st->have_energy;
        last_it = st->newton_max_iter;
    }
    if (threadIdx.x < 3) s_more[threadIdx.x] = 0;
    __syncthreads();
    for (int s = 0; s < nsteps; ++s) {
        // moments and the source-free part of the collision (the same in every
        // inner iteration); l^(0) = l
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            const double f0 = o[x], f1 = o[n + x], f2 = o[2 * n + x];
            const double th = f0 + f1 + f2;
            o[x] = f0 - (f0 - w0 * th) * om;
            o[n + x] = f1 - (f1 - w1 * th) * om;
            o[2 * n + x] = f2 - (f2 - w2 * th) * om;
            lb[0][x] = el[x];
        }
        __syncthreads();
        // streamed f^(k)(y) from Omega_i(x) = o_i(x) + (w_i/Ste)(l(x) - l^(k-1)(x)),
        // the closures on the unknown one at a wall; returns the three values
        auto stream = [&](int y, const double* lp, double& q0, double& q1, double& q2) {
            q0 = o[y] + c0 * (el[y] - lp[y]);
            q1 = y > 0 ? o[n + y - 1] + c1 * (el[y - 1] - lp[y - 1]) : 0.0;
            q2 = y < n - 1 ? o[2 * n + y + 1] + c2 * (el[y + 1] - lp[y + 1]) : 0.0;
            if (y == 0)   // west wall: f_1 (e = +1) is unknown
                q1 = dirW ? thW - q0 - q2 : (mirror ? q2 : o[2 * n] + c2 * (el[0] - lp[0]));
            if (y == n - 1)   // east wall: f_2 (e = -1) is unknown
                q2 = dirE ? thE - q0 - q1 : (mirror ? q1 : o[n + n - 1] + c1 * (el[n - 1] - lp[n - 1]));
        };
        int it = 0, cur = 0;
        bool conv = false;
        while (!conv && it < pb.maxit) {   // it, gk, cur and conv are the same in every thread
            const double* lp = lb[cur];
            double* ln = lb[cur ^ 1];
            const int slot = gk % 3;
            ++it;
            ++gk;
            // H^(k) = M0(f^(k)) + l^(k-1)/Ste and the lever rule; Dirichlet nodes keep
            // the phase of their wall value
            bool more = false;
            for (int y = threadIdx.x; y < n; y += blockDim.x) {
                double lk;
                if (y == 0 && dirW) {
                    lk = thW > 0.0 ? 1.0 : 0.0;
                } else if (y == n - 1 && dirE) {
                    lk = thE > 0.0 ? 1.0 : 0.0;
                } else {
                    double q0, q1, q2;
                    stream(y, lp, q0, q1, q2);
                    lk = ilf_lever(q0 + q1 + q2 + lp[y] * inv_ste, ste, inv_ste);
                }
                more |= fabs(lk - lp[y]) > tol;
                ln[y] = lk;
            }
            // flag of this iteration; thread 0 clears the next iteration's flag, last read
            // two iterations ago (every thread read it before the previous barrier) and
            // next set after this iteration's barrier
            if (more) s_more[slot] = 1;
            if (threadIdx.x == 0) s_more[(slot + 1) % 3] = 0;
            __syncthreads();
            conv = s_more[slot] == 0;
            cur ^= 1;
        }
        failed |= !conv;
        // f~ = f^(k) (streamed with the source of l^(k-1)) into the other buffer,
        // l~ = l^(k); the boundary flux is filled minus leaving at the two walls
        const double* lp = lb[cur ^ 1];
        const double* ln = lb[cur];
        double e = 0.0, fl = 0.0;
        for (int y = threadIdx.x; y < n; y += blockDim.x) {
            double q0, q1, q2;
            stream(y, lp, q0, q1, q2);
            if (y == 0) fl += q1 - (o[2 * n] + c2 * (el[0] - lp[0]));
            if (y == n - 1) fl += q2 - (o[n + n - 1] + c1 * (el[n - 1] - lp[n - 1]));
            fn[y] = q0;
            fn[n + y] = q1;
            fn[2 * n + y] = q2;
            e += (q0 + q1 + q2) + ln[y] * inv_ste;
        }
        e = warp_sum(e);
        fl = warp_sum(fl);
        const int h = s & 1;
        if ((threadIdx.x & 31) == 0) {
            red_e[h][threadIdx.x >> 5] = e;
            red_f[h][threadIdx.x >> 5] = fl;
        }
        __syncthreads();   // every read of o, el and l^(k-1) of this step is done
        for (int y = threadIdx.x; y < n; y += blockDim.x) el[y] = ln[y];
        double* t = o;
        o = fn;
        fn = t;
        if (threadIdx.x == 0) {
            // the warps' sums in a fixed order; a half of red_* is written again two
            // steps later, after the next step's barriers, which thread 0 reaches
            // only after this
            double es = 0.0, fs = 0.0;
            for (int k = 0; k < kIlfWarps; ++k) {
                es += red_e[h][k];
                fs += red_f[h][k];
            }
            if (have) {
                imb = es - E - fs;
                if (fabs(imb) > imb_max) imb_max = fabs(imb);
            }
            E_prev = E;
            E = es;
            flux = fs;
            have = 1;
            last_it = it;
        }
    }
    if (threadIdx.x == 0) {
        st->energy = E;
        st->energy_prev = E_prev;
        st->imbalance = imb;
        st->imbalance_max = imb_max;
        st->flux = flux;
        st->have_energy = have;
        st->steps += nsteps;
        st->newton_nodes = 0;
        st->newton_max_iter = last_it;   // inner iterations of the last step
    }
    if (failed && threadIdx.x == 0) atomicOr(&st->error, 3);   // LBM_ERR_NEWTON: inner loop at its limit
    double* dst = static_cast<double*>(pb.state[a.parity ^ (nsteps & 1)]);
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        for (int i = 0; i < 3; ++i) dst[i * pl + row + x] = o[i * n + x];
        dst[3 * pl + row + x] = el[x];
    }
}

// ---------------------------------------------------------------- 2D lattices
// ILFBM on D2Q9 and D2Q5 (Q = 9 or 5; the D2Q5 velocities are D2Q9's first
// five), FP64, all steps of a call in one cooperative launch.  A step is
//   first      S0(y) = sum_i Omega0_i(y - e_i), Omega0 the source-free collision, and the
//              first iterate l^(1)(y) = l(S0 + l/Ste) (its source vanishes)
//   iterations l^(k)(y) = l(H^(k)(y)), H^(k) = S0(y) + sum_i (w_i/Ste)
//              (l - l^(k-1))(y - e_i) + l^(k-1)(y)/Ste at interior nodes, the
//              closed streamed populations at wall nodes, until no l moves by
//              more than tol
//   last       f~_i(y) = Omega_i(y - e_i) with the source of l^(K-1) and the
//              closures, l~ = l^(K); collided in place for the next step
// with a grid barrier after each.  What bounds it is the chain of some 80
// barriers per step.  An iterate is a function of l^(k-1) at the node and its
// neighbours, so it repeats bit for bit where they did not change: only units
// (32 columns of one row) next to a change are evaluated, the mushy nodes and
// their surroundings, and the two buffers of l agree everywhere else.  One
// launch per iteration over all nodes took 2,550 us per step on the 401^2
// cavity (400 launches, 77 of them with work).
// Scratch (nx*ny doubles each): S0, l^(k) x 2, l - l^(k) x 2 (the stencil reads
// the differences, so an iteration spends one FMA per velocity), and a byte per
// unit for each of three iterations (changed).
struct Ilf2Args : ResidentCommon {
    Problem pb;              // by value
    int parity;
    double* s0;
    double* lb[2];           // l^(k) in lb[(base + k) & 1]
    double* dl[2];           // l - l^(k), likewise
    unsigned char* chg[3];   // unit changed in iteration k: chg[k % 3]
};

template <int Q>
__device__ __forceinline__ bool ilf2_known(const Problem& pb, int x, int y, int i)
{
    const int sx = x - d2_ex(i), sy = y - d2_ey(i);
    return sx >= 0 && sx < pb.nx && sy >= 0 && sy < pb.ny;
}

__device__ __forceinline__ int ilf2_dirichlet(const Problem& pb, int x, int y)
{
    const int walls = (x == 0 ? 1 : 0) | (x == pb.nx - 1 ? 2 : 0) | (y == 0 ? 4 : 0) | (y == pb.ny - 1 ? 8 : 0);
    for (int k = 0; k < 4; ++k)
        if (((walls >> k) & 1) && pb.wall_kind[k] == 1) return k;
    return -1;
}

// Omega_i at node (x, y) with the source of the iterate lp: Omega0_i + (w_i/Ste)(l - lp)
template <int Q>
__device__ __forceinline__ double ilf2_omega(const Problem& pb, const double* st, const double* lp, int i, int x, int y)
{
    const long long nd = (long long)y * pb.nx + x;
    const double* lq = st + Q * pb.plane;
    return st[i * pb.plane + (long long)(y + 1) * pb.pitch + x] +
           lat_w(Q, i) * pb.inv_ste * (lq[(long long)(y + 1) * pb.pitch + x] - lp[nd]);
}

// the streamed populations of node (x, y) with the source of lp, closed at a wall
// (Dirichlet: the unknowns share theta_D - sum(known) by weight; bounce-back:
// mirror where the opposite is known, else link-wise); returns the flux term
// (filled minus leaving) when `flux` is set
template <int Q>
__device__ __forceinline__ double ilf2_streamed(const Problem& pb, const double* st, const double* lp, int x, int y,
                                                double (&q)[Q], bool flux)
{
    unsigned unk = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (ilf2_known<Q>(pb, x, y, i)) q[i] = ilf2_omega<Q>(pb, st, lp, i, x - d2_ex(i), y - d2_ey(i));
        else { q[i] = 0.0; unk |= 1u << i; }
    }
    if (!unk) return 0.0;
    const int wk = ilf2_dirichlet(pb, x, y);
    double in = 0.0, out = 0.0;
    if (wk >= 0) {
        double rest = pb.wall_theta[wk], wu = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if ((unk >> i) & 1) wu += lat_w(Q, i);
            else rest -= q[i];
        }
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if ((unk >> i) & 1) q[i] = lat_w(Q, i) * rest / wu;
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if ((unk >> i) & 1) {
                const int o = d2_opp(i);
                q[i] = (pb.bb_mode == 0 && !((unk >> o) & 1)) ? q[o] : ilf2_omega<Q>(pb, st, lp, o, x, y);
            }
    }
    if (flux) {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if ((unk >> i) & 1) {
                in += q[i];
                out += ilf2_omega<Q>(pb, st, lp, d2_opp(i), x, y);   // Omega leaving through the wall
            }
    }
    return in - out;
}

// One thread: its block's arrival at the inner barrier number `turn`, `more` if
// the block moved some l by more than tol, and the wait for the others; any:
// whether some block did (seen: what this barrier's high bits held after its
// previous turn).  false: a wait ran out.  Two barriers alternate, so nobody
// arrives at one again before everybody has read it.
__device__ __forceinline__ bool inner_barrier(const Ilf2Args& a, unsigned turn, unsigned nb, bool more, unsigned& seen, bool& any)
{
    unsigned long long* c = &a.bar->inner[turn & 1u];
    const unsigned long long target = (turn / 2ull + 1ull) * nb;
    fence_gpu();
    atomicAdd(c, 1ull | (more ? 1ull << 48 : 0ull));
    unsigned long long v, t0 = 0;
    for (unsigned i = 0;; ++i) {
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(c) : "memory");
        if ((v & 0xffffffffffffull) >= target) break;
        if ((i & 63u) == 63u) {
            if (ld_acquire(&a.bar->abort)) return false;
            if (t0 == 0) t0 = global_ns();
            else if ((long long)(global_ns() - t0) > a.wait_ns) {
                atomicExch(&a.bar->abort, 1u);
                return false;
            }
        }
    }
    fence_gpu();
    any = (unsigned)(v >> 48) != seen;   // (modulo 2^16; a turn adds at most one per block)
    seen = (unsigned)(v >> 48);
    return true;
}

constexpr int kIlf2Threads = 512;
constexpr int kIlf2Steps = 256;   // steps of one launch

template <int Q>
__global__ void __launch_bounds__(kIlf2Threads, 1) ilf2_kernel(const __grid_constant__ Ilf2Args a)
{
    __shared__ ResidentSlot wsum[2][kIlf2Threads / 32];   // by step parity
    __shared__ bool ok_s, any_s;
    const Problem& pb = a.pb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int nwb = kIlf2Threads / 32;
    const int nb = gridDim.x - 1;   // computing blocks; the last block adds up the statistics
    if ((int)blockIdx.x == nb) {
        resident_stats(a, pb, (unsigned)nb);
        bar_leave(a.bar);
        return;
    }
    const int nx = pb.nx, ny = pb.ny;
    const int nseg = (nx + 31) / 32, units = nseg * ny;
    const int W = nb * nwb, w0 = warp * nb + (int)blockIdx.x;   // units w0, w0 + W, ...: neighbours on other SMs
    const double om = pb.omega, inv_ste = pb.inv_ste;
    unsigned turn = 0, seen[2] = {0u, 0u};
    bool ok = true;
    // every thread: the inner barrier; false: a wait ran out
    auto barrier = [&](bool more, bool& any) -> bool {
        const int m = __syncthreads_or(more ? 1 : 0);
        if (threadIdx.x == 0) {
            bool some = false;
            ok_s = inner_barrier(a, turn, (unsigned)nb, m != 0, seen[turn & 1u], some);
            any_s = some;
        }
        ++turn;
        __syncthreads();
        any = any_s;
        return ok_s;
    };
    if (threadIdx.x < 2 * nwb) wsum[threadIdx.x / nwb][threadIdx.x % nwb] = ResidentSlot{};
    // the launch's first step: collide its state in place, l^(0) = l
    {
        double* st = static_cast<double*>(pb.state[a.parity]);
        for (int u = w0; u < units; u += W) {
            const int y = u / nseg, x = (u - y * nseg) * 32 + lane;
            if (x >= nx) continue;
            const long long at = (long long)(y + 1) * pb.pitch + x;
            double f[Q], th = 0.0;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                f[i] = st[i * pb.plane + at];
                th += f[i];
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) st[i * pb.plane + at] = f[i] - (f[i] - lat_w(Q, i) * th) * om;
            a.lb[0][(long long)y * nx + x] = st[Q * pb.plane + at];
        }
        bool any;
        ok = barrier(false, any);
    }
    int base = 0;
    for (int s = 0; ok && s < a.nsteps; ++s) {
        const int p = (a.parity + s) & 1;
        const double* st = static_cast<const double*>(pb.state[p]);
        double* dst = static_cast<double*>(pb.state[p ^ 1]);
        const double* lq = st + Q * pb.plane;
        // first iterate: l - l^(0) = 0
        bool more = false, any = true;
        for (int u = w0; u < units; u += W) {
            const int y = u / nseg, x = (u - y * nseg) * 32 + lane;
            bool changed = false;
            if (x < nx) {
                const long long nd = (long long)y * nx + x;
                const double lp = a.lb[base][nd];
                const int wk = ilf2_dirichlet(pb, x, y);
                double lk;
                if (wk >= 0) {
                    lk = pb.wall_theta[wk] > 0.0 ? 1.0 : 0.0;
                } else {
                    double H;
                    if (x > 0 && x < nx - 1 && y > 0 && y < ny - 1) {
                        H = 0.0;
#pragma unroll
                        for (int i = 0; i < Q; ++i)
                            H += st[i * pb.plane + (long long)(y - d2_ey(i) + 1) * pb.pitch + x - d2_ex(i)];
                        a.s0[nd] = H;
                    } else {
                        double q[Q];
                        (void)ilf2_streamed<Q>(pb, st, a.lb[base], x, y, q, false);
                        H = 0.0;
#pragma unroll
                        for (int i = 0; i < Q; ++i) H += q[i];
                    }
                    H += lp * inv_ste;
                    lk = ilf_lever(H, pb.ste, inv_ste);
                }
                more |= fabs(lk - lp) > pb.tol;
                changed = lk != lp;
                a.lb[base ^ 1][nd] = lk;
                a.dl[base][nd] = 0.0;
                a.dl[base ^ 1][nd] = lq[(long long)(y + 1) * pb.pitch + x] - lk;
            }
            const bool c = __any_sync(kFull, changed);
            if (lane == 0) {
                a.chg[1][u] = c;
                a.chg[2][u] = 0;
            }
        }
        ok = barrier(more, any);
        int k = 1;
        while (ok && any && k < pb.maxit) {
            ++k;
            const double* lp = a.lb[(base + k - 1) & 1];
            const double* dp = a.dl[(base + k - 1) & 1];
            double* ln = a.lb[(base + k) & 1];
            double* dn = a.dl[(base + k) & 1];
            const unsigned char* prev = a.chg[(k - 1) % 3];
            unsigned char* cur = a.chg[k % 3];
            unsigned char* next = a.chg[(k + 1) % 3];
            more = false;
            for (int u0 = w0; u0 < units; u0 += 32 * W) {
                // a lane per unit: is it next to a change of iteration k - 1?
                const long long ul = (long long)u0 + (long long)lane * W;
                bool active = false;
                if (ul < units) {
                    const int u = (int)ul, y = u / nseg, sg = u - y * nseg;
                    unsigned f = 0;
#pragma unroll
                    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                        for (int dx = -1; dx <= 1; ++dx)
                            if (y + dy >= 0 && y + dy < ny && sg + dx >= 0 && sg + dx < nseg) f |= prev[u + dy * nseg + dx];
                    active = f != 0u;
                    next[u] = 0;
                }
                unsigned todo = __ballot_sync(kFull, active);
                while (todo) {
                    const int l = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const int u = u0 + l * W, y = u / nseg, x = (u - y * nseg) * 32 + lane;
                    bool changed = false;
                    if (x < nx) {
                        const long long nd = (long long)y * nx + x;
                        const double l0 = lp[nd];
                        const int wk = ilf2_dirichlet(pb, x, y);
                        if (wk < 0) {
                            double H;
                            if (x > 0 && x < nx - 1 && y > 0 && y < ny - 1) {
                                H = a.s0[nd];
#pragma unroll
                                for (int i = 0; i < Q; ++i)
                                    H += lat_w(Q, i) * inv_ste * dp[nd - (long long)d2_ey(i) * nx - d2_ex(i)];
                            } else {
                                double q[Q];
                                (void)ilf2_streamed<Q>(pb, st, lp, x, y, q, false);
                                H = 0.0;
#pragma unroll
                                for (int i = 0; i < Q; ++i) H += q[i];
                            }
                            H += l0 * inv_ste;
                            const double lk = ilf_lever(H, pb.ste, inv_ste);
                            more |= fabs(lk - l0) > pb.tol;
                            changed = lk != l0;
                            ln[nd] = lk;
                            dn[nd] = lq[(long long)(y + 1) * pb.pitch + x] - lk;
                        } else {   // its wall's phase since the first iterate
                            ln[nd] = l0;
                            dn[nd] = dp[nd];
                        }
                    }
                    if (__any_sync(kFull, changed) && lane == 0) cur[u] = 1;
                }
            }
            ok = barrier(more, any);
        }
        if (!ok) break;
        // f~ with the source of l^(k-1), l~ = l^(k); collided for the launch's next step
        const double* lp = a.lb[(base + k - 1) & 1];
        const double* dp = a.dl[(base + k - 1) & 1];
        const double* ln = a.lb[(base + k) & 1];
        const bool last = s + 1 == a.nsteps;
        Fx e{0, 0ull}, fx{0, 0ull};
        for (int u = w0; u < units; u += W) {
            const int y = u / nseg, x = (u - y * nseg) * 32 + lane;
            if (x >= nx) continue;
            const long long nd = (long long)y * nx + x, at = (long long)(y + 1) * pb.pitch + x;
            double q[Q];
            if (x > 0 && x < nx - 1 && y > 0 && y < ny - 1) {
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    q[i] = st[i * pb.plane + at - (long long)d2_ey(i) * pb.pitch - d2_ex(i)] +
                           lat_w(Q, i) * inv_ste * dp[nd - (long long)d2_ey(i) * nx - d2_ex(i)];
            } else {
                fx_add(fx, to_fixed(ilf2_streamed<Q>(pb, st, lp, x, y, q, true)));
            }
            double th = 0.0;
#pragma unroll
            for (int i = 0; i < Q; ++i) th += q[i];
#pragma unroll
            for (int i = 0; i < Q; ++i)
                dst[i * pb.plane + at] = last ? q[i] : q[i] - (q[i] - lat_w(Q, i) * th) * om;
            const double l = ln[nd];
            dst[Q * pb.plane + at] = l;
            fx_add(e, to_fixed(th + l * inv_ste));
        }
        e = fx_tree(e);
        fx = fx_tree(fx);
        if (lane == 0) {
            ResidentSlot* w = &wsum[s & 1][warp];
            w->e = e;
            w->f = fx;
            w->maxit = k;   // inner iterations of the step
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (any && blockIdx.x == 0) atomicOr(&a.stats->error, 3);   // LBM_ERR_NEWTON: the inner loop reached its limit
            bar_arrive(&a.bar->count);
            ok_s = last || bar_wait(a.bar, &a.bar->count, (unsigned)(s + 1) * nb, a.wait_ns);
        } else if (warp == 1) {
            resident_emit(a, s, nb, lane, nwb, wsum[s & 1]);   // while thread 0 waits
        }
        __syncthreads();
        ok = ok_s;
        base = (base + k) & 1;
    }
    if (threadIdx.x == 0) bar_arrive(&a.bar->count);   // the last step's sums are out
    bar_leave(a.bar);
}

static size_t ilf2_units(int nx, int ny) { return (size_t)((nx + 31) / 32) * ny; }
// nx*ny doubles x 5, then three bytes per unit
size_t ilfbm_2d_scratch(int nx, int ny) { return sizeof(double) * 5 * (size_t)nx * ny + 3 * ilf2_units(nx, ny); }

int ilfbm_2d_blocks(int q, int nx, int ny)
{
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        (q == 9 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, ilf2_kernel<9>, kIlf2Threads, 0)
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, ilf2_kernel<5>, kIlf2Threads, 0)) != cudaSuccess)
        return 0;
    const long long want = ((long long)ilf2_units(nx, ny) + kIlf2Threads / 32 - 1) / (kIlf2Threads / 32) + 1;
    return (int)(want < (long long)sms * per ? want : (long long)sms * per);
}

cudaError_t launch_ilfbm_2d(const Problem& hp, int parity, int nsteps, void* scratch, DevStats* stats, void* slots,
                            ResidentBar* bar, long long wait_ns, cudaStream_t s)
{
    const int blocks = ilfbm_2d_blocks(hp.q, hp.nx, hp.ny);
    if (blocks < 2) return cudaErrorCooperativeLaunchTooLarge;
    Ilf2Args a;
    const size_t n = (size_t)hp.nx * hp.ny, units = ilf2_units(hp.nx, hp.ny);
    double* d = static_cast<double*>(scratch);
    a.pb = hp;
    a.stats = stats;
    a.slots = static_cast<ResidentSlot*>(slots);
    a.bar = bar;
    a.wait_ns = wait_ns;
    a.s0 = d;
    a.lb[0] = d + n;
    a.lb[1] = d + 2 * n;
    a.dl[0] = d + 3 * n;
    a.dl[1] = d + 4 * n;
    for (int k = 0; k < 3; ++k) a.chg[k] = reinterpret_cast<unsigned char*>(d + 5 * n) + k * units;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kIlf2Threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    while (nsteps > 0) {
        a.parity = parity;
        a.nsteps = nsteps < kIlf2Steps ? nsteps : kIlf2Steps;
        const cudaError_t e = hp.q == 9 ? cudaLaunchKernelEx(&cfg, ilf2_kernel<9>, a) : cudaLaunchKernelEx(&cfg, ilf2_kernel<5>, a);
        if (e != cudaSuccess) return e;
        parity ^= a.nsteps & 1;
        nsteps -= a.nsteps;
    }
    return cudaSuccess;
}

static size_t ilfbm_smem(int nx) { return (size_t)9 * nx * sizeof(double); }

bool ilfbm_d1q3_fits(int nx) { return ilfbm_smem(nx) <= 200 * 1024; }

cudaError_t launch_ilfbm_d1q3(const StepArgs& a, const Problem& hp, int nsteps, cudaStream_t s)
{
    const size_t sm = ilfbm_smem(hp.nx);
    cudaError_t e = cudaFuncSetAttribute(ilfbm_d1q3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    ilfbm_d1q3_kernel<<<1, kIlfThreads, sm, s>>>(a, nsteps);
    return cudaGetLastError();
}

}  // namespace lbm
