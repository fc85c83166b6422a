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
// The loop's test is a maximum over the lattice, so the iterations of a step
// are separated by lattice-wide barriers.  D1Q3: a lattice of the paper's sizes
// (N <= 1601) fits in one thread block's shared memory (72 bytes per node): one
// block runs all steps of a call, its barriers are __syncthreads, and HBM is
// touched only at the start and the end of the call.  The block's SM issues one
// FP64 warp instruction in 19 cycles, which bounds what all nodes do, and a lone
// warp one in 64, which bounds an inner iteration.  So
//  * an iterate is a function of l^(k-1) at the node and its neighbours and
//    repeats bit for bit where they did not change: an iteration evaluates only
//    segments of 32 nodes next to a change (the mushy zone is a node or two wide;
//    the two buffers of l agree everywhere else);
//  * the source-free sum S0 of the streamed populations is formed once per step,
//    an iteration adds the three source terms;
//  * the first iterate has no source; the last streaming adds it only near a
//    change, and collides for the next step;
//  * sums are fixed point, comparisons work on the bits, and a warp of its own
//    adds up the statistics while the next step runs.
// 801 nodes: 86 us per step with every node in every iteration.
#include <algorithm>

#include "resident.cuh"

namespace lbm {

constexpr int kIlfThreads = 512;                // computing threads
constexpr int kIlfWarps = kIlfThreads / 32;
constexpr int kIlfSegs = 96;                    // segments of 32 nodes, at most (2,844 nodes)

__device__ __forceinline__ double ilf_lever(double H, double ste, double inv_ste)
{
    // sign and order from the bits
    const long long b = __double_as_longlong(H);
    if ((b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll) return H;   // NaN
    return b < 0 ? 0.0 : (b > __double_as_longlong(inv_ste) ? 1.0 : ste * H);
}

// |d| > tol, tol > 0 (NaN: no)
__device__ __forceinline__ bool ilf_above(double d, double tol)
{
    const long long b = __double_as_longlong(d) & 0x7fffffffffffffffll;
    return b > __double_as_longlong(tol) && b <= 0x7ff0000000000000ll;
}

template <bool DEV>
__global__ void __launch_bounds__(kIlfThreads + 32) ilfbm_d1q3_kernel(StepArgs a, const __grid_constant__ Problem pbv, int nsteps)
{
    const Problem& pb = DEV ? a.probs[0] : pbv;   // (device: for launches that a caller's graph keeps)
    extern __shared__ double sm[];
    __shared__ Fx red_e[2][kIlfWarps], red_f[2][kIlfWarps];   // per-step sums, step parity
    __shared__ unsigned red_b[2][kIlfWarps];                  // kLostEnergy, kLostFlux
    __shared__ unsigned char chg[3][kIlfSegs + 2];            // segment changed in iteration k: chg[k % 3][segment + 1]
    __shared__ unsigned char ever[kIlfSegs + 2];              // ... in some iteration of the step
    DevStats* st = &a.stats[pb.stats];
    const int n = pb.nx, nseg = (n + 31) / 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool stats_warp = w == kIlfWarps;   // no nodes; takes part in the barriers
    const int seg0 = stats_warp ? nseg : w;
    double* o = sm;              // Omega_i of the step without the source
    double* fn = sm + 3 * n;     // next step's; during the iterations: l - l^(k) (two buffers), S0
    double* el = sm + 6 * n;     // l at time t
    double* lb[2] = {el + n, el + 2 * n};   // l^(k), alternating
    const long long pl = pb.plane, row = pb.pitch;
    const double om = pb.omega, ste = pb.ste, inv_ste = pb.inv_ste, tol = pb.tol;
    const double w1 = d1_w(1);
    const double c0 = d1_w(0) * inv_ste, c1 = w1 * inv_ste;   // (w_i/Ste)
    const bool dirW = pb.wall_kind[0] == 1, dirE = pb.wall_kind[1] == 1;
    const double thW = pb.wall_theta[0], thE = pb.wall_theta[1];
    const bool mirror = pb.bb_mode == 0;
    // Omega_i = f_i - (f_i - w_i theta) omega, theta = sum f_i: in this form (1 - omega and
    // omega w_i do not appear as rounded factors) theta does not drift over many steps
    auto collide = [&](const double (&f)[3], double th, double (&g)[3]) {
        g[0] = fma(-om, fma(-d1_w(0), th, f[0]), f[0]);
        g[1] = fma(-om, fma(-w1, th, f[1]), f[1]);
        g[2] = fma(-om, fma(-w1, th, f[2]), f[2]);
    };
    // the state at time t: f_i, collided, and l
    const double* src = static_cast<const double*>(pb.state[a.parity]);
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        const double f[3] = {src[row + x], src[pl + row + x], src[2 * pl + row + x]};
        double g[3];
        collide(f, sum_q<3>(f), g);
        for (int i = 0; i < 3; ++i) o[i * n + x] = g[i];
        lb[0][x] = src[3 * pl + row + x];
    }
    if (threadIdx.x < kIlfSegs + 2) chg[0][threadIdx.x] = chg[1][threadIdx.x] = chg[2][threadIdx.x] = ever[threadIdx.x] = 0;
    bool failed = false;
    // the statistics warp: carried across the steps of this launch
    double E = st->energy, E_prev = st->energy_prev, imb = st->imbalance, imb_max = st->imbalance_max, flux = st->flux;
    int have = st->have_energy, last_it = st->newton_max_iter;
    __syncthreads();
    int base = 0;
    for (int s = 0; s < nsteps; ++s) {
        double* S0 = fn + 2 * n;
        // first iterate: l^(0) = l, no source
        bool more = false;
        for (int sg = seg0; sg < nseg; sg += kIlfWarps) {
            const int y = sg * 32 + lane;
            bool changed = false;
            if (y < n) {
                const double l0 = lb[base][y];
                el[y] = l0;
                double lk;
                if (y == 0 && dirW) {
                    lk = thW > 0.0 ? 1.0 : 0.0;
                } else if (y == n - 1 && dirE) {
                    lk = thE > 0.0 ? 1.0 : 0.0;
                } else {
                    double q[3] = {o[y], y > 0 ? o[n + y - 1] : 0.0, y < n - 1 ? o[2 * n + y + 1] : 0.0};
                    if (y == 0) q[1] = mirror ? q[2] : o[2 * n];
                    if (y == n - 1) q[2] = mirror ? q[1] : o[n + n - 1];
                    const double sum = sum_q<3>(q);
                    S0[y] = sum;
                    lk = ilf_lever(fma(l0, inv_ste, sum), ste, inv_ste);
                }
                const double d = l0 - lk;
                more |= ilf_above(d, tol);
                changed = lk != l0;
                lb[base ^ 1][y] = lk;
                fn[base * n + y] = 0.0;
                fn[(base ^ 1) * n + y] = d;
            }
            const bool c = __any_sync(kFull, changed);
            if (lane == 0) {
                chg[1][sg + 1] = ever[sg + 1] = c;
                chg[2][sg + 1] = 0;
            }
        }
        bool any = __syncthreads_or(more ? 1 : 0) != 0;
        int k = 1;
        while (any && k < pb.maxit) {   // k and any are the same in every thread
            ++k;
            const int pv = (base + k - 1) & 1;
            const double* lp = lb[pv];
            const double* dp = fn + pv * n;
            double* ln = lb[pv ^ 1];
            double* dn = fn + (pv ^ 1) * n;
            const unsigned char* prev = chg[(k - 1) % 3];
            unsigned char* cur = chg[k % 3];
            unsigned char* next = chg[(k + 1) % 3];
            more = false;
            for (int sg = seg0; sg < nseg; sg += kIlfWarps) {
                bool changed = false;
                if (prev[sg] | prev[sg + 1] | prev[sg + 2]) {
                    const int y = sg * 32 + lane;
                    if (y < n) {
                        const double l0 = lp[y];
                        double lk = l0;   // a Dirichlet node keeps its wall's phase
                        if (!((y == 0 && dirW) || (y == n - 1 && dirE))) {
                            // S0 and the source terms c_i (l - l^(k-1)); a wall's unknown one is
                            // the opposite one's, mirrored or of the node itself
                            const double d0 = dp[y];
                            double d1 = y > 0 ? dp[y - 1] : 0.0, d2 = y < n - 1 ? dp[y + 1] : 0.0;
                            if (y == 0) d1 = mirror ? d2 : d0;
                            if (y == n - 1) d2 = mirror ? d1 : d0;
                            double H = fma(c0, d0, S0[y]);
                            H = fma(c1, d1, H);
                            H = fma(c1, d2, H);
                            lk = ilf_lever(fma(l0, inv_ste, H), ste, inv_ste);
                        }
                        more |= ilf_above(lk - l0, tol);
                        changed = lk != l0;
                        ln[y] = lk;
                        dn[y] = el[y] - lk;
                    }
                    changed = __any_sync(kFull, changed);
                }
                if (lane == 0) {
                    next[sg + 1] = 0;
                    if (changed) cur[sg + 1] = ever[sg + 1] = 1;
                }
            }
            any = __syncthreads_or(more ? 1 : 0) != 0;
        }
        failed |= any;
        // f~ with the source of l^(k-1), l~ = l^(k); the boundary flux is filled minus leaving
        // at the two walls; collided for the launch's next step
        const double* lp = lb[(base + k - 1) & 1];
        const double* ln = lb[(base + k) & 1];
        const bool last = s + 1 == nsteps;
        Fx e{0, 0ull}, fl{0, 0ull};
        unsigned emag = 0u, fmag = 0u;
        bool wall = false;
        for (int sg = seg0; sg < nseg; sg += kIlfWarps) {
            const int y = sg * 32 + lane;
            if (y >= n) continue;
            const bool near = (ever[sg] | ever[sg + 1] | ever[sg + 2]) != 0;
            double q0 = o[y], q1 = y > 0 ? o[n + y - 1] : 0.0, q2 = y < n - 1 ? o[2 * n + y + 1] : 0.0;
            double o1 = o[n + y], o2 = o[2 * n + y];   // leaving at a wall
            if (near) {
                const double d0 = el[y] - lp[y];
                q0 = fma(c0, d0, q0);
                if (y > 0) q1 = fma(c1, el[y - 1] - lp[y - 1], q1);
                if (y < n - 1) q2 = fma(c1, el[y + 1] - lp[y + 1], q2);
                o1 = fma(c1, d0, o1);
                o2 = fma(c1, d0, o2);
            }
            if (y == 0) {   // west wall: f_1 (e = +1) is unknown
                q1 = dirW ? thW - q0 - q2 : (mirror ? q2 : o2);
                fx_add(fl, to_fixed(q1 - o2));
                fmag = max(fmag, fx_mag(q1 - o2));
                wall = true;
            }
            if (y == n - 1) {   // east wall: f_2 (e = -1) is unknown
                q2 = dirE ? thE - q0 - q1 : (mirror ? q1 : o1);
                fx_add(fl, to_fixed(q2 - o1));
                fmag = max(fmag, fx_mag(q2 - o1));
                wall = true;
            }
            const double q[3] = {q0, q1, q2};
            const double th = sum_q<3>(q);
            const double H = fma(ln[y], inv_ste, th);
            fx_add(e, to_fixed(H));
            emag = max(emag, fx_mag(H));
            double g[3] = {q0, q1, q2};
            if (!last) collide(q, th, g);
            for (int i = 0; i < 3; ++i) fn[i * n + y] = g[i];
        }
        e = fx_tree(e);
        if (__any_sync(kFull, wall)) fl = fx_tree(fl);
        const unsigned lost = __reduce_or_sync(kFull, (emag >= kFxMag ? kLostEnergy : 0u) | (fmag >= kFxMag ? kLostFlux : 0u));
        const int h = s & 1;
        if (lane == 0 && !stats_warp) {
            red_b[h][w] = lost;
            red_e[h][w] = e;
            red_f[h][w] = fl;
        }
        __syncthreads();   // the next step's populations and the sums are complete
        double* t = o;
        o = fn;
        fn = t;
        base = (base + k) & 1;
        if (stats_warp) {
            const bool mine = lane < kIlfWarps;
            const unsigned b = __reduce_or_sync(kFull, mine ? red_b[h][lane] : 0u);
            const double ev = fx_value(fx_tree(mine ? red_e[h][lane] : Fx{0, 0ull}));
            const double fv = fx_value(fx_tree(mine ? red_f[h][lane] : Fx{0, 0ull}));
            const double es = b & kLostEnergy ? nan_d() : ev, fs = b & kLostFlux ? nan_d() : fv;
            if (have) {
                imb = es - E - fs;
                if (fabs(imb) > imb_max) imb_max = fabs(imb);
            }
            E_prev = E;
            E = es;
            flux = fs;
            have = 1;
            last_it = k;
        }
    }
    if (stats_warp && lane == 0) {
        st->energy = E;
        st->energy_prev = E_prev;
        st->imbalance = imb;
        st->imbalance_max = imb_max;
        st->flux = flux;
        st->have_energy = have;
        st->steps += nsteps;
        st->newton_nodes = 0;
        st->newton_max_iter = last_it;   // inner iterations of the last step
        if (failed) atomicOr(&st->error, 3);   // LBM_ERR_NEWTON: inner loop at its limit
    }
    double* dst = static_cast<double*>(pb.state[a.parity ^ (nsteps & 1)]);
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        for (int i = 0; i < 3; ++i) dst[i * pl + row + x] = o[i * n + x];
        dst[3 * pl + row + x] = lb[base][x];
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
    if ((int)turn != a.withhold || blockIdx.x != 0) atomicAdd(c, 1ull | (more ? 1ull << 48 : 0ull));
    unsigned long long v;
    WaitClock clock;
    for (unsigned i = 0;; ++i) {
        v = ld_relaxed(c);
        if ((v & 0xffffffffffffull) >= target) break;
        if ((i & 63u) == 63u) {
            if (ld_acquire(&a.bar->abort)) return false;
            if (wait_over(a.bar, v, clock, a.wait_ns)) {
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
constexpr int kIlf2Steps = 256;   // steps of one launch, at most (and 2^24 node updates: some 50 ms)

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
        unsigned emag = 0u, fmag = 0u;
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
                const double f = ilf2_streamed<Q>(pb, st, lp, x, y, q, true);
                fx_add(fx, to_fixed(f));
                fmag = max(fmag, fx_mag(f));
            }
            double th = 0.0;
#pragma unroll
            for (int i = 0; i < Q; ++i) th += q[i];
#pragma unroll
            for (int i = 0; i < Q; ++i)
                dst[i * pb.plane + at] = last ? q[i] : q[i] - (q[i] - lat_w(Q, i) * th) * om;
            const double l = ln[nd];
            dst[Q * pb.plane + at] = l;
            const double H = th + l * inv_ste;
            fx_add(e, to_fixed(H));
            emag = max(emag, fx_mag(H));
        }
        e = fx_tree(e);
        fx = fx_tree(fx);
        const unsigned lost = __reduce_or_sync(kFull, (emag >= kFxMag ? kLostEnergy : 0u) | (fmag >= kFxMag ? kLostFlux : 0u));
        if (lane == 0) {
            ResidentSlot* w = &wsum[s & 1][warp];
            w->e = e;
            w->f = fx;
            w->maxit = k;   // inner iterations of the step
            w->lost = lost;
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
        return 2;
    const long long want = ((long long)ilf2_units(nx, ny) + kIlf2Threads / 32 - 1) / (kIlf2Threads / 32) + 1;
    return (int)std::max(2ll, std::min(want, (long long)sms * per));
}

cudaError_t launch_ilfbm_2d(const Problem& hp, int* parity, int* nsteps, int* blocks, void* scratch, DevStats* stats,
                            void* slots, ResidentBar* bar, const ResidentLimits& lim, cudaStream_t s)
{
    Ilf2Args a;
    const size_t n = (size_t)hp.nx * hp.ny, units = ilf2_units(hp.nx, hp.ny);
    double* d = static_cast<double*>(scratch);
    a.pb = hp;
    a.stats = stats;
    a.slots = static_cast<ResidentSlot*>(slots);
    a.bar = bar;
    a.wait_ns = lim.wait_ns;
    a.withhold = lim.withhold;
    a.s0 = d;
    a.lb[0] = d + n;
    a.lb[1] = d + 2 * n;
    a.dl[0] = d + 3 * n;
    a.dl[1] = d + 4 * n;
    for (int k = 0; k < 3; ++k) a.chg[k] = reinterpret_cast<unsigned char*>(d + 5 * n) + k * units;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kIlf2Threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int most = (int)std::max<size_t>(2, std::min<size_t>(kIlf2Steps, ((size_t)1 << 24) / n));
    if (lim.max_steps > 0) most = std::min(most, lim.max_steps);
    while (*nsteps > 0) {
        a.parity = *parity;
        a.nsteps = std::min(*nsteps, most);
        cfg.gridDim = dim3((unsigned)*blocks);
        cudaError_t e = cudaErrorCooperativeLaunchTooLarge;
        if (!lim.refuses(*blocks))
            e = hp.q == 9 ? cudaLaunchKernelEx(&cfg, ilf2_kernel<9>, a) : cudaLaunchKernelEx(&cfg, ilf2_kernel<5>, a);
        if (e == cudaErrorCooperativeLaunchTooLarge && *blocks > 2) {
            // the grid does not fit here (SMs held back from this process): the kernel's blocks
            // take the lattice in strides, so any number of them will do
            (void)cudaGetLastError();
            *blocks = std::max(2, *blocks / 2);
            continue;
        }
        if (e != cudaSuccess) return e;
        *parity ^= a.nsteps & 1;
        *nsteps -= a.nsteps;
    }
    return cudaSuccess;
}

static size_t ilfbm_smem(int nx) { return (size_t)9 * nx * sizeof(double); }

bool ilfbm_d1q3_fits(int nx) { return ilfbm_smem(nx) <= 200 * 1024; }

cudaError_t launch_ilfbm_d1q3(const StepArgs& a, const Problem& hp, int nsteps, bool from_device, cudaStream_t s)
{
    const size_t sm = ilfbm_smem(hp.nx);
    const auto kernel = from_device ? ilfbm_d1q3_kernel<true> : ilfbm_d1q3_kernel<false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kernel<<<1, kIlfThreads + 32, sm, s>>>(a, hp, nsteps);
    return cudaGetLastError();
}

}  // namespace lbm
