// D1Q3 IREBM step (Algorithm 3 on the 1D lattice of Sec. 3.2).
//
// Two kernels share the per-node update:
//  * d1q3_step_kernel: one thread per node, one launch per step (any size);
//  * d1q3_fused_kernel: one thread block keeps the whole lattice in shared
//    memory and runs many steps per launch, synchronizing the block between
//    steps.  A 512-node lattice is far too small to fill the GPU, so the
//    per-step cost is launch latency unless the steps are fused.
// Moments are summed exactly from both storage precisions (three terms).
// EEBM (Algorithm 2) runs in the same kernels (method 1 of the problem).
#include "step_common.cuh"

namespace lbm {

struct NodeOut {
    double theta_new;   // theta' of the node
    double energy;      // theta' + phi(theta')/Ste, a saturated liquid node's less 1/Ste
    double flux;        // boundary flux contribution
    int liquid;         // 1 at a saturated liquid node
    int newton;         // 1 if the Newton iteration ran
    int iters;
    bool fail;
};

// One node: u = Omega(x) at time t, ql/qr = Omega_1(x-1), Omega_2(x+1) (ignored at walls).
// One block's SM issues one FP64 warp instruction in 19 cycles (64 for a lone
// warp), so a saturated node spends five: the moment is summed with integers
// (sum_q), the test for saturation runs on FP32 sums, w_i c takes one
// multiplication by a weight (2/3 is 4 times 1/6, and so is its rounding) and the energy is
// fixed point.
template <typename P>
__device__ __forceinline__ NodeOut d1q3_node(const Problem& pb, int x, const P (&u)[3], P ql, P qr, P (&o)[3])
{
    NodeOut r;
    r.flux = 0.0;
    r.liquid = 0;
    r.newton = 0;
    r.iters = 0;
    r.fail = false;
    auto dbl = [](P v) -> double {
        if constexpr (sizeof(P) == 4) return widen(v);
        else return v;
    };
    const double ud[3] = {dbl(u[0]), dbl(u[1]), dbl(u[2])};
    double q[3] = {ud[0], dbl(ql), dbl(qr)};
    bool dir = false;
    double thd = 0.0;
    int side = 0;
    const bool west = x == 0, east = x == pb.nx - 1;
    if (west || east) {
        // nx >= 2: the west node misses q_1 (e = +1), the east node q_2 (e = -1) (Sec. 4.2)
        side = west ? 0 : 1;
        const int iu = west ? 1 : 2, io = west ? 2 : 1;
        const double out = ud[io];   // Omega leaving through this wall
        if (pb.wall_kind[side] == 1) {
            dir = true;
            thd = pb.wall_theta[side];
            // Eq. (16): the single unknown closes M0(q), with M0(q) from Eq. (14) at theta' = theta_D
            // (EEBM: the wall value's enthalpy, Algorithm 2 keeps H = M0)
            const double m0t = dir_m0_target_d(ud[0] + ud[1] + ud[2], side, pb);
            q[iu] = (double)(P)(m0t - q[0] - q[io]);
        } else {
            // bounce-back q_iu = q_io (Sec. 4.2.2), or link-wise q_iu = Omega_io at the node
            q[iu] = pb.bb_mode == 0 ? q[io] : out;
        }
        r.flux = q[iu] - out;
    }
    const double m0 = sum_q<3>(q);
    const double omc = pb.omc, w1 = d1_w(1);
    if (pb.method == 1) {
        // EEBM (Algorithm 2): H = M0(q), theta = Theta(H), relaxation toward
        // w_i theta (i != 0) and H - (1 - w_0) theta (i = 0); the energy is H
        const double t = eebm_theta(m0, pb.inv_ste), om = pb.omega;
        o[0] = (P)fma(omc, q[0], om * eebm_rest(m0, t, d1_w(0), 0.0));
        const double v = (om * w1) * t;
        o[1] = (P)fma(omc, q[1], v);
        o[2] = (P)fma(omc, q[2], v);
        r.theta_new = t;
        r.energy = m0;
        return r;
    }
    const float tf = (approx_float(ud[0]) + approx_float(ud[1])) + approx_float(ud[2]), mf = approx_float(m0);
    const float thr = (float)kSat * pb.delta_f, marg = 1e-5f * (1.0f + fabsf(tf));
    const bool liq = tf >= thr + marg && mf >= thr + marg;
    const bool sat = liq || (tf <= -thr - marg && mf <= -thr - marg);
    double v;   // w_1 c, c = theta' - (1 - omega) m0
    if (dir) {
        v = w1 * (thd - omc * m0);
        r.theta_new = thd;
        r.energy = thd + pb.wall_phi[side] * pb.inv_ste;
    } else if (sat) {
        v = w1 * fma(-omc, m0, m0);   // (not (omega w_1) m0: a constant's rounding would enter every step)
        r.theta_new = m0;
        r.energy = m0;
        r.liquid = liq ? 1 : 0;
    } else {
        const NewtonNode nr = newton_mixed<false>(m0, sum_q<3>(ud), 0.0, pb);
        r.fail = !nr.ok;
        v = w1 * fma(-omc, m0, nr.tns);
        r.theta_new = nr.tns;
        r.energy = nr.ens;
        r.newton = 1;
        r.iters = nr.iters;
    }
    o[0] = (P)fma(omc, q[0], scale2(v, 2));
    o[1] = (P)fma(omc, q[1], v);
    o[2] = (P)fma(omc, q[2], v);
    return r;
}

template <typename P>
__global__ void __launch_bounds__(128) d1q3_step_kernel(StepArgs a)
{
    const Problem& pb = a.probs[0];
    DevStats* st = &a.stats[pb.stats];
    const P* src = static_cast<const P*>(pb.state[a.parity]);
    P* dst = static_cast<P*>(pb.state[a.parity ^ 1]);
    const long long pl = pb.plane, row = pb.pitch;   // row 0 of a plane starts at +pitch
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    Fx e{0, 0ull}, f{0, 0ull};
    unsigned lost = 0u;
    int nn = 0, mi = 0, nl = 0;
    if (x < pb.nx) {
        P u[3], o[3];
        for (int i = 0; i < 3; ++i) u[i] = src[i * pl + row + x];
        const P ql = x > 0 ? src[1 * pl + row + x - 1] : (P)0;
        const P qr = x < pb.nx - 1 ? src[2 * pl + row + x + 1] : (P)0;
        NodeOut r = d1q3_node<P>(pb, x, u, ql, qr, o);
        for (int i = 0; i < 3; ++i) dst[i * pl + row + x] = o[i];
        if (a.rec) a.rec[x] = r.theta_new;
        if (r.fail) atomicOr(&st->error, 3);
        e = to_fixed(r.energy);
        f = to_fixed(r.flux);
        lost = (fx_mag(r.energy) >= kFxMag ? kLostEnergy : 0u) | (fx_mag(r.flux) >= kFxMag ? kLostFlux : 0u);
        nn = r.newton;
        mi = r.iters;
        nl = r.liquid;
    }
    e = fx_tree(e);
    f = fx_tree(f);
    nn = warp_sum_i(nn);
    nl = warp_sum_i(nl);
    mi = warp_max_i(mi);
    lost = __reduce_or_sync(kFull, lost);
    if ((threadIdx.x & 31) == 0) {
        acc_add_fx(&my_stripe(st)->energy, e);
        acc_add_fx(&my_stripe(st)->flux, f);
        if (nn) atomicAdd(&my_stripe(st)->newton, (unsigned long long)nn);
        if (nl) atomicAdd(&my_stripe(st)->liquid, (unsigned long long)nl);
        if (mi) atomicMax(&st->cur_maxit, mi);
        if (lost) atomicOr(&st->cur_lost, lost);
    }
    finish_launch(a.stats, 1, a.ticket, a.probs);
}

constexpr int kFusedThreads = 512;               // computing threads
constexpr int kFusedWarps = kFusedThreads / 32;

// One block keeps the lattice in shared memory and runs `nsteps` steps.  A
// step ends at a single barrier.  The warps' sums go to a per-step parity half
// of a small array; a warp of its own adds them up and keeps the statistics
// while the others run the next step (a half is written again two steps later,
// after a barrier that warp reaches only when it has read it).  What bounds a
// step is the longest warp's chain: a Newton solve, 43 FP64 instructions of 64
// cycles and the FP32 stage; the saturated warps run beside it.
// 512 nodes with a front: 15.3 us per step with a library tanh and FP64 sums,
// 9.3 with the shorter solve alone.
template <typename P, bool DEV>
__global__ void __launch_bounds__(kFusedThreads + 32)
    d1q3_fused_kernel(StepArgs a, const __grid_constant__ Problem pbv, int nsteps, double* rec)
{
    const Problem& pb = DEV ? a.probs[0] : pbv;
    extern __shared__ unsigned char smem_raw[];
    __shared__ Fx red_e[2][kFusedWarps], red_f[2][kFusedWarps];
    __shared__ int red_n[2][kFusedWarps], red_m[2][kFusedWarps], red_l[2][kFusedWarps], red_i[2][kFusedWarps];
    __shared__ unsigned red_b[2][kFusedWarps];   // kLostEnergy, kLostFlux
    DevStats* st = &a.stats[pb.stats];
    const int n = pb.nx;
    P* buf[2] = {reinterpret_cast<P*>(smem_raw), reinterpret_cast<P*>(smem_raw) + 3 * n};
    const long long pl = pb.plane, row = pb.pitch;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const P* src = static_cast<const P*>(pb.state[a.parity]);
    for (int x = threadIdx.x; x < n; x += blockDim.x)
        for (int i = 0; i < 3; ++i) buf[0][i * n + x] = src[i * pl + row + x];
    __syncthreads();
    if (w == kFusedWarps) {
        // the statistics, carried across the steps of this launch
        double E = st->energy, E_prev = st->energy_prev, imb = st->imbalance, imb_max = st->imbalance_max, flux = st->flux;
        int have = st->have_energy, last_n = (int)st->newton_nodes, last_m = st->newton_max_iter;
        long long last_i = st->newton_iters;
        for (int s = 0; s < nsteps; ++s) {
            __syncthreads();   // the sums of step s are in
            const int h = s & 1;
            const bool mine = l < kFusedWarps;
            const Fx e = fx_tree(mine ? red_e[h][l] : Fx{0, 0ull});
            const Fx f = fx_tree(mine ? red_f[h][l] : Fx{0, 0ull});
            last_n = __reduce_add_sync(kFull, mine ? red_n[h][l] : 0);
            last_i = __reduce_add_sync(kFull, mine ? red_i[h][l] : 0);
            last_m = __reduce_max_sync(kFull, mine ? red_m[h][l] : 0);
            const int nl = __reduce_add_sync(kFull, mine ? red_l[h][l] : 0);
            const unsigned lost = __reduce_or_sync(kFull, mine ? red_b[h][l] : 0u);
            const double es = lost & kLostEnergy ? nan_d() : fx_value(e) + (double)nl * pb.inv_ste;
            const double fs = lost & kLostFlux ? nan_d() : fx_value(f);
            if (have) {
                imb = es - E - fs;
                if (fabs(imb) > imb_max) imb_max = fabs(imb);
            }
            E_prev = E;
            E = es;
            flux = fs;
            have = 1;
        }
        if (l == 0) {
            st->energy = E;
            st->energy_prev = E_prev;
            st->imbalance = imb;
            st->imbalance_max = imb_max;
            st->flux = flux;
            st->have_energy = have;
            st->steps += nsteps;
            st->newton_nodes = last_n;
            st->newton_iters = last_i;
            st->newton_max_iter = last_m;
        }
    } else {
        bool fail = false;
        int cur = 0;
        for (int s = 0; s < nsteps; ++s) {
            const P* in = buf[cur];
            P* out = buf[cur ^ 1];
            Fx e{0, 0ull}, f{0, 0ull};
            unsigned emag = 0u, fmag = 0u;
            int nn = 0, mi = 0, nl = 0, ni = 0;
            bool wall = false;
            for (int x = threadIdx.x; x < n; x += kFusedThreads) {
                P u[3] = {in[x], in[n + x], in[2 * n + x]}, o[3];
                const P ql = x > 0 ? in[n + x - 1] : (P)0;
                const P qr = x < n - 1 ? in[2 * n + x + 1] : (P)0;
                NodeOut r = d1q3_node<P>(pb, x, u, ql, qr, o);
                out[x] = o[0];
                out[n + x] = o[1];
                out[2 * n + x] = o[2];
                if (rec) rec[(long long)s * pb.pitch + x] = r.theta_new;
                fx_add(e, to_fixed(r.energy));
                emag = max(emag, fx_mag(r.energy));
                if (x == 0 || x == n - 1) {
                    fx_add(f, to_fixed(r.flux));
                    fmag = max(fmag, fx_mag(r.flux));
                    wall = true;
                }
                nn += r.newton;
                nl += r.liquid;
                ni += r.iters;
                mi = max(mi, r.iters);
                fail |= r.fail;
            }
            e = fx_tree(e);
            if (__any_sync(kFull, wall)) f = fx_tree(f);
            nn = __reduce_add_sync(kFull, nn);
            nl = __reduce_add_sync(kFull, nl);
            if (nn) {
                ni = __reduce_add_sync(kFull, ni);
                mi = __reduce_max_sync(kFull, mi);
            }
            const unsigned lost =
                __reduce_or_sync(kFull, (emag >= kFxMag ? kLostEnergy : 0u) | (fmag >= kFxMag ? kLostFlux : 0u));
            const int h = s & 1;
            if (l == 0) {
                red_b[h][w] = lost;
                red_e[h][w] = e;
                red_f[h][w] = f;
                red_n[h][w] = nn;
                red_l[h][w] = nl;
                red_i[h][w] = ni;
                red_m[h][w] = mi;
            }
            __syncthreads();   // the step's writes of `out` and of the sums are complete
            cur ^= 1;
        }
        if (fail) atomicOr(&st->error, 3);
    }
    __syncthreads();
    P* dst = static_cast<P*>(pb.state[a.parity ^ (nsteps & 1)]);
    for (int x = threadIdx.x; x < n; x += blockDim.x)
        for (int i = 0; i < 3; ++i) dst[i * pl + row + x] = buf[nsteps & 1][i * n + x];
}

static size_t fused_smem(int precision, int nx) { return (size_t)2 * 3 * nx * (precision == 1 ? 4 : 8); }

bool d1q3_fused_fits(int precision, int nx) { return fused_smem(precision, nx) <= 200 * 1024; }

cudaError_t launch_d1q3_step(int precision, const StepArgs& a, const Problem& hp, cudaStream_t s)
{
    const int grid = (hp.nx + 127) / 128;
    if (precision == 1) d1q3_step_kernel<float><<<grid, 128, 0, s>>>(a);
    else d1q3_step_kernel<double><<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_d1q3_fused(int precision, const StepArgs& a, const Problem& hp, int nsteps, int start_parity,
                              double* rec, bool from_device, cudaStream_t s)
{
    StepArgs b = a;
    b.parity = start_parity;
    const size_t sm = fused_smem(precision, hp.nx);
    const auto kernel = precision == 1 ? (from_device ? d1q3_fused_kernel<float, true> : d1q3_fused_kernel<float, false>)
                                       : (from_device ? d1q3_fused_kernel<double, true> : d1q3_fused_kernel<double, false>);
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kernel<<<1, kFusedThreads + 32, sm, s>>>(b, hp, nsteps, rec);
    return cudaGetLastError();
}

}  // namespace lbm
