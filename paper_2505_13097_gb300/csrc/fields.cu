// State initialization and field extraction.
//  * init: f_i = w_i theta0 (equilibrium, so Omega_i = w_i theta0), with nodes on
//    a Dirichlet wall set to the wall value; accumulates E(0).  EEBM: the
//    equilibrium of H(theta0); ILFBM: also l = [theta0 > 0] in plane q.
//  * fields: theta = M0(f) = sum_i Omega_i, phi(theta), H = theta + phi/Ste (Sec. 2);
//    EEBM: theta = Theta(H); ILFBM: phi = l.
#include "lbm_device.cuh"

namespace lbm {

__device__ __forceinline__ bool dirichlet_value(const Problem& pb, int x, int y, double& td)
{
    const int walls = (x == 0 ? 1 : 0) | (x == pb.nx - 1 ? 2 : 0) |
                      (pb.q != 3 ? ((y == 0 ? 4 : 0) | (y == pb.ny - 1 ? 8 : 0)) : 0);
    for (int k = 0; k < 4; ++k)
        if (((walls >> k) & 1) && pb.wall_kind[k] == 1) {
            td = pb.wall_theta[k];
            return true;
        }
    return false;
}

// A block's exact sum in thread 0 (256 threads); mag: the largest fx_mag of the
// thread's terms, lost: some thread's has no fixed-point value.
__device__ __forceinline__ Fx block_sum(Fx v, unsigned mag, bool& lost)
{
    __shared__ Fx part[8];
    v = fx_tree(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    lost = __syncthreads_or(mag >= kFxMag ? 1 : 0) != 0;
    if (threadIdx.x == 0)
        for (int w = 1; w < 8; ++w) fx_add(v, part[w]);
    return v;
}

// The blocks' exact sums meet in the stripes of one accumulator (S: its offset
// in a stripe); the last block to arrive (st->ticket, zero before and after)
// gets the total in its first warp, as a double (NaN if a block lost a term), and
// clears the stripes.  Returns whether this is that block's first warp.
template <AccSum StepStripe::*S>
__device__ __forceinline__ bool last_block_total(DevStats* st, const Fx& v, bool lost, double& total)
{
    __shared__ bool last;
    if (threadIdx.x == 0) {
        acc_add_fx(&(st->cur[blockIdx.x % kStripes].*S), v);
        if (lost) atomicOr(&st->cur_lost, kLostEnergy);
        __threadfence();
        last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return false;
    __threadfence();
    AccSum a;
    unsigned long long* own = (st->cur[threadIdx.x].*S).limb;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        a.limb[j] = __ldcg(own + j);
        own[j] = 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a.limb[j] += __shfl_xor_sync(kFull, a.limb[j], o);
    }
    total = __ldcg(&st->cur_lost) ? nan_d() : acc_read(&a);
    __syncwarp();
    if (threadIdx.x == 0) {
        st->ticket = 0u;
        st->cur_lost = 0u;
    }
    return true;
}

// The shift s of an FP32 state (its populations are stored less w_i s),
// written to the tail of both buffers: half the mean over the nodes of the
// initial M0 (theta0; EEBM: H(theta0)), rounded to a float.  A stored value's
// rounding error scales with its size, |M0 - s| w_i.  Storing Omega_i itself
// (s = 0) lets the rounding of a smooth field far from the front drift
// coherently (on the 4096^2 melting workload, 2.45e-5 of theta after 10,000
// steps against the FP64 form); s = the mean of M0 removes that but makes the
// values at the melting point (M0 = 0, where phi' is largest) the large ones
// (max |d phi| 1.04e-4).  Halfway between the two bounds both.  An exact sum
// over the whole grid, 9 us for 0.5 M nodes: one block took 240 us for 0.8 M
// and 1.2 ms for 4.2 M.
__global__ void __launch_bounds__(256) shift_kernel(const Problem* dprob, const double* __restrict__ theta0, DevStats* st)
{
    const Problem& pb = *dprob;
    const unsigned n = (unsigned)pb.nx * (unsigned)pb.ny;
    Fx v{0, 0ull};
    unsigned mag = 0u;
    for (unsigned k = blockIdx.x * 256u + threadIdx.x; k < n; k += gridDim.x * 256u) {
        const double th = theta0[k], m = pb.method == 1 ? th + (th > 0.0 ? pb.inv_ste : 0.0) : th;
        fx_add(v, to_fixed(m));
        mag = max(mag, fx_mag(m));
    }
    bool lost;
    v = block_sum(v, mag, lost);
    double total;
    const bool mine = last_block_total<&StepStripe::flux>(st, v, lost, total);
    if (mine && isnan(total)) {
        // a term without a fixed-point value: the plain sum, which may be NaN, infinite or huge
        total = 0.0;
        for (unsigned k = threadIdx.x; k < n; k += 32u) {
            const double th = theta0[k];
            total += pb.method == 1 ? th + (th > 0.0 ? pb.inv_ste : 0.0) : th;
        }
        total = warp_sum(total);
    }
    if (mine && threadIdx.x == 0) {
        const float sh = (float)(0.5 * total / (double)n);
        for (int b = 0; b < 2; ++b) *reinterpret_cast<float*>(static_cast<char*>(pb.state[b]) + pb.tail_off) = sh;
    }
}

// Initial populations; E(0) is summed exactly and published by the last block.
template <typename P>
__global__ void __launch_bounds__(256) init_state_kernel(const Problem* dprob, const double* __restrict__ theta0, int parity,
                                                         DevStats* st)
{
    const Problem& pb = *dprob;
    P* s = static_cast<P*>(pb.state[parity]);
    // FP32: the populations are stored less w_i sh
    const double sh = sizeof(P) == 4 ? (double)state_shift(pb, parity) : 0.0;
    const unsigned nx = (unsigned)pb.nx, n = nx * (unsigned)pb.ny;
    Fx e{0, 0ull};
    unsigned mag = 0u;
    auto add = [&](double v) {
        fx_add(e, to_fixed(v));
        mag = max(mag, fx_mag(v));
    };
    for (unsigned k = blockIdx.x * 256u + threadIdx.x; k < n; k += gridDim.x * 256u) {
        const int y = (int)(k / nx), x = (int)(k - (unsigned)y * nx);
        const long long at = (long long)(y + 1) * pb.pitch + x;
        double th = theta0[k], td;
        if (dirichlet_value(pb, x, y, td)) th = td;
        if (pb.method == 1) {
            // EEBM: equilibrium of H = theta + [theta > 0]/Ste (Algorithm 2): w_i theta,
            // and H - (1 - w_0) theta for i = 0
            const double H = th + (th > 0.0 ? pb.inv_ste : 0.0);
            for (int i = 0; i < pb.q; ++i)
                s[i * pb.plane + at] =
                    (P)(i == 0 ? H - (1.0 - lat_w(pb.q, 0)) * th - lat_w(pb.q, 0) * sh : lat_w(pb.q, i) * (th - sh));
            add(H);
            continue;
        }
        // one product per weight
        const P w0 = (P)(lat_w(pb.q, 0) * (th - sh)), w1 = (P)(lat_w(pb.q, 1) * (th - sh));
        s[at] = w0;
        for (int i = 1; i < min(pb.q, 5); ++i) s[i * pb.plane + at] = w1;
        if (pb.q == 9) {
            const P w2 = (P)(lat_w(9, 5) * (th - sh));
            for (int i = 5; i < 9; ++i) s[i * pb.plane + at] = w2;
        }
        if (pb.method == 2) {
            // ILFBM (Algorithm 1): the liquid fraction of the initial phase, plane q
            const double l = th > 0.0 ? 1.0 : 0.0;
            s[pb.q * pb.plane + at] = (P)l;
            add(th + l * pb.inv_ste);
            continue;
        }
        add(th + phi_of(th, pb.inv_delta) * pb.inv_ste);
    }
    bool lost;
    e = block_sum(e, mag, lost);
    double total;
    if (last_block_total<&StepStripe::energy>(st, e, lost, total) && threadIdx.x == 0) {
        st->energy = total;
        st->energy_prev = total;
        st->have_energy = 1;
    }
}

__global__ void wall_constants_kernel(Problem* probs, int nprob)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nprob) return;
    Problem& pb = probs[p];
    for (int k = 0; k < 4; ++k) {
        const double t = tanh(pb.wall_theta[k] * pb.inv_delta);
        pb.wall_tanh[k] = t;
        pb.wall_phi[k] = 0.5 + 0.5 * t;
        pb.wall_th_hi[k] = (float)pb.wall_theta[k];
        pb.wall_th_lo[k] = (float)(pb.wall_theta[k] - (double)pb.wall_th_hi[k]);
        pb.wall_slope[k] = (float)(0.5 * (1.0 - t) * (1.0 + t) * pb.inv_delta * pb.inv_ste);
    }
    pb.wall_dth_max = (float)(1e-4 * pb.delta);
    for (int k = 0; k < 4; ++k) {
        pb.wall_H[k] = pb.wall_theta[k] + (pb.wall_theta[k] > 0.0 ? pb.inv_ste : 0.0);
        pb.wall_H_hi[k] = (float)pb.wall_H[k];
        pb.wall_H_lo[k] = (float)(pb.wall_H[k] - (double)pb.wall_H_hi[k]);
    }
}

cudaError_t launch_wall_constants(Problem* dprobs, int nprob, cudaStream_t s)
{
    wall_constants_kernel<<<(nprob + 127) / 128, 128, 0, s>>>(dprobs, nprob);
    return cudaGetLastError();
}

template <typename P>
__global__ void fields_kernel(const Problem* dprob, int parity, double* theta, double* phi, double* H,
                              double* theta_plane)
{
    const Problem& pb = *dprob;
    const P* s = static_cast<const P*>(pb.state[parity]);
    const double sh = sizeof(P) == 4 ? (double)state_shift(pb, parity) : 0.0;   // FP32: stored less w_i sh
    const unsigned nx = (unsigned)pb.nx, n = nx * (unsigned)pb.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int y = (int)(k / nx), x = (int)(k - (unsigned)y * nx);
        double th = sh;
        for (int i = pb.q - 1; i >= 0; --i) th += (double)s[i * pb.plane + (long long)(y + 1) * pb.pitch + x];
        if (pb.method == 1) {
            // EEBM: M0 is the enthalpy; theta = Theta(H), liquid fraction min(max(Ste H, 0), 1)
            const double h = th;
            th = eebm_theta(h, pb.inv_ste);
            if (theta) theta[k] = th;
            if (phi) phi[k] = fmin(fmax(h * pb.ste, 0.0), 1.0);
            if (H) H[k] = h;
            if (theta_plane) theta_plane[(long long)y * pb.pitch + x] = th;
            continue;
        }
        // ILFBM: the liquid fraction is a field of its own (plane q)
        const double ph = pb.method == 2 ? (double)s[pb.q * pb.plane + (long long)(y + 1) * pb.pitch + x]
                                         : phi_of(th, pb.inv_delta);
        if (theta) theta[k] = th;
        if (phi) phi[k] = ph;
        if (H) H[k] = th + ph * pb.inv_ste;
        if (theta_plane) theta_plane[(long long)y * pb.pitch + x] = th;
    }
}

// Interface position along the lattice lines that start at `wall` (0 W, 1 E,
// 2 S, 3 N; node 0 on the wall), one warp per line: the first sign change of
// theta = M0(f) from the wall node's sign, linearly interpolated (node units;
// 0 if theta is 0 on the wall node, n - 1 if the sign never changes), and the
// wall side's phase fraction summed along the line minus the wall half cell.
// out[line] and out[nlines + line].
template <typename P>
__global__ void front_kernel(const Problem* dprob, int parity, int wall, double* out)
{
    const Problem& pb = *dprob;
    const P* s = static_cast<const P*>(pb.state[parity]);
    const bool rows = wall <= 1;
    const int nlines = rows ? pb.ny : pb.nx;
    const int n = rows ? pb.nx : pb.ny;
    const double sh = sizeof(P) == 4 ? (double)state_shift(pb, parity) : 0.0;   // FP32: stored less w_i sh
    const int lane = threadIdx.x & 31;
    const int w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int line = w0; line < nlines; line += nw) {
        auto theta_at = [&](int i) -> double {
            int x, y;
            if (wall == 0) { x = i; y = line; }
            else if (wall == 1) { x = pb.nx - 1 - i; y = line; }
            else if (wall == 2) { x = line; y = i; }
            else { x = line; y = pb.ny - 1 - i; }
            double th = sh;
            for (int k = pb.q - 1; k >= 0; --k) th += (double)s[k * pb.plane + (long long)(y + 1) * pb.pitch + x];
            return pb.method == 1 ? eebm_theta(th, pb.inv_ste) : th;
        };
        const double t0 = __shfl_sync(kFull, lane == 0 ? theta_at(0) : 0.0, 0);
        const bool hot = t0 > 0.0;
        double fz = t0 == 0.0 ? 0.0 : -1.0;   // -1: not found yet
        double prev_last = t0;                // theta of the node before this chunk
        double sum = 0.0;
        for (int c = 0; c < n; c += 32) {
            const int i = c + lane;
            const double th = i < n ? theta_at(i) : 0.0;
            if (i < n) {
                const double ph = phi_of(th, pb.inv_delta);
                sum += hot ? ph : 1.0 - ph;
            }
            if (fz < 0.0) {
                const bool cross = i >= 1 && i < n && (hot ? th <= 0.0 : th >= 0.0);
                const unsigned m = __ballot_sync(kFull, cross);
                double before = __shfl_up_sync(kFull, th, 1);
                if (lane == 0) before = prev_last;
                if (m) {
                    const int first = __ffs(m) - 1;
                    const double a = __shfl_sync(kFull, before, first);
                    const double b = __shfl_sync(kFull, th, first);
                    fz = (double)(c + first - 1) + a / (a - b);
                }
            }
            prev_last = __shfl_sync(kFull, th, 31);
        }
        if (fz < 0.0) fz = (double)(n - 1);
        sum = warp_sum(sum);
        if (lane == 0) {
            out[line] = fz;
            out[nlines + line] = sum - 0.5;
        }
    }
}

cudaError_t launch_front(int precision, const Problem* dprob, const Problem& hp, int parity, int wall, double* out,
                         cudaStream_t s)
{
    const int nlines = wall <= 1 ? hp.ny : hp.nx;
    const int blocks = (nlines + 3) / 4;
    if (precision == 1) front_kernel<float><<<blocks, 128, 0, s>>>(dprob, parity, wall, out);
    else front_kernel<double><<<blocks, 128, 0, s>>>(dprob, parity, wall, out);
    return cudaGetLastError();
}

// 256-thread blocks, at most eight per SM (every block adds to the last one's total)
static int grid_for(long long n) { return (int)((n + 255) / 256 < 152 * 8 ? (n + 255) / 256 : 152 * 8); }

cudaError_t launch_init_state(int precision, const Problem* dprob, const Problem& hp, const double* theta0,
                              int parity, DevStats* st, cudaStream_t s)
{
    const int g = grid_for((long long)hp.nx * hp.ny);
    // FP32 D2Q9 / D2Q5 states carry a shift (FP64 and D1Q3 tails stay zero)
    if (precision == 1 && hp.q != 3) {
        shift_kernel<<<g, 256, 0, s>>>(dprob, theta0, st);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (precision == 1) init_state_kernel<float><<<g, 256, 0, s>>>(dprob, theta0, parity, st);
    else init_state_kernel<double><<<g, 256, 0, s>>>(dprob, theta0, parity, st);
    return cudaGetLastError();
}

cudaError_t launch_fields(int precision, const Problem* dprob, const Problem& hp, int parity, double* theta,
                          double* phi, double* H, double* theta_plane, cudaStream_t s)
{
    const int g = grid_for((long long)hp.nx * hp.ny);
    if (precision == 1) fields_kernel<float><<<g, 256, 0, s>>>(dprob, parity, theta, phi, H, theta_plane);
    else fields_kernel<double><<<g, 256, 0, s>>>(dprob, parity, theta, phi, H, theta_plane);
    return cudaGetLastError();
}

}  // namespace lbm
