// D2Q9 and D2Q5 steps in one resident launch: a cooperative grid keeps its
// blocks on the SMs for all the steps of a call, four nodes per thread (FP64:
// one), the Newton solve of Eq. (14) in place, one grid barrier per step.
//
// What bounds it.  A step of a small lattice launched kernel by kernel is a
// chain of latencies: the wall kernels, the stencil, the side and the last
// Newton launch and the publication of the statistics, 45 us whatever the size
// (130 x 64 nodes, FP32).  Here a step ends at one barrier (load, arrival, poll
// and fence: 4 to 5 us on a lattice of a few hundred nodes), and its sums are
// added up by a block of their own while the next step runs.  Measured on the same
// states, us per step by the separate kernels / here: D2Q9 FP32 130 x 64 33 / 9.2,
// 1021 x 777 39 / 15.8, 4096^2 235 / 216; D2Q9 FP64 2048^2 310 / 154; D2Q5 FP32
// 4096^2 179 / 123, FP64 401^2 117 / 17.
//
// A step has two passes over what a block owns, between barriers of the block:
//  1. plain nodes.  A warp takes a group of 32 N consecutive columns of one of
//     the rows 1 .. ny-2 (N = 4 in FP32, one 128-bit load per plane, as the
//     flat kernel; 1 in FP64).  Saturated nodes are updated, the nodes that
//     need the Newton solve go to a queue in shared memory.
//  2. items of 32 nodes, one per lane: the queued nodes, gathered densely so
//     that a solve (a chain of 43 or 44 FP64 instructions of 64 cycles) serves full
//     warps, the rows 0 and ny-1, and the column groups at the W and E walls.
// Groups of a wave lie side by side (their halo rows and columns meet in L1 and
// L2), and a block's place in the wave rotates from wave to wave, so that the
// groups of a front band spread over all SMs.  A lattice of few nodes has no
// first pass: every node is an item.
//
// Memory order.  A step reads state[p] and writes state[p ^ 1].  Every read of
// a state is a plain load (never the read-only path, which is not coherent
// with stores of the same launch); the barrier's fences make a step's stores
// visible and drop stale L1 lines.
//
// Arithmetic: that of the kernels in step_d2q9.cu / step_d2q5.cu node by node.
// FP64 form: the zeroth moment is summed in block floating point with integer
// instructions (sum_q) and w_i c takes two multiplications, 11 FP64
// instructions per D2Q9 node instead of 28, on a pipe that takes one warp
// instruction per 64 cycles of an SM quarter.  That pipe is 63 % busy at 2048^2
// and DRAM 46 % of its peak; the rest is latency at 24 warps per SM (stalls per
// issue: loads 3.6, fixed latencies 2.6, barrier 2.1, shared memory 1.9).
#include <algorithm>

#include "d2q5_row.cuh"
#include "d2q9_row.cuh"
#include "resident.cuh"

// Lattices of up to this many units (32 columns of a row) per computing block take no
// first pass.  us per step with items alone / with two passes: D2Q9 FP32 128^2 9.0 /
// 14.5, 160^2 10.1 / 10.9, 256^2 14.2 / 10.6, FP64 128^2 13.3 / 16.9, 256^2 28.9 / 17.1,
// D2Q5 FP32 128^2 8.1 / 20.8, 160^2 9.1 / 11.5, 256^2 12.7 / 11.6 (8 units per block lie
// near 195^2).
#ifndef LBM_RES_SCALAR
#define LBM_RES_SCALAR 8
#endif

namespace lbm {

// ---------------------------------------------------------------- arguments
struct ResidentArgs : ResidentCommon {
    Problem pb;                 // by value: constants come from the parameter bank
    int parity;
    double* rec;                // theta' planes of the steps (ny x pitch each), or NULL
    int strips, th, tiles;      // first pass: column strips, rows of a tile, tiles (0: no first pass)
    int nseg;                   // 32-column segments of a row (the items of full rows)
    int items;                  // second pass: items without the queue
    int rot;
};

// ---------------------------------------------------------------- one node
template <typename P> struct LaneAcc;
template <> struct LaneAcc<float> {
    ff s{0.f, 0.f};
    __device__ void add(float v) { ff_add(s, v); }
    __device__ bool lost() const { return false; }
    __device__ Fx total() const
    {
        ff t = s;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(kFull, t.hi, o), l = __shfl_xor_sync(kFull, t.lo, o);
            ff_add(t, h);
            t.lo += l;
        }
        Fx f = float_to_fixed(t.hi);
        fx_add(f, float_to_fixed(t.lo));
        return f;
    }
};
template <> struct LaneAcc<double> {
    Fx s{0, 0ull};
    unsigned mag = 0u;
    __device__ void add(double v)
    {
        fx_add(s, to_fixed(v));
        mag = max(mag, fx_mag(v));
    }
    __device__ bool lost() const { return __any_sync(kFull, mag >= kFxMag); }
    __device__ Fx total() const { return fx_tree(s); }
};

// One item: a node (x, y) per lane, anywhere in the lattice (idle lanes: not
// valid).  w: the warp's sums in shared memory, where lane 0 adds what few
// items have.  A resident state has fewer than 2^31 elements (32-bit indices).
template <typename P, int Q, bool EEBM>
__device__ __forceinline__ void item_update(const Problem& pb, DevStats* st, const P* src, P* dst, double* rec, int x, int y,
                                            bool valid, int lane, float sh, LaneAcc<P>& acc, ResidentSlot* w)
{
    const int nx = pb.nx, ny = pb.ny, pitch = pb.pitch, plane = (int)pb.plane;
    const int at = (y + 1) * pitch + x;
    P u[Q], q[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        u[i] = q[i] = (P)0;
        if (valid) {
            u[i] = src[at + i * plane];
            q[i] = i == 0 ? u[0] : src[at + i * plane - d2_ey(i) * pitch - d2_ex(i)];   // Omega_i(y - e_i)
        }
    }
    int wall = -1;
    const bool edge = valid && (x == 0 || x == nx - 1 || y == 0 || y == ny - 1);
    if (__any_sync(kFull, edge)) {
        Fx fl{0, 0ull};
        unsigned mag = 0u;
        if (edge) {
            // copies: the closures take addresses, and u, q stay in registers elsewhere
            P qq[Q], uu[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                qq[i] = q[i];
                uu[i] = u[i];
            }
            if constexpr (Q == 9) {
                if constexpr (sizeof(P) == 4) {
                    const ff t = wall_closure_f(qq, uu, x, y, pb, wall, sh);
                    fl = float_to_fixed(t.hi);
                    fx_add(fl, float_to_fixed(t.lo));
                } else {
                    const double t = wall_closure_d(qq, uu, x, y, pb, wall);
                    fl = to_fixed(t);
                    mag = fx_mag(t);
                }
            } else {
                P nq[5];
                if (pb.bb_mode == 2) pulled5_inward<P>(src, pb, x, y, nq);
                if constexpr (sizeof(P) == 4) {
                    const ff t = wall5_closure_f(qq, uu, nq, x, y, pb, wall, sh);
                    fl = float_to_fixed(t.hi);
                    fx_add(fl, float_to_fixed(t.lo));
                } else {
                    const double t = wall5_closure_d(qq, uu, nq, x, y, pb, wall);
                    fl = to_fixed(t);
                    mag = fx_mag(t);
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) q[i] = qq[i];
        }
        fl = fx_tree(fl);
        const bool lost = sizeof(P) == 8 && __any_sync(kFull, mag >= kFxMag);
        if (lane == 0) {
            fx_add(w->f, fl);
            if (lost) w->lost |= kLostFlux;
        }
    }
    const P omc = sizeof(P) == 4 ? (P)pb.omc_f : (P)pb.omc;
    if constexpr (EEBM) {
        // Algorithm 2: H = M0(q), theta = Theta(H); stored values less w_i sh
        const P om = (P)1 - omc, w0 = lat_wp<P>(Q, 0);
        P Hs = (P)0;
        if constexpr (sizeof(P) == 8) {
            Hs = sum_q<Q>(q);
        } else {
#pragma unroll
            for (int i = Q - 1; i >= 0; --i) Hs += q[i];
        }
        const P H = Hs + (P)sh;
        const P th = eebm_theta(H, (P)pb.inv_ste);
        if (valid) {
            acc.add(Hs);
            dst[at] = fma(omc, q[0], om * eebm_rest(H, th, w0, (P)sh));
            const P tr = th - (P)sh;
#pragma unroll
            for (int i = 1; i < Q; ++i) dst[at + i * plane] = fma(omc, q[i], om * lat_wp<P>(Q, i) * tr);
            if (rec) rec[y * pitch + x] = (double)th;
        }
        if constexpr (sizeof(P) == 4) {
            const unsigned n = (unsigned)__popc(__ballot_sync(kFull, valid));
            if (lane == 0) w->shifted += n;
        }
        return;
    }
    // saturation from FP32 sums
    float tf = 0.f;
    P m0;        // FP32: M0(q) less sh, the plain sum
    float mt;
    if constexpr (sizeof(P) == 4) {
        if constexpr (Q == 9) {
#pragma unroll
            for (int i = 0; i < Q; ++i) tf += u[i];
        } else {
#pragma unroll
            for (int i = Q - 1; i >= 0; --i) tf += u[i];
        }
        tf += sh;
        m0 = 0.f;
#pragma unroll
        for (int i = Q - 1; i >= 0; --i) m0 += q[i];
        mt = m0 + sh;
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) tf += approx_float(u[i]);
        m0 = sum_q<Q>(q);
        mt = approx_float(m0);
    }
    const float marg = 1e-5f * (1.0f + fabsf(tf)), thr = pb.sat_f;
    const bool liq = tf >= thr + marg && mt >= thr + marg;
    const bool sat = liq || (tf <= -thr - marg && mt <= -thr - marg);
    const bool dir = wall >= 0;
    const bool solve = valid && !dir && !sat;
    const unsigned solving = __ballot_sync(kFull, solve);
    const bool plain = valid && !dir && sat;
    {
        const unsigned n = (unsigned)__popc(__ballot_sync(kFull, plain && liq));
        const unsigned m = sizeof(P) == 4 ? (unsigned)__popc(__ballot_sync(kFull, plain)) : 0u;
        if (lane == 0) {
            w->liquid += n;
            w->shifted += m;
        }
    }
    if (plain) acc.add(m0);
    // c = theta' - (1 - omega) m0 (FP32: less omega sh); saturated: theta' = m0, c = omega m0
    P c = sizeof(P) == 4 ? (P)(pb.omega_f * (float)m0) : (P)(pb.omega * (double)m0);
    double tn = 0.0;
    if (rec) tn = sizeof(P) == 4 ? widen((float)m0) + widen(sh) : (double)m0;
    if (__any_sync(kFull, dir)) {
        // theta' = theta_D
        Fx e{0, 0ull};
        if (dir) {
            if constexpr (sizeof(P) == 4) {
                ff mm{0.f, 0.f};
#pragma unroll
                for (int i = Q - 1; i >= 0; --i) ff_add(mm, q[i]);
                c = (P)(((pb.wall_th_hi[wall] - sh) - (float)omc * mm.hi) + (pb.wall_th_lo[wall] - (float)omc * mm.lo));
                e = float_to_fixed(pb.wall_th_hi[wall]);
                fx_add(e, float_to_fixed(pb.wall_th_lo[wall]));
            } else {
                c = (P)(pb.wall_theta[wall] - pb.omc * (double)m0);
                e = to_fixed(pb.wall_theta[wall]);
            }
            tn = pb.wall_theta[wall];
        }
        e = fx_tree(e);
        if (lane == 0) fx_add(w->e, e);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned b = __ballot_sync(kFull, dir && wall == k);
            if (lane == 0) w->dir[k] += (unsigned)__popc(b);
        }
    }
    if (solving) {
        // the local Newton solve of Eq. (14)
        Fx e{0, 0ull};
        int it = 0;
        if (solve) {
            double mm, tt, shd = 0.0;   // m0 and theta less the shift
            if constexpr (sizeof(P) == 4) {
                ff fm{0.f, 0.f}, ft{0.f, 0.f};
#pragma unroll
                for (int i = Q - 1; i >= 0; --i) {
                    ff_add(ft, u[i]);
                    ff_add(fm, q[i]);
                }
                shd = widen(sh);
                mm = ff_to_double(fm);
                tt = ff_to_double(ft);
            } else {
                mm = (double)m0;
                tt = sum_q<Q>(u);
            }
            const NewtonNode nr = newton_mixed<sizeof(P) == 4>(mm, tt, shd, pb);
            if (!nr.ok) atomicCAS(&st->error, 0, 3);
            tn = nr.tns + shd;
            c = (P)fma(-pb.omc, mm, nr.tns);
            e = to_fixed(nr.ens);   // FP32: less the shift
            it = nr.iters;
        }
        e = fx_tree(e);
        const unsigned its = __reduce_add_sync(kFull, (unsigned)it);
        const int mx = __reduce_max_sync(kFull, it);
        if (lane == 0) {
            fx_add(w->e, e);
            w->newton += (unsigned)__popc(solving);
            if (sizeof(P) == 4) w->shifted += (unsigned)__popc(solving);
            w->iters += its;
            w->maxit = max(w->maxit, mx);
        }
    }
    // Omega~_i = (1-omega) q_i + w_i c
    P wc[3];
    if constexpr (sizeof(P) == 4) {
        wc[0] = lat_wp<P>(Q, 0) * c;
        wc[1] = lat_wp<P>(Q, 1) * c;
        wc[2] = Q == 9 ? lat_wp<P>(Q, Q - 1) * c : (P)0;
    } else {
        // one multiplication: 4/9 and 1/36 are 4 and 1/4 times 1/9 (D2Q5: 1/3 = 2/6),
        // and so are their roundings
        const double v = lat_wp<double>(Q, 1) * (double)c;
        wc[0] = (P)scale2(v, Q == 9 ? 2 : 1);
        wc[1] = (P)v;
        wc[2] = Q == 9 ? (P)scale2(v, -2) : (P)0;
    }
    if (valid) {
#pragma unroll
        for (int i = 0; i < Q; ++i) dst[at + i * plane] = fma(omc, q[i], wc[i == 0 ? 0 : (i <= 4 ? 1 : 2)]);
        if (rec) rec[y * pitch + x] = tn;
    }
}

// ---------------------------------------------------------------- plain nodes
// The columns x0 .. x0 + N - 1 per lane of row y, 1 <= y <= ny-2 (the same for
// the warp).  Lanes that hold column 0 or nx-1 or reach past nx leave theirs to
// the second pass (cold).  Nodes to solve: queued, q left for the second pass.
__device__ __forceinline__ void ld4(const float* p, float (&v)[4])
{
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

// The queue (dynamic shared memory) has room for every node of kResidentWaves
// waves of the first pass; the second pass follows that many waves.  FP32: 64 and
// 96 KB; more costs L1 (8 / 16 waves, us per step: D2Q9 4096^2 218 / 222, EEBM 201 / 210,
// D2Q5 124 / 156).  FP64: 48 KB (8 / 16 waves: D2Q9 2048^2 177 / 166, 4096^2 608 / 571).
template <typename P> constexpr int kResidentWaves = sizeof(P) == 4 ? 8 : 16;

struct ResidentQueue {
    unsigned count;
    unsigned* node;     // (y << 16) + x
};

template <int Q, bool EEBM>
__device__ __forceinline__ void plain_update(const Problem& pb, const float* src, float* dst, double* rec, int x0,
                                             int y, int lane, float sh, LaneAcc<float>& acc, ResidentSlot* w,
                                             ResidentQueue* queue)
{
    const int nx = pb.nx, pitch = pb.pitch, plane = (int)pb.plane;
    const int at = (y + 1) * pitch + x0;
    const bool cold = x0 == 0 || x0 + 3 >= nx - 1;
    const float* row = src + at;
    // every load of a cold lane stays inside the buffer
    float u[Q][4], q[Q][4];
#pragma unroll
    for (int i = 0; i < Q; ++i) ld4(row + i * plane, u[i]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        float v[4];
        const float* p = row + i * plane - d2_ey(i) * pitch;
        if (d2_ey(i) == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = u[i][k];
        } else {
            ld4(p, v);
        }
        if (d2_ex(i) == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) q[i][k] = v[k];
        } else if (d2_ex(i) == 1) {
            q[i][0] = p[-1];
            q[i][1] = v[0]; q[i][2] = v[1]; q[i][3] = v[2];
        } else {
            q[i][0] = v[1]; q[i][1] = v[2]; q[i][2] = v[3];
            q[i][3] = p[4];
        }
    }
    const float omc = pb.omc_f;
    if constexpr (EEBM) {
        const float om = 1.0f - omc, inv_ste = pb.inv_ste_f, w0 = lat_wp<float>(Q, 0);
        float hs = 0.f;
        double thn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float Hs = 0.f;   // H less the shift
#pragma unroll
            for (int i = Q - 1; i >= 0; --i) Hs += q[i][k];
            hs += Hs;
            const float H = Hs + sh;
            const float th = eebm_theta(H, inv_ste);
            thn[k] = widen(th);
            q[0][k] = fmaf(omc, q[0][k], om * eebm_rest(H, th, w0, sh));
            const float tr = th - sh;
#pragma unroll
            for (int i = 1; i < Q; ++i) q[i][k] = fmaf(omc, q[i][k], om * lat_wp<float>(Q, i) * tr);
        }
        const unsigned n = (unsigned)__popc(__ballot_sync(kFull, !cold));
        if (lane == 0) w->shifted += 4u * n;
        if (!cold) {
            acc.add(hs);
#pragma unroll
            for (int i = 0; i < Q; ++i) stv_n(dst + at + i * plane, q[i]);
            if (rec) st_rec<4>(rec + y * pitch + x0, thn);
        }
        return;
    }
    const float om_f = pb.omega_f, thr = pb.sat_f;
    float c[4], m0[4], esum = 0.f;
    unsigned solve = 0, liquid = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float tf = 0.f, mf = 0.f;
        if constexpr (Q == 9) {
#pragma unroll
            for (int i = 0; i < Q; ++i) tf += u[i][k];
        } else {
#pragma unroll
            for (int i = Q - 1; i >= 0; --i) tf += u[i][k];
        }
        tf += sh;   // theta
#pragma unroll
        for (int i = Q - 1; i >= 0; --i) mf += q[i][k];   // M0(q) - sh
        const float mt = mf + sh;
        const float marg = 1e-5f * (1.0f + fabsf(tf));
        const bool liq = tf >= thr + marg && mt >= thr + marg;
        const bool sat = liq || (tf <= -thr - marg && mt <= -thr - marg);
        c[k] = om_f * mf;   // c - omega sh = omega (m0 - sh)
        m0[k] = mf;
        if (sat) {
            esum += mf;
            liquid += liq ? 1u : 0u;
        } else {
            solve |= 1u << k;
        }
    }
    if (cold) {
        solve = liquid = 0u;
        esum = 0.f;
    }
    acc.add(esum);
    // the warp's counts: liquid, and plain nodes (whose energy terms lack the shift)
    const unsigned plainc = cold ? 0u : 4u - (unsigned)__popc(solve);
    const unsigned n = __reduce_add_sync(kFull, liquid | (plainc << 16));
    if (lane == 0) {
        w->liquid += n & 0xffffu;
        w->shifted += n >> 16;
    }
    if (!cold) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float wi = lat_wp<float>(Q, i);
            float o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = fmaf(omc, q[i][k], wi * c[k]);
            stv_n(dst + at + i * plane, o);   // (a queued node's values are replaced by the second pass)
        }
        if (rec) {
            double thn[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) thn[k] = widen(m0[k]) + widen(sh);
            st_rec<4>(rec + y * pitch + x0, thn);
        }
    }
    if (__any_sync(kFull, solve != 0u)) {
        const unsigned cnt = (unsigned)__popc(solve);
        unsigned incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        unsigned base = 0;
        if (lane == 31) base = atomicAdd(&queue->count, incl);
        unsigned slot = __shfl_sync(kFull, base, 31) + incl - cnt;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((solve >> k) & 1u) queue->node[slot++] = ((unsigned)y << 16) + (unsigned)(x0 + k);
    }
}

// FP64: one column per lane.
template <int Q, bool EEBM>
__device__ __forceinline__ void plain_update(const Problem& pb, const double* src, double* dst, double* rec, int x,
                                             int y, int lane, float sh, LaneAcc<double>& acc, ResidentSlot* w,
                                             ResidentQueue* queue)
{
    const int nx = pb.nx, pitch = pb.pitch, plane = (int)pb.plane;
    const int at = (y + 1) * pitch + x;
    const bool cold = x == 0 || x >= nx - 1;
    double q[Q];
    float tf = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) q[i] = src[at + i * plane - d2_ey(i) * pitch - d2_ex(i)];
    if constexpr (!EEBM) {
        float u[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) u[i] = approx_float(i == 0 ? q[0] : src[at + i * plane]);
#pragma unroll
        for (int i = 0; i < Q; ++i) tf += u[i];
    }
    const double m0 = sum_q<Q>(q);
    if constexpr (EEBM) {
        const double th = eebm_theta(m0, pb.inv_ste), omc = pb.omc, om = 1.0 - omc;
        if (!cold) {
            acc.add(m0);
            dst[at] = fma(omc, q[0], om * eebm_rest(m0, th, lat_wp<double>(Q, 0), 0.0));
            const double t1 = (om * lat_wp<double>(Q, 1)) * th;
            const double t2 = Q == 9 ? scale2(t1, -2) : 0.0;
#pragma unroll
            for (int i = 1; i < Q; ++i) dst[at + i * plane] = fma(omc, q[i], i <= 4 ? t1 : t2);
            if (rec) rec[y * pitch + x] = th;
        }
        return;
    }
    const float mt = approx_float(m0), thr = pb.sat_f;
    const float marg = 1e-5f * (1.0f + fabsf(tf));
    const bool liq = tf >= thr + marg && mt >= thr + marg;
    const bool sat = liq || (tf <= -thr - marg && mt <= -thr - marg);
    const bool solve = !cold && !sat;
    const unsigned nliq = (unsigned)__popc(__ballot_sync(kFull, !cold && liq));
    if (lane == 0) w->liquid += nliq;
    if (!cold && sat) {
        // w_i c, c = omega m0: one multiplication by a weight, 4/9 and 1/36 being 4 and 1/4
        // times 1/9 (D2Q5: 1/3 = 2/6), and so their roundings.  Not (omega w_i) m0, which would
        // save the other one: the rounding of omega w_i, up to 2^-53 of it whatever m0, would
        // enter every node at every step (at tau = 0.62 the coefficients would miss a sum of 1
        // by 1.4e-16 on D2Q9, 2.2e-16 on D2Q5, against 0.9e-16 by the weights alone)
        acc.add(m0);
        const double v = lat_wp<double>(Q, 1) * (pb.omega * m0);
        const double v0 = scale2(v, Q == 9 ? 2 : 1), v2 = Q == 9 ? scale2(v, -2) : 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) dst[at + i * plane] = fma(pb.omc, q[i], i == 0 ? v0 : (i <= 4 ? v : v2));
        if (rec) rec[y * pitch + x] = m0;
    }
    const unsigned solving = __ballot_sync(kFull, solve);
    if (solving) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&queue->count, (unsigned)__popc(solving));
        const unsigned slot = __shfl_sync(kFull, base, 0) + (unsigned)__popc(solving & ((1u << lane) - 1u));
        if (solve) queue->node[slot] = ((unsigned)y << 16) + (unsigned)x;
    }
}

// One block per SM.  D2Q9 in FP32: 512 threads leave 128 registers, without spills,
// and 16 warps take two 8-row tiles at a time (us per step with 768 / 512 threads:
// 4096^2 221 / 218, EEBM 212 / 201); D2Q5 in FP32 streams less per node and wants
// the warps (4096^2, 640 / 768: 140 / 124), and so does FP64, whose sums are integer
// work beside the FP64 pipe (2048^2, 640 / 768: D2Q9 183 / 166, D2Q5 145 / 130).
template <typename P, int Q> constexpr int kResidentThreads = sizeof(P) == 4 && Q == 9 ? 512 : 768;

template <typename P, int Q, bool EEBM>
__global__ void __launch_bounds__(kResidentThreads<P, Q>, 1) resident_kernel(const __grid_constant__ ResidentArgs a)
{
    __shared__ ResidentSlot wsum[2][kResidentThreads<P, Q> / 32];   // by step parity
    __shared__ ResidentQueue queue;
    extern __shared__ unsigned queue_nodes[];
    __shared__ unsigned next_item;
    __shared__ bool ok_s;
    constexpr int N = sizeof(P) == 4 ? 4 : 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int nb = gridDim.x - 1;   // computing blocks; the last block adds up the statistics
    if ((int)blockIdx.x == nb) {
        resident_stats(a, a.pb, (unsigned)nb);
    } else {
        const Problem& pb = a.pb;
        const int nx = pb.nx, ny = pb.ny;
        const float sh = sizeof(P) == 4 ? state_shift(pb, 0) : 0.f;   // the same in both buffers
        const int row_tiles = a.tiles ? a.tiles / a.strips : 0;       // a strip's tiles follow one another
        const int g = nwb / a.th;                                     // tiles a block takes at a time
        const int xe = max(N, (nx - 1) / N * N);                      // the E wall's column group
        if (threadIdx.x == 0) {
            queue.count = next_item = 0u;
            queue.node = queue_nodes;
        }
        for (int k = threadIdx.x; k < 2 * nwb * (int)(sizeof(ResidentSlot) / 16); k += blockDim.x)
            reinterpret_cast<uint4*>(k < nwb * (int)(sizeof(ResidentSlot) / 16) ? wsum[0] : wsum[1])
                [k % (nwb * (int)(sizeof(ResidentSlot) / 16))] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        bool ok = true;
        for (int s = 0; ok && s < a.nsteps; ++s) {
            const int p = (a.parity + s) & 1;
            const P* src = static_cast<const P*>(pb.state[p]);
            P* dst = static_cast<P*>(pb.state[p ^ 1]);
            double* rec = a.rec ? a.rec + (long long)s * ny * pb.pitch : nullptr;
            ResidentSlot* w = &wsum[s & 1][warp];
            LaneAcc<P> acc;
            // the items that are not queued: this block's share of the rows 0 and ny-1 (or of all
            // rows) and of the W and E column groups
            unsigned own = a.items > (int)blockIdx.x ? (unsigned)(a.items - 1 - (int)blockIdx.x) / nb + 1u : 0u;
            int place = blockIdx.x, t0 = 0;
            do {
                for (int k = 0; k < kResidentWaves<P> && t0 < a.tiles; ++k, t0 += nb * g) {
                    // a wave: g tiles of every block, the tiles of a strip dealt round the blocks
                    const int t = t0 + warp / a.th * nb + place;
                    place += a.rot;
                    if (place >= nb) place -= nb;
                    if (warp / a.th >= g || t >= a.tiles) continue;
                    const int strip = t / row_tiles;
                    const int y = 1 + (t - strip * row_tiles) * a.th + warp % a.th;
                    const int x0 = (strip * 32 + lane) * N;
                    if (y < ny - 1) plain_update<Q, EEBM>(pb, src, dst, rec, x0, y, lane, sh, acc, w, &queue);
                }
                if (a.tiles) __syncthreads();
                const unsigned queued = queue.count;
                const unsigned total = own + (queued + 31u) / 32u;
                // the first items, the block's own among them, are dealt, the others taken: an FP32
                // lane adds its nodes' terms in float pairs, whose rounding depends on their order;
                // the queued nodes' terms are added exactly
                const unsigned dealt = own > (unsigned)nwb ? (own + nwb - 1u) / nwb * nwb : (unsigned)nwb;
                unsigned it = (unsigned)warp;
                while (it < total) {
                    int x = 0, y = 0;
                    bool valid;
                    if (it < own) {
                        const int e = (int)(it * nb + blockIdx.x);
                        const int rows = a.tiles ? 2 * a.nseg : a.items;
                        if (e < rows) {
                            const int r = e / a.nseg;
                            x = (e - r * a.nseg) * 32 + lane;
                            y = a.tiles ? (r ? ny - 1 : 0) : r;
                            valid = x < nx;
                        } else {
                            // 2 N columns of 32 / (2 N) rows
                            const int k = lane % (2 * N);
                            y = 1 + (e - rows) * (32 / (2 * N)) + lane / (2 * N);
                            x = k < N ? k : xe + k - N;
                            valid = y < ny - 1 && x < nx;
                        }
                    } else {
                        const unsigned j = (it - own) * 32u + (unsigned)lane;
                        valid = j < queued;
                        if (valid) {
                            const unsigned n = queue.node[j];
                            x = (int)(n & 0xffffu);
                            y = (int)(n >> 16);
                        }
                    }
                    item_update<P, Q, EEBM>(pb, a.stats, src, dst, rec, x, y, valid, lane, sh, acc, w);
                    it += nwb;
                    if (it < dealt) continue;
                    if (total <= dealt) break;
                    if (lane == 0) it = dealt + atomicAdd(&next_item, 1u);
                    it = __shfl_sync(kFull, it, 0);
                }
                own = 0u;
                if (t0 < a.tiles) {
                    __syncthreads();
                    if (threadIdx.x == 0) queue.count = next_item = 0u;
                    __syncthreads();
                }
            } while (t0 < a.tiles);
            const Fx e = acc.total();
            const bool lost = acc.lost();
            if (lane == 0) {
                fx_add(w->e, e);
                if (lost) w->lost |= kLostEnergy;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                queue.count = next_item = 0u;
                if (s != a.withhold || blockIdx.x != 0) bar_arrive(&a.bar->count);
                ok_s = s + 1 == a.nsteps || bar_wait(a.bar, &a.bar->count, (unsigned)(s + 1) * nb, a.wait_ns);
            } else if (warp == 1) {
                // while thread 0 waits
                resident_emit(a, s, nb, lane, nwb, wsum[s & 1]);
            }
            __syncthreads();
            ok = ok_s;
        }
        if (threadIdx.x == 0) bar_arrive(&a.bar->count);   // the last step's sums are out
    }
    bar_leave(a.bar);
}

// ---------------------------------------------------------------- batches, FP32 D2Q9
// Many problems in one resident launch.  A warp takes a whole unit of one
// problem: a tile of 128 columns x 8 rows, whose nodes to solve it queues for
// itself and solves right after the rows (280 of a vertical front's tile fill
// nine warps' worth densely), so that solves, bound by latency and the FP64 pipe,
// and streaming run side by side on every SM; a stretch of an S or N row; or 32
// rows of the W and E column groups.  Sums go to the unit's problem by atomics,
// in sets by step parity that the statistics block reads, clears and publishes
// while the next step runs.  256 problems of 64^2 to 1024^2 (58.6 M nodes, 3.9 M of
// them solved), us per step: 1,440 by separate kernels, whose solves came after the
// streaming for the most part; 1,320 here with the units dealt to the warps, 1,025
// with a counter per block (a front's tile lasts several times a plain one's).
struct ResidentBatchArgs : ResidentCommon {
    const Problem* probs;
    int count;                  // problems
    const int4* units;          // (problem, kind: 0 tile, 1 row, 2 column groups; strip or side; first row)
    int nunits, parity;
    StepStripe* acc;            // 2 x count x kBatchStripes
    int* maxit;                 // 2 x count
};

constexpr int kBatchThreads = 512, kBatchWarps = kBatchThreads / 32;
constexpr int kBatchStripes = 4;

// Adds the warp's sums to its problem's and clears them.
__device__ __forceinline__ void batch_flush(StepStripe* c, int* maxit, LaneAcc<float>& acc, ResidentSlot* w, int lane)
{
    const Fx e = acc.total();
    acc = LaneAcc<float>{};
    if (lane == 0) {
        fx_add(w->e, e);
        acc_add_fx(&c->energy, w->e);
        acc_add_fx(&c->flux, w->f);
        if (w->liquid) atomicAdd(&c->liquid, (unsigned long long)w->liquid);
        if (w->shifted) atomicAdd(&c->shifted, (unsigned long long)w->shifted);
        for (int k = 0; k < 4; ++k)
            if (w->dir[k]) atomicAdd(&c->dir[k], (unsigned long long)w->dir[k]);
        if (w->newton) {
            atomicAdd(&c->newton, (unsigned long long)w->newton);
            atomicAdd(&c->iters, (unsigned long long)w->iters);
            atomicMax(maxit, w->maxit);
        }
        *w = ResidentSlot{};
    }
    __syncwarp();
}

// The statistics block: a thread per problem.
static __device__ __noinline__ void batch_stats(const ResidentBatchArgs& a, unsigned nb, bool* ok_s)
{
    bool ok = true;
    for (int s = 0; ok && s < a.nsteps; ++s) {
        if (threadIdx.x == 0) *ok_s = bar_wait(a.bar, &a.bar->count, (unsigned)(s + 1) * nb, a.wait_ns);
        __syncthreads();
        ok = *ok_s;
        if (!ok) break;
        for (int p = threadIdx.x; p < a.count; p += blockDim.x) {
            StepStripe* c = a.acc + ((size_t)(s & 1) * a.count + p) * kBatchStripes;
            int* mx = a.maxit + (size_t)(s & 1) * a.count + p;
            StatSums t = {};
            for (int k = 0; k < kBatchStripes; ++k) stripe_take(c + k, t);
            DevStats* st = &a.stats[a.probs[p].stats];
            st->cur_maxit = *reinterpret_cast<volatile int*>(mx);
            *reinterpret_cast<volatile int*>(mx) = 0;
            __threadfence();
            publish_totals(st, &a.probs[p], t);
        }
        __syncthreads();
        if (threadIdx.x == 0) bar_arrive(&a.bar->read[0]);   // the step's set is read and clear
    }
    if (!ok && threadIdx.x == 0)
        for (int p = 0; p < a.count; ++p) atomicExch(&a.stats[p].error, 4);   // LBM_ERR_TIMEOUT
}

// A block at its end; after a wait that ran out the last one clears the sums that
// nobody has read, so that the next launch does not add to them.
static __device__ __noinline__ void batch_leave(const ResidentBatchArgs& a)
{
    if (!bar_leave(a.bar)) return;
    unsigned long long* w = reinterpret_cast<unsigned long long*>(a.acc);
    for (size_t k = threadIdx.x; k < (size_t)2 * a.count * kBatchStripes * (sizeof(StepStripe) / 8); k += blockDim.x) w[k] = 0ull;
    for (int k = threadIdx.x; k < 2 * a.count; k += blockDim.x) a.maxit[k] = 0;
}

__global__ void __launch_bounds__(kBatchThreads, 1) resident_batch_kernel(const __grid_constant__ ResidentBatchArgs a)
{
    __shared__ ResidentSlot wsum[kBatchWarps];
    __shared__ ResidentQueue queues[kBatchWarps];
    __shared__ unsigned next_unit;
    __shared__ bool ok_s;
    extern __shared__ unsigned batch_nodes[];   // 1,024 per warp: a tile's nodes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nb = gridDim.x - 1;   // computing blocks; the last block publishes the statistics
    if ((int)blockIdx.x == nb) {
        batch_stats(a, (unsigned)nb, &ok_s);
        batch_leave(a);
        return;
    }
    ResidentSlot* w = &wsum[warp];
    ResidentQueue* queue = &queues[warp];
    if (lane == 0) {
        *w = ResidentSlot{};
        queue->count = 0u;
        queue->node = batch_nodes + warp * 1024;
        next_unit = 0u;
    }
    __syncthreads();
    const int rot = (int)(0.618f * nb);
    bool ok = true;
    for (int s = 0; ok && s < a.nsteps; ++s) {
        const int p = (a.parity + s) & 1;
        LaneAcc<float> acc;
        // a block's units are dealt (one of every nb in a row, at a rotating place) and its warps
        // take them from a counter: a front's tile lasts several times a plain one's
        for (;;) {
            unsigned i = 0;
            if (lane == 0) i = atomicAdd(&next_unit, 1u);
            i = __shfl_sync(kFull, i, 0);
            const int u = (int)i * nb + (int)((blockIdx.x + i * (unsigned)rot) % (unsigned)nb);
            if ((int)i * nb >= a.nunits) break;
            if (u >= a.nunits) continue;
            const int4 e = __ldg(a.units + u);
            const Problem& pb = a.probs[e.x];
            DevStats* st = &a.stats[pb.stats];
            const float* src = static_cast<const float*>(pb.state[p]);
            float* dst = static_cast<float*>(pb.state[p ^ 1]);
            const float sh = state_shift(pb, 0);   // the same in both buffers
            const int nx = pb.nx, ny = pb.ny;
            if (e.y == 0) {
                const int x0 = e.z * 128 + 4 * lane;
                for (int y = max(e.w, 1); y < min(e.w + 8, ny - 1); ++y)
                    plain_update<9, false>(pb, src, dst, nullptr, x0, y, lane, sh, acc, w, queue);
                __syncwarp();
            }
            // the items: the tile's queue; 4 stretches of 32 nodes of a row; 8 times 4 rows of the
            // W and E column groups
            const unsigned queued = e.y == 0 ? queue->count : 0u;
            const int items = e.y == 0 ? (int)((queued + 31u) / 32u) : (e.y == 1 ? 4 : 8);
            const int xe = max(4, (nx - 1) / 4 * 4);
            for (int i = 0; i < items; ++i) {
                int x, y;
                bool valid;
                if (e.y == 0) {
                    const unsigned j = (unsigned)(i * 32 + lane);
                    valid = j < queued;
                    const unsigned n = valid ? queue->node[j] : 0u;
                    x = (int)(n & 0xffffu);
                    y = (int)(n >> 16);
                } else if (e.y == 1) {
                    x = e.z * 128 + i * 32 + lane;
                    y = e.w;
                    valid = x < nx;
                } else {
                    const int k = lane & 7;
                    y = e.w + 4 * i + (lane >> 3);
                    x = k < 4 ? k : xe + k - 4;
                    valid = y < ny - 1 && x < nx;
                }
                if (!__any_sync(kFull, valid)) continue;
                item_update<float, 9, false>(pb, st, src, dst, nullptr, x, y, valid, lane, sh, acc, w);
            }
            __syncwarp();
            if (lane == 0) queue->count = 0u;
            const size_t c = (size_t)(s & 1) * a.count + e.x;
            batch_flush(a.acc + c * kBatchStripes + u % kBatchStripes, a.maxit + c, acc, w, lane);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            next_unit = 0u;
            if (s != a.withhold || blockIdx.x != 0) bar_arrive(&a.bar->count);
            // the next step adds to the set of step s - 1
            ok_s = s + 1 == a.nsteps || (bar_wait(a.bar, &a.bar->count, (unsigned)(s + 1) * nb, a.wait_ns) &&
                                         bar_wait(a.bar, &a.bar->read[0], (unsigned)s, a.wait_ns));
        }
        __syncthreads();
        ok = ok_s;
    }
    batch_leave(a);
}

static size_t batch_smem() { return sizeof(unsigned) * 1024 * kBatchWarps; }

int resident_batch_blocks()
{
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(resident_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem()) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, resident_batch_kernel, kBatchThreads, batch_smem()) != cudaSuccess)
        return 0;
    return sms * per;
}

size_t resident_batch_bytes(int count) { return (size_t)2 * count * (kBatchStripes * sizeof(StepStripe) + sizeof(int)); }

cudaError_t launch_resident_batch(const Problem* probs, int count, const int4* units, int nunits, int blocks, int parity,
                                  int nsteps, DevStats* stats, void* sums, ResidentBar* bar, const ResidentLimits& lim,
                                  cudaStream_t s)
{
    if (lim.refuses(blocks)) return cudaErrorCooperativeLaunchTooLarge;
    ResidentBatchArgs a;
    a.nsteps = nsteps;
    a.stats = stats;
    a.slots = nullptr;
    a.bar = bar;
    a.wait_ns = lim.wait_ns;
    a.withhold = lim.withhold;
    a.probs = probs;
    a.count = count;
    a.units = units;
    a.nunits = nunits;
    a.parity = parity;
    a.acc = static_cast<StepStripe*>(sums);
    a.maxit = reinterpret_cast<int*>(a.acc + (size_t)2 * count * kBatchStripes);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kBatchThreads);
    cfg.dynamicSmemBytes = batch_smem();
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident_batch_kernel, a);
}

// ---------------------------------------------------------------- launch
// the queue of a block with a first pass
template <typename P, int Q>
static size_t resident_smem(bool first_pass)
{
    return first_pass ? sizeof(unsigned) * kResidentWaves<P> * kResidentThreads<P, Q> * (sizeof(P) == 4 ? 4 : 1) : 0;
}

template <typename P, int Q, bool EEBM>
static cudaError_t resident_go(ResidentArgs& a, int nblocks, int threads, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cfg.dynamicSmemBytes = resident_smem<P, Q>(a.tiles > 0);
    const cudaError_t e = cudaFuncSetAttribute(resident_kernel<P, Q, EEBM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)resident_smem<P, Q>(true));
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // every block resident: they wait on one another
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, resident_kernel<P, Q, EEBM>, a);
}

template <typename P, int Q, bool EEBM>
static int resident_capacity_t()
{
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(resident_kernel<P, Q, EEBM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)resident_smem<P, Q>(true)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, resident_kernel<P, Q, EEBM>, kResidentThreads<P, Q>,
                                                      resident_smem<P, Q>(true)) != cudaSuccess)
        return 0;
    return sms * per;
}

template <typename P, int Q>
static ResidentPlan resident_plan_t(int nx, int ny)
{
    ResidentPlan r;
    const int cap = std::min(resident_capacity_t<P, Q, false>(), resident_capacity_t<P, Q, true>());
    if (cap < 2 || nx >= 65536 || ny >= 65536) return r;
    const int most = kResidentThreads<P, Q> / 32, N = sizeof(P) == 4 ? 4 : 1;
    r.nseg = (nx + 31) / 32;
    const long long units = (long long)r.nseg * ny;
    const long long vec = ny > 2 ? (long long)((nx + 32 * N - 1) / (32 * N)) * (ny - 2) : 0;
    if (units <= (long long)LBM_RES_SCALAR * (cap - 1) || vec == 0) {
        // few nodes: all of them items, two warps per block, or as many as give every warp one
        int wpb = 2;
        while (wpb < most && wpb * (long long)(cap - 1) < units) wpb = std::min(2 * wpb, most);
        r.items = (int)units;
        r.blocks = (int)std::min<long long>(cap - 1, (units + wpb - 1) / wpb) + 1;
        r.threads = wpb * 32;
    } else {
        r.strips = (nx + 32 * N - 1) / (32 * N);
        // tall tiles share their halo rows; short ones spread a front band over the blocks and leave
        // fewer warps idle in the last wave.  us per step with 8 / 2 rows, the line (16 units per
        // warp) at 2232^2 in FP32 D2Q9, 1367^2 in FP64, 2733^2 in FP32 D2Q5: D2Q9 FP32 512^2
        // 13.3 / 11.9, 1400^2 36.6 / 33.5, 3000^2 123.7 / 125.3, 4096^2 214.3 / 215.5; D2Q9 FP64
        // 1200^2 72.1 / 67.8, 1600^2 111.0 / 108.3, 2048^2 166.6 / 170.8; D2Q5 FP32 1800^2 36.7 /
        // 29.9, 3200^2 84.7 / 77.8, 4096^2 122.6 / 122.3; D2Q5 FP64 1600^2 85.4 / 82.9, 2048^2
        // 130.3 / 132.7.  (In FP64 and D2Q5 2 rows still gain up to a tenth just beyond the line.)
        r.th = vec >= 16ll * most * cap ? 8 : 2;
        r.tiles = r.strips * ((ny - 2 + r.th - 1) / r.th);
        r.items = 2 * r.nseg + (ny - 2 + 32 / (2 * N) - 1) / (32 / (2 * N));
        r.blocks = cap;
        // as many warps as the waves need, so that all have as many units
        const long long waves = (vec + (long long)(cap - 1) * most - 1) / ((long long)(cap - 1) * most);
        const long long per = (vec + (cap - 1) * waves - 1) / ((cap - 1) * waves);
        r.threads = 32 * (int)std::min<long long>(most, (per + r.th - 1) / r.th * r.th);
    }
    r.slots = kResidentRing * (size_t)(r.blocks - 1);
    r.rot = (int)(0.618 * (r.blocks - 1));
    return r;
}

size_t resident_slot_bytes() { return sizeof(ResidentSlot); }

ResidentPlan resident_plan(int precision, int q, int nx, int ny)
{
    if (q == 9) return precision == 1 ? resident_plan_t<float, 9>(nx, ny) : resident_plan_t<double, 9>(nx, ny);
    if (q == 5) return precision == 1 ? resident_plan_t<float, 5>(nx, ny) : resident_plan_t<double, 5>(nx, ny);
    return ResidentPlan{};
}

cudaError_t launch_resident(int precision, const ResidentPlan& plan, const Problem& hp, int parity, int nsteps, double* rec,
                            DevStats* stats, void* slots, ResidentBar* bar, const ResidentLimits& lim, cudaStream_t s)
{
    if (lim.refuses(plan.blocks)) return cudaErrorCooperativeLaunchTooLarge;
    ResidentArgs a;
    a.pb = hp;
    a.parity = parity;
    a.nsteps = nsteps;
    a.rec = rec;
    a.stats = stats;
    a.slots = static_cast<ResidentSlot*>(slots);
    a.bar = bar;
    a.strips = plan.strips;
    a.th = plan.th;
    a.tiles = plan.tiles;
    a.nseg = plan.nseg;
    a.items = plan.items;
    a.rot = plan.rot;
    a.wait_ns = lim.wait_ns;
    a.withhold = lim.withhold;
    const bool eebm = hp.method == 1;
    if (hp.q == 9) {
        if (precision == 1)
            return eebm ? resident_go<float, 9, true>(a, plan.blocks, plan.threads, s)
                        : resident_go<float, 9, false>(a, plan.blocks, plan.threads, s);
        return eebm ? resident_go<double, 9, true>(a, plan.blocks, plan.threads, s)
                    : resident_go<double, 9, false>(a, plan.blocks, plan.threads, s);
    }
    if (precision == 1)
        return eebm ? resident_go<float, 5, true>(a, plan.blocks, plan.threads, s)
                    : resident_go<float, 5, false>(a, plan.blocks, plan.threads, s);
    return eebm ? resident_go<double, 5, true>(a, plan.blocks, plan.threads, s)
                : resident_go<double, 5, false>(a, plan.blocks, plan.threads, s);
}

}  // namespace lbm
