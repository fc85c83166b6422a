// Wall closures of the D2Q5 step kernels (Sec. 4.2): Dirichlet (Eqs. 15-16),
// bounce-back and the Neumann closure of Eq. (17).
#pragma once

#include "step_common.cuh"

namespace lbm {

// ---------------------------------------------------------------- closures
// A D2Q5 wall node (nx, ny >= 3): q_1 is unknown at x = 0, q_3 at x = nx - 1,
// q_2 at y = 0, q_4 at y = ny - 1.
struct Wall5 {
    unsigned unk;   // bit i: q_i not defined by streaming
    int wall;       // Dirichlet wall (first of W, E, S, N), -1 if none
    int sx, sy;     // Eq. (17): the node one step inwards (the diagonal one at a corner)
};

__device__ __forceinline__ Wall5 wall5_info(int x, int y, const Problem& pb)
{
    Wall5 w;
    const bool W = x == 0, E = x == pb.nx - 1, S = y == 0, N = y == pb.ny - 1;
    w.unk = (W ? 2u : 0u) | (S ? 4u : 0u) | (E ? 8u : 0u) | (N ? 16u : 0u);
    const int walls = (W ? 1 : 0) | (E ? 2 : 0) | (S ? 4 : 0) | (N ? 8 : 0);
    w.wall = -1;
    for (int k = 0; k < 4; ++k)
        if (((walls >> k) & 1) && pb.wall_kind[k] == 1) {
            w.wall = k;
            break;
        }
    w.sx = x + (W ? 1 : (E ? -1 : 0));
    w.sy = y + (S ? 1 : (N ? -1 : 0));
    return w;
}

// The streamed populations of the interior node one step inwards of the wall
// node (x, y), read from the source state (Eq. 17).
template <typename P>
__device__ __forceinline__ void pulled5_inward(const P* src, const Problem& pb, int x, int y, P (&q)[5])
{
    const Wall5 w = wall5_info(x, y, pb);
    x = w.sx;
    y = w.sy;
    const long long pl = pb.plane, pitch = pb.pitch;
    const P* r = src + (long long)(y + 1) * pitch + x;
    q[0] = r[0];
    q[1] = r[pl - 1];
    q[2] = r[2 * pl - pitch];
    q[3] = r[3 * pl + 1];
    q[4] = r[4 * pl + pitch];
}

// FP64 form.  q holds the pulled values (unknown entries are overwritten), u
// the node's own Omega, nq the streamed populations of the node one step
// inwards (read for Eq. 17 only).  Returns the boundary flux (filled q minus
// Omega that leaves the lattice); wall reports the node's Dirichlet wall or -1.
static __device__ __noinline__ double wall5_closure_d(double* q, const double* u, const double* nq, int x, int y,
                                                      const Problem& pb, int& wall)
{
    const Wall5 wi = wall5_info(x, y, pb);
    wall = wi.wall;
    double out = 0.0, in = 0.0;
#pragma unroll
    for (int j = 1; j < 5; ++j)
        if ((wi.unk >> d2_opp(j)) & 1) out += u[j];
    if (wi.wall >= 0 || pb.bb_mode == 2) {
        double m0t;
        if (wi.wall >= 0) {
            double th = 0.0;
#pragma unroll
            for (int i = 4; i >= 0; --i) th += u[i];
            m0t = dir_m0_target_d(th, wi.wall, pb);
        } else {
            m0t = 0.0;
#pragma unroll
            for (int i = 4; i >= 0; --i) m0t += nq[i];
        }
        // the unknown q share what the known ones leave, in proportion to w_i (equal)
        double known = 0.0;
        int nu = 0;
#pragma unroll
        for (int i = 4; i >= 0; --i) {
            if ((wi.unk >> i) & 1) ++nu;
            else known += q[i];
        }
        const double r = (m0t - known) / (double)nu;
#pragma unroll
        for (int i = 1; i < 5; ++i)
            if ((wi.unk >> i) & 1) {
                q[i] = r;
                in += r;
            }
    } else {
        // bounce-back: the opposite direction is always known on D2Q5 with nx, ny >= 3
#pragma unroll
        for (int i = 1; i < 5; ++i)
            if ((wi.unk >> i) & 1) {
                const int o = d2_opp(i);
                q[i] = pb.bb_mode == 0 ? q[o] : u[o];
                in += q[i];
            }
    }
    return in - out;
}

// FP32 form with float-float sums; sh: the state's shift.
static __device__ __noinline__ ff wall5_closure_f(float* q, const float* u, const float* nq, int x, int y,
                                                  const Problem& pb, int& wall, float sh)
{
    const Wall5 wi = wall5_info(x, y, pb);
    wall = wi.wall;
    ff out{0.f, 0.f}, in{0.f, 0.f};
#pragma unroll
    for (int j = 1; j < 5; ++j)
        if ((wi.unk >> d2_opp(j)) & 1) ff_add(out, u[j]);
    if (wi.wall >= 0 || pb.bb_mode == 2) {
        ff m0t{0.f, 0.f};   // target of M0(q), less the state's shift sh (q, u are Omega - w_i sh)
        if (wi.wall >= 0) {
            ff th{0.f, 0.f};
#pragma unroll
            for (int i = 4; i >= 0; --i) ff_add(th, u[i]);
            ff_add(th, sh);
            m0t = dir_m0_target_f(th, wi.wall, pb);
            ff_add(m0t, -sh);
        } else {
#pragma unroll
            for (int i = 4; i >= 0; --i) ff_add(m0t, nq[i]);
        }
        ff known{0.f, 0.f};
        int nu = 0;
#pragma unroll
        for (int i = 4; i >= 0; --i) {
            if ((wi.unk >> i) & 1) ++nu;
            else ff_add(known, q[i]);
        }
        const float r = ((m0t.hi - known.hi) + (m0t.lo - known.lo)) / (float)nu;
#pragma unroll
        for (int i = 1; i < 5; ++i)
            if ((wi.unk >> i) & 1) {
                q[i] = r;
                ff_add(in, r);
            }
    } else {
#pragma unroll
        for (int i = 1; i < 5; ++i)
            if ((wi.unk >> i) & 1) {
                const int o = d2_opp(i);
                q[i] = pb.bb_mode == 0 ? q[o] : u[o];
                ff_add(in, q[i]);
            }
    }
    ff f{in.hi, in.lo};
    ff_add(f, -out.hi);
    f.lo -= out.lo;
    return f;
}

}  // namespace lbm
