// Device helpers of the IREBM kernels: lattice constants, float-float sums,
// the regularized liquid fraction, the local Newton solve of Eq. (14),
// deterministic fixed-point reductions and the end-of-launch statistics.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lbm_internal.h"

namespace lbm {

constexpr unsigned kFull = 0xffffffffu;

// |x| >= kSat * delta  =>  tanh(x/delta) is +-1 in FP64 (1 - tanh(19.5) ~ 2e-17,
// below half an ulp of 1), so phi is exactly 0 or 1 there and phi' is 0.
constexpr double kSat = 19.5;

// ---------------------------------------------------------------- D2Q9 / D1Q3 / D2Q5
// D2Q9 velocities (Sec. 3.2): 0 rest; 1..4 = (+1,0),(0,+1),(-1,0),(0,-1);
// 5..8 = (+1,+1),(-1,+1),(-1,-1),(+1,-1).  Weights 4/9, 1/9, 1/36 (c_s^2 = 1/3).
__host__ __device__ constexpr int d2_ex(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__host__ __device__ constexpr int d2_ey(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
__host__ __device__ constexpr int d2_opp(int i) { return i == 0 ? 0 : (i <= 4 ? ((i + 1) & 3) + 1 : ((i - 3) & 3) + 5); }
__host__ __device__ constexpr double d2_w(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }
// D1Q3: 0 rest, 1 = +1, 2 = -1; weights 2/3, 1/6, 1/6.
__host__ __device__ constexpr int d1_ex(int i) { return i == 1 ? 1 : (i == 2 ? -1 : 0); }
__host__ __device__ constexpr double d1_w(int i) { return i == 0 ? 2.0 / 3.0 : 1.0 / 6.0; }
// D2Q5: 0 rest, 1..4 = (+1,0),(0,+1),(-1,0),(0,-1) as in D2Q9; weights 1/3, 1/6 (c_s^2 = 1/3).
__host__ __device__ constexpr double d5_w(int i) { return i == 0 ? 1.0 / 3.0 : 1.0 / 6.0; }
// weight i of the lattice with q velocities (3, 5 or 9)
__host__ __device__ constexpr double lat_w(int q, int i) { return q == 9 ? d2_w(i) : (q == 5 ? d5_w(i) : d1_w(i)); }

// FP32 weights.  The nearest floats to 4/9, 1/9, 1/36 sum to 1 + 2^-27, and
// those to 1/3, 1/6 (D2Q5) to 1 + 2^-25.  A relaxation toward w_i c in FP32
// multiplies the zeroth moment by that sum every step: on the 4096^2 melting
// workload (tau = 1) theta drifted by 7.5e-9 of itself per step, 2.5e-5 after
// 10,000 steps.  Here one weight of each set is one ulp below the nearest
// float (1/36, resp. 1/3), so that each set sums to exactly 1; the products
// w_i c still round, but without a bias.
__host__ __device__ constexpr float d2_wf(int i) { return i == 0 ? 0x1.c71c72p-2f : (i <= 4 ? 0x1.c71c72p-4f : 0x1.c71c70p-6f); }
__host__ __device__ constexpr float d5_wf(int i) { return i == 0 ? 0x1.555554p-2f : 0x1.555556p-3f; }
// the weights of the population precision P (float: the exact-sum sets above)
template <typename P> __host__ __device__ constexpr P lat_wp(int q, int i);
template <> __host__ __device__ constexpr float lat_wp<float>(int q, int i)
{
    return q == 9 ? d2_wf(i) : (q == 5 ? d5_wf(i) : (float)d1_w(i));
}
template <> __host__ __device__ constexpr double lat_wp<double>(int q, int i) { return lat_w(q, i); }

// ---------------------------------------------------------------- float-float
// Unevaluated sum hi + lo of two floats; two_sum is Knuth's error-free
// transformation (no fast-math: the compiler keeps the order of operations).
struct ff {
    float hi, lo;
};
__device__ __forceinline__ void ff_add(ff& a, float b)
{
    float s = __fadd_rn(a.hi, b);
    float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    a.hi = s;
    a.lo = __fadd_rn(a.lo, e);
}

// Approximate float of a double from its high word only (sign, exponent and
// 20 mantissa bits; relative error < 2^-20), using the integer pipe.  Values
// below 2^-126 in magnitude give 0; non-finite or huge values give NaN.
__device__ __forceinline__ float approx_float(double d)
{
    int hi = __double2hiint(d);
    int e = (hi >> 20) & 0x7ff;
    int bits = (hi & 0x80000000) | (((hi & 0x7fffffff) - (896 << 20)) << 3);
    float r = __int_as_float(bits);
    return e <= 896 ? 0.0f : (e >= 1151 ? __int_as_float(0x7fc00000) : r);
}

// The same truncated to all 23 mantissa bits (relative error < 2^-23).
__device__ __forceinline__ float trunc_float(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d);
    const int e = (int)((hi >> 20) & 0x7ff);
    const unsigned bits = (hi & 0x80000000u) |
                          (__funnelshift_l((unsigned)__double2loint(d), (hi & 0x7fffffffu) - (896u << 20), 3) & 0x7fffffffu);
    return e <= 896 ? 0.0f : (e >= 1151 ? __int_as_float(0x7fc00000) : __uint_as_float(bits));
}

// A float as a double with integer operations (a conversion instruction runs
// on the FP64 pipe, an SM's narrowest: 64 cycles of a quarter's issue slots).
// Exact; infinities, NaN and subnormal floats take the conversion.
__device__ __forceinline__ double widen(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu;
    if (e == 0xffu || (e == 0u && (b << 1) != 0u)) return (double)f;
    const unsigned hi = e == 0u ? 0u : (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20));
    return __hiloint2double((int)hi, e == 0u ? 0 : (int)(b << 29));
}

__device__ __forceinline__ double ff_to_double(const ff& a) { return widen(a.hi) + widen(a.lo); }

// ---------------------------------------------------------------- liquid fraction
// EEBM (Algorithm 2): temperature of an enthalpy, Theta(H) = H below 0, 0 on
// the melting plateau [0, 1/Ste], H - 1/Ste above it.
__device__ __forceinline__ double eebm_theta(double H, double inv_ste)
{
    // (sign and order from the bits: an FP64 comparison takes the FP64 pipe)
    const long long b = __double_as_longlong(H);
    if (b < 0) return H;
    return b > __double_as_longlong(inv_ste) ? H - inv_ste : 0.0;
}
__device__ __forceinline__ float eebm_theta(float H, float inv_ste)
{
    return H < 0.0f ? H : (H > inv_ste ? H - inv_ste : 0.0f);
}

// H - (1 - w0) theta - w0 sh, the rest population's EEBM equilibrium less w0 sh.
// The fused operations are spelled out, so that every kernel rounds alike.
__device__ __forceinline__ float eebm_rest(float H, float theta, float w0, float sh)
{
    return __fmaf_rn(-w0, sh, __fmaf_rn(w0 - 1.0f, theta, H));
}
__device__ __forceinline__ double eebm_rest(double H, double theta, double w0, double sh)
{
    return fma(-w0, sh, fma(w0 - 1.0, theta, H));
}

// 2^(j/256), rounded to nearest
static __device__ const double kExp2[256] = {
    0x1p+0, 0x1.00b1afa5abcbfp+0, 0x1.0163da9fb3335p+0, 0x1.02168143b0281p+0,
    0x1.02c9a3e778061p+0, 0x1.037d42e11bbccp+0, 0x1.04315e86e7f85p+0, 0x1.04e5f72f654b1p+0,
    0x1.059b0d3158574p+0, 0x1.0650a0e3c1f89p+0, 0x1.0706b29ddf6dep+0, 0x1.07bd42b72a836p+0,
    0x1.0874518759bc8p+0, 0x1.092bdf66607e0p+0, 0x1.09e3ecac6f383p+0, 0x1.0a9c79b1f3919p+0,
    0x1.0b5586cf9890fp+0, 0x1.0c0f145e46c85p+0, 0x1.0cc922b7247f7p+0, 0x1.0d83b23395decp+0,
    0x1.0e3ec32d3d1a2p+0, 0x1.0efa55fdfa9c5p+0, 0x1.0fb66affed31bp+0, 0x1.1073028d7233ep+0,
    0x1.11301d0125b51p+0, 0x1.11edbab5e2ab6p+0, 0x1.12abdc06c31ccp+0, 0x1.136a814f204abp+0,
    0x1.1429aaea92de0p+0, 0x1.14e95934f312ep+0, 0x1.15a98c8a58e51p+0, 0x1.166a45471c3c2p+0,
    0x1.172b83c7d517bp+0, 0x1.17ed48695bbc0p+0, 0x1.18af9388c8deap+0, 0x1.1972658375d2fp+0,
    0x1.1a35beb6fcb75p+0, 0x1.1af99f8138a1cp+0, 0x1.1bbe084045cd4p+0, 0x1.1c82f95281c6bp+0,
    0x1.1d4873168b9aap+0, 0x1.1e0e75eb44027p+0, 0x1.1ed5022fcd91dp+0, 0x1.1f9c18438ce4dp+0,
    0x1.2063b88628cd6p+0, 0x1.212be3578a819p+0, 0x1.21f49917ddc96p+0, 0x1.22bdda27912d1p+0,
    0x1.2387a6e756238p+0, 0x1.2451ffb82140ap+0, 0x1.251ce4fb2a63fp+0, 0x1.25e85711ece75p+0,
    0x1.26b4565e27cddp+0, 0x1.2780e341ddf29p+0, 0x1.284dfe1f56381p+0, 0x1.291ba7591bb70p+0,
    0x1.29e9df51fdee1p+0, 0x1.2ab8a66d10f13p+0, 0x1.2b87fd0dad990p+0, 0x1.2c57e39771b2fp+0,
    0x1.2d285a6e4030bp+0, 0x1.2df961f641589p+0, 0x1.2ecafa93e2f56p+0, 0x1.2f9d24abd886bp+0,
    0x1.306fe0a31b715p+0, 0x1.31432edeeb2fdp+0, 0x1.32170fc4cd831p+0, 0x1.32eb83ba8ea32p+0,
    0x1.33c08b26416ffp+0, 0x1.3496266e3fa2dp+0, 0x1.356c55f929ff1p+0, 0x1.36431a2de883bp+0,
    0x1.371a7373aa9cbp+0, 0x1.37f26231e754ap+0, 0x1.38cae6d05d866p+0, 0x1.39a401b7140efp+0,
    0x1.3a7db34e59ff7p+0, 0x1.3b57fbfec6cf4p+0, 0x1.3c32dc313a8e5p+0, 0x1.3d0e544ede173p+0,
    0x1.3dea64c123422p+0, 0x1.3ec70df1c5175p+0, 0x1.3fa4504ac801cp+0, 0x1.40822c367a024p+0,
    0x1.4160a21f72e2ap+0, 0x1.423fb2709468ap+0, 0x1.431f5d950a897p+0, 0x1.43ffa3f84b9d4p+0,
    0x1.44e086061892dp+0, 0x1.45c2042a7d232p+0, 0x1.46a41ed1d0057p+0, 0x1.4786d668b3237p+0,
    0x1.486a2b5c13cd0p+0, 0x1.494e1e192aed2p+0, 0x1.4a32af0d7d3dep+0, 0x1.4b17dea6db7d7p+0,
    0x1.4bfdad5362a27p+0, 0x1.4ce41b817c114p+0, 0x1.4dcb299fddd0dp+0, 0x1.4eb2d81d8abffp+0,
    0x1.4f9b2769d2ca7p+0, 0x1.508417f4531eep+0, 0x1.516daa2cf6642p+0, 0x1.5257de83f4eefp+0,
    0x1.5342b569d4f82p+0, 0x1.542e2f4f6ad27p+0, 0x1.551a4ca5d920fp+0, 0x1.56070dde910d2p+0,
    0x1.56f4736b527dap+0, 0x1.57e27dbe2c4cfp+0, 0x1.58d12d497c7fdp+0, 0x1.59c0827ff07ccp+0,
    0x1.5ab07dd485429p+0, 0x1.5ba11fba87a03p+0, 0x1.5c9268a5946b7p+0, 0x1.5d84590998b93p+0,
    0x1.5e76f15ad2148p+0, 0x1.5f6a320dceb71p+0, 0x1.605e1b976dc09p+0, 0x1.6152ae6cdf6f4p+0,
    0x1.6247eb03a5585p+0, 0x1.633dd1d1929fdp+0, 0x1.6434634ccc320p+0, 0x1.652b9febc8fb7p+0,
    0x1.6623882552225p+0, 0x1.671c1c70833f6p+0, 0x1.68155d44ca973p+0, 0x1.690f4b19e9538p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6b052fa75173ep+0, 0x1.6c012750bdabfp+0, 0x1.6cfdcddd47645p+0,
    0x1.6dfb23c651a2fp+0, 0x1.6ef9298593ae5p+0, 0x1.6ff7df9519484p+0, 0x1.70f7466f42e87p+0,
    0x1.71f75e8ec5f74p+0, 0x1.72f8286ead08ap+0, 0x1.73f9a48a58174p+0, 0x1.74fbd35d7cbfdp+0,
    0x1.75feb564267c9p+0, 0x1.77024b1ab6e09p+0, 0x1.780694fde5d3fp+0, 0x1.790b938ac1cf6p+0,
    0x1.7a11473eb0187p+0, 0x1.7b17b0976cfdbp+0, 0x1.7c1ed0130c132p+0, 0x1.7d26a62ff86f0p+0,
    0x1.7e2f336cf4e62p+0, 0x1.7f3878491c491p+0, 0x1.80427543e1a12p+0, 0x1.814d2add106d9p+0,
    0x1.82589994cce13p+0, 0x1.8364c1eb941f7p+0, 0x1.8471a4623c7adp+0, 0x1.857f4179f5b21p+0,
    0x1.868d99b4492edp+0, 0x1.879cad931a436p+0, 0x1.88ac7d98a6699p+0, 0x1.89bd0a478580fp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8be05bad61778p+0, 0x1.8cf3216b5448cp+0, 0x1.8e06a5e0866d9p+0,
    0x1.8f1ae99157736p+0, 0x1.902fed0282c8ap+0, 0x1.9145b0b91ffc6p+0, 0x1.925c353aa2fe2p+0,
    0x1.93737b0cdc5e5p+0, 0x1.948b82b5f98e5p+0, 0x1.95a44cbc8520fp+0, 0x1.96bdd9a7670b3p+0,
    0x1.97d829fde4e50p+0, 0x1.98f33e47a22a2p+0, 0x1.9a0f170ca07bap+0, 0x1.9b2bb4d53fe0dp+0,
    0x1.9c49182a3f090p+0, 0x1.9d674194bb8d5p+0, 0x1.9e86319e32323p+0, 0x1.9fa5e8d07f29ep+0,
    0x1.a0c667b5de565p+0, 0x1.a1e7aed8eb8bbp+0, 0x1.a309bec4a2d33p+0, 0x1.a42c980460ad8p+0,
    0x1.a5503b23e255dp+0, 0x1.a674a8af46052p+0, 0x1.a799e1330b358p+0, 0x1.a8bfe53c12e59p+0,
    0x1.a9e6b5579fdbfp+0, 0x1.ab0e521356ebap+0, 0x1.ac36bbfd3f37ap+0, 0x1.ad5ff3a3c2774p+0,
    0x1.ae89f995ad3adp+0, 0x1.afb4ce622f2ffp+0, 0x1.b0e07298db666p+0, 0x1.b20ce6c9a8952p+0,
    0x1.b33a2b84f15fbp+0, 0x1.b468415b749b1p+0, 0x1.b59728de5593ap+0, 0x1.b6c6e29f1c52ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.b928cf22749e4p+0, 0x1.ba5b030a1064ap+0, 0x1.bb8e0b79a6f1fp+0,
    0x1.bcc1e904bc1d2p+0, 0x1.bdf69c3f3a207p+0, 0x1.bf2c25bd71e09p+0, 0x1.c06286141b33dp+0,
    0x1.c199bdd85529cp+0, 0x1.c2d1cd9fa652cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c544778fafb22p+0,
    0x1.c67f12e57d14bp+0, 0x1.c7ba88988c933p+0, 0x1.c8f6d9406e7b5p+0, 0x1.ca3405751c4dbp+0,
    0x1.cb720dcef9069p+0, 0x1.ccb0f2e6d1675p+0, 0x1.cdf0b555dc3fap+0, 0x1.cf3155b5bab74p+0,
    0x1.d072d4a07897cp+0, 0x1.d1b532b08c968p+0, 0x1.d2f87080d89f2p+0, 0x1.d43c8eacaa1d6p+0,
    0x1.d5818dcfba487p+0, 0x1.d6c76e862e6d3p+0, 0x1.d80e316c98398p+0, 0x1.d955d71ff6075p+0,
    0x1.da9e603db3285p+0, 0x1.dbe7cd63a8315p+0, 0x1.dd321f301b460p+0, 0x1.de7d5641c0658p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e11676b197d17p+0, 0x1.e264614f5a129p+0, 0x1.e3b333b16ee12p+0,
    0x1.e502ee78b3ff6p+0, 0x1.e653924676d76p+0, 0x1.e7a51fbc74c83p+0, 0x1.e8f7977cdb740p+0,
    0x1.ea4afa2a490dap+0, 0x1.eb9f4867cca6ep+0, 0x1.ecf482d8e67f1p+0, 0x1.ee4aaa2188510p+0,
    0x1.efa1bee615a27p+0, 0x1.f0f9c1cb6412ap+0, 0x1.f252b376bba97p+0, 0x1.f3ac948dd7274p+0,
    0x1.f50765b6e4540p+0, 0x1.f6632798844f8p+0, 0x1.f7bfdad9cbe14p+0, 0x1.f91d802243c89p+0,
    0x1.fa7c1819e90d8p+0, 0x1.fbdba3692d514p+0, 0x1.fd3c22b8f71f1p+0, 0x1.fe9d96b2a23d9p+0,
};

// exp(-w) for w in [0, 39) by table-driven reduction (P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point arithmetic",
// ACM TOMS 15, 1989): N the integer next to 256 w / ln 2 (found in FP32: any
// integer that leaves |r| <= 0.0014 will do), r = N ln2/256 - w with ln2/256 in two
// parts, e^r from its Taylor polynomial (the remainder r^5/120 is below 5e-17),
// times 2^(-N/256), from the table and added to the exponent.  Seven FP64
// instructions, no branch.
__device__ __forceinline__ double exp_neg(double w)
{
    const float t = fmaf(trunc_float(w), 369.32993f, 12582912.0f);   // the integer N in the low bits
    const int n = 0x4b400000 - __float_as_int(t);                      // -N
    const double nd = widen(t - 12582912.0f);
    double r = fma(nd, 0x1.62e42fefa0000p-9, -w);
    r = fma(nd, 0x1.cf79abc9e3b3ap-48, r);
    double p = fma(r, 1.0 / 24.0, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(r * r, p, r);
    const double T = __ldg(&kExp2[n & 255]);
    const double e = fma(T, p, T);
    return __hiloint2double(__double2hiint(e) + ((n >> 8) << 20), __double2loint(e));
}

// 1/(1 + E) for E in [0, 1]: an FP32 reciprocal r0 (relative error e < 2^-21) and
// one third-order step, r0 (1 + e + e^2), remainder e^3 < 2^-63.  e = (1 - r0) - E r0,
// whose difference is exact, so 1 + E is not rounded: half an ulp of the result
// (with e from the rounded sum an ulp and a half, which theta' inherits over Ste).
__device__ __forceinline__ double logistic(double E)
{
    const double r0 = widen(__frcp_rn(1.0f + trunc_float(E)));
    double e = fma(-E, r0, 1.0 - r0);
    e = fma(e, e, e);
    return fma(r0, e, r0);
}

// The liquid fraction phi(x) = (1 + tanh(x/delta))/2 (Sec. 4.1) as the logistic
// function it is, 1/(1 + exp(-2x/delta)): with E = exp(-2|x|/delta) and
// r = 1/(1 + E), phi = r for x >= 0 and E r below, and phi' = 2 E r^2 / delta.
// One exponential and one reciprocal, without a branch between ranges (a warp
// whose lanes straddle the ranges of a library tanh runs both): 13 FP64
// instructions.  |x| >= 19.5 delta: E = 0, where tanh rounds to +-1.
struct Phi {
    double E, r;   // NaN for a NaN x
    bool neg;
    __device__ __forceinline__ double value() const { return neg ? E * r : r; }
    __device__ __forceinline__ double s() const { return E * r * r; }   // phi (1 - phi) = phi' delta / 2
};

// of z = 2 x / delta
__device__ __forceinline__ Phi phi_z(double z)
{
    const int h = __double2hiint(z) & 0x7fffffff;
    Phi p;
    p.neg = __double2hiint(z) < 0;
    if (h >= 0x40438000) {   // |z| >= 39, infinite or NaN
        const bool nan = h > 0x7ff00000 || (h == 0x7ff00000 && __double2loint(z) != 0);
        p.E = nan ? z : 0.0;
        p.r = nan ? z : 1.0;
    } else {
        p.E = exp_neg(__hiloint2double(h, __double2loint(z)));
        p.r = logistic(p.E);
    }
    return p;
}

__device__ __forceinline__ Phi phi_parts(double x, double two_inv_delta) { return phi_z(x * two_inv_delta); }

__device__ __forceinline__ double phi_of(double x, double inv_delta) { return phi_parts(x, inv_delta + inv_delta).value(); }

// Local Newton solve of Eq. (14): the root of
//   F(x) = (x - m0) + (phi(x) - phi(theta))/Ste,   F' = 1 + phi'(x)/Ste >= 1,
// from x = theta (Algorithm 3).  Safeguard: the root lies in
// [m0 + (phi(theta) - 1)/Ste, m0 + phi(theta)/Ste]; a Newton iterate that
// leaves the current bracket, or does not at least halve the update before
// last, is replaced by the bracket midpoint (this also breaks 2-cycles).
// Converged when an update moves x by at most tol*max(1,|x|) (tested before
// the safeguard), when F = 0, or when the bracket is that narrow.
struct NewtonOut {
    double root;
    double phi_root;
    int iters;
    bool ok;
};

// Not inlined: the mixed-precision solve below falls back to it, which is rare.
static __device__ __noinline__ NewtonOut newton_solve(double m0, double theta, double phi_theta, double inv_ste,
                                                      double inv_delta, double tol, int maxit)
{
    // (widened by their rounding: a root at an end, as that of a node that leaves the band at
    // once, must not fall outside: bisecting towards it takes more steps than maxit)
    const double slack = 0x1p-51 * (fabs(m0) + inv_ste);
    double lo = m0 + (phi_theta - 1.0) * inv_ste - slack, hi = m0 + phi_theta * inv_ste + slack;
    double x = theta;
    double step_old = hi - lo, step = step_old;
    NewtonOut r;
    for (int k = 0; k < maxit; ++k) {
        const Phi p = phi_parts(x, 2.0 * inv_delta);
        const double ph = p.value();
        double F = (x - m0) + (ph - phi_theta) * inv_ste;
        if (F == 0.0) {
            r.root = x; r.phi_root = ph; r.iters = k; r.ok = true;
            return r;
        }
        if (F < 0.0) lo = fmax(lo, x);
        else hi = fmin(hi, x);
        double dph = 2.0 * p.s() * inv_delta;
        double xn = x - F / (1.0 + dph * inv_ste);
        double sc = tol * fmax(1.0, fabs(x));
        if (fabs(xn - x) <= sc) {
            // |xn - x| <= ~1e-14: phi(xn) = ph + phi'(x)(xn - x) to far below one ulp
            r.root = xn; r.phi_root = ph + dph * (xn - x); r.iters = k + 1; r.ok = true;
            return r;
        }
        if (!(xn >= lo && xn <= hi) || fabs(xn - x) > 0.5 * step_old) {
            step_old = step;
            step = 0.5 * (hi - lo);
            xn = lo + step;
            if (step <= tol * fmax(1.0, fabs(xn))) {
                r.root = xn; r.phi_root = phi_of(xn, inv_delta); r.iters = k + 1; r.ok = true;
                return r;
            }
        } else {
            step_old = step;
            step = fabs(xn - x);
        }
        x = xn;
    }
    r.root = x; r.phi_root = phi_of(x, inv_delta); r.iters = maxit; r.ok = false;
    return r;
}

// Mixed-precision form of the same solve (same root, same stopping rule), for
// m0 = mm + sh and theta = tt + sh (SHIFTED: sh is the state's shift; else 0, the
// FP64 form), as theta' = m0 + (phi(theta) - phi(root))/Ste.
//  1. FP32 Newton for the step u = x - theta.  The equation is
//     u - (m0 - theta) + (phi(theta + u) - phi(theta))/Ste = 0 with the
//     difference of phi from expm1 (no cancellation: with b = 2u/delta and
//     m = expm1(-b), phi(theta + u) - phi(theta) = -E m r r1, r1 = 1/(1 + E(1 + m)),
//     for theta >= 0; theta < 0 is its mirror image), so u is good to a few
//     FP32 ulps of itself.  It stops when an update is below 1e-3 delta: the
//     next error is then of the order of 1e-6 delta.
//  2. FP64 step from x0 = theta + u: phi(x0) gives F, F' and the Newton update
//     dn = -F/F' (1/F' from an FP32 reciprocal and one FP64 Newton step:
//     relative error ~1e-14).  The second and third derivatives enter as
//     corrections of relative size 1e-4 at most and are formed in FP32: Halley's
//     update d = dn / (1 + dn F_2/(2F')).  Halley's error e is about
//     |F_2^2/(4F'^2) - F_3/(6F')| |dn|^3, and theta' inherits it as (F' - 1) e;
//     when F' e is below 0.1 tol max(1,|x|) and |d| <= 3e-5 delta, x0 + d is
//     accepted and phi(x0 + d) comes from the cubic Taylor expansion (the quartic
//     remainder is below (d/delta)^4 / 12 < 1e-19).  Otherwise the FP64 iteration
//     goes on.  Iterations of both precisions count against maxit.
//  3. Anything unexpected (no FP32 convergence, an FP64 update larger than
//     1e-3 delta) falls back to newton_solve from theta.
// A solve is bound by the FP64 pipe, one warp instruction per 64 cycles of an SM
// quarter, so only differences of phi are formed (phi = r, or 1 - r for x < 0,
// and the sides agree as a rule), the arguments of phi and theta' come in one
// fused operation each, and the energy theta' + phi(theta')/Ste is
// m0 + phi(theta)/Ste: 43 FP64 instructions (44 with a shift) per node with the
// sums before and the collision after (236 with the library's tanh, conversion
// instructions and FP64 corrections; counted per warp on the front band of a
// 1021 x 777 lattice).  Error of theta' against 113-bit arithmetic, theta within
// 19.5 delta, m0 - theta from 1e-12 to 1/Ste, Ste 0.01 to 1, in units of
// 2^-53/Ste: at most 2.0, standard deviation at most 0.37 (with the library's tanh
// and FP64 corrections from an FP32-accurate start 2.2 and 0.41).
struct NewtonNode {
    double tns;      // theta' - sh
    double ens;      // theta' + phi(theta')/Ste - sh
    int iters;
    bool ok;
};

__device__ __forceinline__ double flip_sign(double v, bool neg)
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}

template <bool SHIFTED>
__device__ __forceinline__ NewtonNode newton_mixed(double mm, double tt, double sh, const Problem& pb)
{
    const double inv_ste = pb.inv_ste, tid = pb.two_inv_delta;
    const int maxit = pb.maxit;
    // theta first: near the band the shift cancels exactly (2 sh/delta would round by its own
    // size, up to 100 times that of z, and phi(theta) with it)
    const double z = (SHIFTED ? tt + sh : tt) * tid;
    const Phi pt = phi_z(z);
    const double dmd = mm - tt;   // m0 - theta
    const float isf = pb.inv_ste_f, idf2 = 2.0f * pb.inv_delta_f;
    const float zf = fabsf(trunc_float(z));
    const float dm0 = trunc_float(dmd);
    const float dm = pt.neg ? -dm0 : dm0;            // mirrored to theta >= 0
    const float E = trunc_float(pt.E), r0 = trunc_float(pt.r);
    const float slack = 0x1p-21f * (fabsf(dm) + isf);   // rounding of the bracket, as in newton_solve
    float lo = dm + (r0 - 1.0f) * isf - slack, hi = dm + r0 * isf + slack;
    const float small = 1e-3f * pb.delta_f, di = idf2 * isf;
    // the first iterate from x = theta (F = -dm there) needs no exponential
    float u = __fdividef(dm, fmaf(E * r0 * r0, di, 1.0f));
    if (dm > 0.0f) lo = fmaxf(lo, 0.0f);
    else hi = fminf(hi, 0.0f);
    if (!(u >= lo && u <= hi)) u = 0.5f * (lo + hi);
    float step_prev = fabsf(u);
    // an update below the FP32 resolution of x is no iteration (a node in equilibrium: m0 = theta)
    int k = idf2 * step_prev <= 0x1p-23f * zf ? 0 : 1;
    for (; k < 16 && step_prev > small; ++k) {
        const float b = idf2 * u, ab = fabsf(b);
        float D, dph;   // phi(theta + u) - phi(theta), phi'(theta + u) delta / 2
        if (ab <= 20.0f) {
            // expm1(-b): its Taylor series to b^7, or the difference where that loses little
            float m = fmaf(-b, 1.0f / 5040.0f, 1.0f / 720.0f);
            m = fmaf(m, -b, 1.0f / 120.0f);
            m = fmaf(m, -b, 1.0f / 24.0f);
            m = fmaf(m, -b, 1.0f / 6.0f);
            m = fmaf(m, -b, 0.5f);
            m = fmaf(m * b, b, -b);
            if (ab > 0.5f) m = expf(-b) - 1.0f;
            const float E1 = fmaf(E, m, E);
            const float r1 = __fdividef(1.0f, 1.0f + E1);
            D = -E * m * r0 * r1;
            dph = E1 * r1 * r1;
        } else {
            const float r1 = 1.0f / (1.0f + expf(-(zf + b)));
            D = r1 - r0;
            dph = r1 * (1.0f - r1);
        }
        const float F = (u - dm) + D * isf;
        if (F == 0.0f) break;
        if (F < 0.0f) lo = fmaxf(lo, u);
        else hi = fminf(hi, u);
        float un = u - __fdividef(F, fmaf(dph, di, 1.0f));
        if (!(un >= lo && un <= hi)) {
            un = 0.5f * (lo + hi);
        } else {
            const float st = fabsf(un - u);
            if (k >= 2 && st >= 0.5f * step_prev) {
                u = un;
                ++k;
                break;
            }
            step_prev = st;
        }
        u = un;
    }
    NewtonNode out;
    const double phi_theta = pt.value();
    out.ens = fma(phi_theta, inv_ste, mm);
    if (isfinite(u)) {
        double ud = widen(pt.neg ? -u : u);   // x - theta
        const double bt = flip_sign(pt.r, pt.neg);
        const float df = pb.delta_f, tolf = trunc_float(pb.tol);
        for (int j = 0; j < 3; ++j) {
            const double z0 = fma(ud, tid, z);
            const Phi p = phi_z(z0);
            // phi(x) - phi(theta); across 0 the 1 goes to r(x) first, where it is exact
            double a = flip_sign(p.r, p.neg);
            if (p.neg != pt.neg) a += p.neg ? 1.0 : -1.0;
            const double dphi = a - bt;
            const double s = p.s();
            const double F = fma(dphi, inv_ste, ud - dmd);
            const double Fp = fma(s, pb.two_inv_delta_ste, 1.0);
            const double g0 = widen(__frcp_rn(trunc_float(Fp)));
            const double rinv = fma(g0, fma(-Fp, g0, 1.0), g0);
            const double dn = -F * rinv;   // Newton update
            const float dnf = trunc_float(dn), adn = fabsf(dnf);
            if (!(adn <= 1e-3f * df)) break;   // FP32 start not close enough (or NaN): full FP64 solve
            // derivatives of phi in units of delta: phi' = 2s/delta, phi'' = -2 t phi'/delta,
            // phi_3 = 2 phi' (3 t^2 - 1)/delta^2, t = tanh(x/delta) = +-(1 - E) r
            const float sf = trunc_float(s), rf = trunc_float(p.r), Ef = trunc_float(p.E);
            const float t = p.neg ? -(1.0f - Ef) * rf : (1.0f - Ef) * rf;
            const float p1 = idf2 * sf;
            const float p2 = -idf2 * t * p1;
            const float p3 = 0.5f * idf2 * idf2 * (3.0f * t * t - 1.0f) * p1;
            const float rif = trunc_float(rinv);
            // Halley update d = dn / (1 + dn F_2/(2F')), 1/(1 + eps) to second order (accepted only
            // for |eps| <= 1e-4: the neglected eps^3 |dn| is below 1e-12 |dn|)
            const float eps = 0.5f * dnf * p2 * isf * rif;
            const double d = fma(dn, widen(eps * eps - eps), dn);
            const float daf = trunc_float(d), ad = fabsf(daf);
            const float sc = tolf * fmaxf(1.0f, fabsf(trunc_float(z0)) * 0.5f * df);
            // theta' = m0 + (phi(theta) - phi(x))/Ste carries a root error e as (F' - 1) e;
            // after the Halley step F' e ~ |F_2^2/(4F') - F_3/6| |dn|^3
            const float g = (0.25f * p2 * p2 * isf * rif + fabsf(p3) * (1.0f / 6.0f)) * isf;
            if (ad <= sc || (ad <= 3e-5f * df && fabsf(eps) <= 1e-4f && g * adn * adn * adn <= 0.1f * sc)) {
                const double c1 = fma(s, tid, widen(daf * (0.5f * p2 + daf * p3 * (1.0f / 6.0f))));
                out.tns = fma(-fma(d, c1, dphi), inv_ste, mm);
                out.iters = k + j + 1;
                out.ok = out.iters <= maxit && isfinite(out.tns);
                return out;
            }
            ud += d;
        }
    }
    // theta' from the m0 that the root was found for: inside the band it hardly depends on it
    const double m0 = SHIFTED ? mm + sh : mm;
    const NewtonOut r = newton_solve(m0, SHIFTED ? tt + sh : tt, phi_theta, inv_ste, pb.inv_delta, pb.tol, maxit);
    out.tns = fma(phi_theta - r.phi_root, inv_ste, m0);
    if (SHIFTED) out.tns -= sh;
    out.iters = r.iters + k;
    out.ok = r.ok && out.iters <= maxit && isfinite(r.root);
    return out;
}

// ---------------------------------------------------------------- exact sums
// sum of Q doubles, to within 2^-6 ulp of the largest per term, rounded once
// (error against 113-bit sums of populations, units of 2^-53 of the largest: at most
// 3.8, 0.95 rms for nine; added one after the other 8.0 and 1.4):
// the mantissas are aligned to the largest exponent with six guard bits (59
// bits; nine of them stay below 2^63) and added as integers, 15 integer
// instructions per term against 64 cycles of FP64 pipe per addition.  Terms
// down to 2^-6 of the largest lose no bit.  Sums of tiny (2^-953), huge (2^1007)
// or non-finite terms go through FP64 additions.
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned s)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));   // 0 for s >= 64
    return r;
}

template <int Q>
__device__ __forceinline__ double sum_q(const double (&q)[Q])
{
    unsigned emax = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) emax = max(emax, (unsigned)__double2hiint(q[i]) & 0x7ff00000u);
    emax >>= 20;
    if (emax < 70u || emax >= 2030u) {
        double s = 0.0;
#pragma unroll
        for (int i = Q - 1; i >= 0; --i) s += q[i];
        return s;
    }
    long long S = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned h = (unsigned)__double2hiint(q[i]), l = (unsigned)__double2loint(q[i]);
        const unsigned sh = emax - ((h >> 20) & 0x7ffu);
        // the mantissa, shifted left by six (a zero's implicit bit is shifted out: sh >= 70)
        const unsigned mh = __funnelshift_l(l, (h & 0xfffffu) | 0x100000u, 6);
        const unsigned long long m = shr64(((unsigned long long)mh << 32) | (l << 6), sh);
        const long long sg = (long long)(int)h >> 63;
        S += ((long long)m ^ sg) - sg;
    }
    const bool neg = S < 0;
    const unsigned long long a = neg ? 0ull - (unsigned long long)S : (unsigned long long)S;
    if (a == 0ull) return 0.0;
    const int lz = __clzll((long long)a);
    const unsigned long long nrm = a << lz;
    // round to nearest even at bit 11; a carry runs into the exponent
    const unsigned low = (unsigned)nrm & 0x7ffu, lsb = ((unsigned)nrm >> 11) & 1u;
    unsigned long long b = (nrm >> 11) + (low + lsb > 0x400u ? 1ull : 0ull);
    b += (unsigned long long)((int)emax - lz + 5 - 1) << 52;   // the implicit bit adds 1
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

// v 2^k for a finite v that stays normal (else by multiplication)
__device__ __forceinline__ double scale2(double v, int k)
{
    const int h = __double2hiint(v), e = (h >> 20) & 0x7ff;
    if (e < 8 || e > 2040) return k > 0 ? v * (double)(1 << k) : v / (double)(1 << -k);
    return __hiloint2double(h + (k << 20), __double2loint(v));
}

// ---------------------------------------------------------------- lane shifts
// A warp-wide row of 32*N values held N per lane, shifted by one element.
// value at x-1 (pull along e_x = +1); h = element left of the segment
template <typename P, int N>
__device__ __forceinline__ void from_left(const P (&v)[N], P h, int lane, P (&s)[N])
{
    P up = __shfl_up_sync(kFull, v[N - 1], 1);
    s[0] = lane == 0 ? h : up;
#pragma unroll
    for (int k = 1; k < N; ++k) s[k] = v[k - 1];
}
// value at x+1 (pull along e_x = -1); h = element right of the segment
template <typename P, int N>
__device__ __forceinline__ void from_right(const P (&v)[N], P h, int lane, P (&s)[N])
{
    P dn = __shfl_down_sync(kFull, v[0], 1);
    s[N - 1] = lane == 31 ? h : dn;
#pragma unroll
    for (int k = 0; k < N - 1; ++k) s[k] = v[k + 1];
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ int warp_sum_i(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ int warp_max_i(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// 128-bit fixed-point value (scaled by 2^60) as a register pair; adding two of
// them is exact, so sums in this form do not depend on the order of terms.
struct Fx {
    long long hi;
    unsigned long long lo;
};

// With integer operations only (an FP64 conversion costs 64 cycles of an SM
// quarter): v = m 2^(e - 1075), scaled by 2^60.  Bits below 2^-60 are dropped;
// values of 2^67 and more, infinities and NaN have no fixed-point value and give
// 0: the caller keeps the largest fx_mag of its terms beside the sum, and one that
// reaches kFxMag makes the published sum NaN.
constexpr unsigned kFxMag = (1023u + 67u) << 20;
__device__ __forceinline__ unsigned fx_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ double nan_d() { return __longlong_as_double(0x7ff8000000000000ll); }

__device__ __forceinline__ Fx to_fixed(double v)
{
    Fx f{0, 0ull};
    const unsigned hw = (unsigned)__double2hiint(v);
    const int e = (int)((hw >> 20) & 0x7ff);
    const unsigned long long m = ((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(v);
    const int sh = e - 1015;   // m * 2^(e - 1075 + 60)
    unsigned long long lo = 0, hi = 0;
    if (sh >= 0) {
        if (sh >= 75) return f;
        lo = sh < 64 ? m << sh : 0ull;
        hi = sh == 0 ? 0ull : (sh < 64 ? m >> (64 - sh) : m << (sh - 64));
    } else if (sh > -64 && e != 0) {
        lo = m >> (-sh);
    }
    if (hw >> 31) {   // two's complement of the 128-bit value
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    f.lo = lo;
    f.hi = (long long)hi;
    return f;
}

__device__ __forceinline__ void fx_add(Fx& a, const Fx& b)
{
    const unsigned long long lo = a.lo + b.lo;
    a.hi += b.hi + (lo < a.lo ? 1 : 0);
    a.lo = lo;
}

__device__ __forceinline__ Fx fx_tree(Fx v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Fx w;
        w.hi = __shfl_xor_sync(kFull, v.hi, o);
        w.lo = __shfl_xor_sync(kFull, v.lo, o);
        fx_add(v, w);
    }
    return v;
}

__device__ __forceinline__ void acc_add_fx(Acc128* a, const Fx& v)
{
    if (v.hi == 0 && v.lo == 0) return;
    const unsigned long long old = atomicAdd(&a->lo, v.lo);
    const long long carry = (old + v.lo < old) ? 1 : 0;
    atomicAdd(reinterpret_cast<unsigned long long*>(&a->hi), (unsigned long long)(v.hi + carry));
}

// Exact fixed-point value of a float with integer operations only (no FP64
// instruction): v = m * 2^(e-150), scaled by 2^60.  Bits below 2^-60 are dropped.
__device__ __forceinline__ Fx float_to_fixed(float v)
{
    Fx f{0, 0ull};
    const unsigned bits = __float_as_uint(v);
    const int e = (bits >> 23) & 0xff;
    unsigned long long m = bits & 0x7fffffu;
    if (e == 0 && m == 0) return f;
    if (e != 0) m |= 0x800000u;
    const int sh = (e == 0 ? 1 : e) - 90;   // m * 2^(e - 150 + 60)
    unsigned long long lo = 0, hi = 0;
    if (sh >= 0) {
        if (sh < 64) {
            lo = m << sh;
            hi = sh > 40 ? (m >> (64 - sh)) : 0ull;
        } else {
            hi = m << (sh - 64);
        }
    } else if (sh > -64) {
        lo = m >> (-sh);
    }
    if (bits >> 31) {   // two's complement of the 128-bit value
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    f.lo = lo;
    f.hi = (long long)hi;
    return f;
}

// Add v to an adjoint accumulator (0..3: g_wall, 4: g_ste, 5: loss).
__device__ __forceinline__ void adj_add(DevStats* st, int k, double v)
{
    if (v == 0.0) return;
    if (fx_mag(v) >= kFxMag) atomicOr(&st->g_lost, 1u << k);
    else acc_add_fx(k < 4 ? &st->g_wall[k] : (k == 4 ? &st->g_ste : &st->loss), to_fixed(v));
}

__device__ __forceinline__ double acc_read(const Acc128* a)
{
    volatile const Acc128* va = a;
    unsigned long long lo = va->lo;
    long long hi = va->hi;
    return (double)hi * 16.0 + (double)lo * 0x1p-60;
}

__device__ __forceinline__ void acc_clear(Acc128* a)
{
    volatile Acc128* va = a;
    va->lo = 0ull;
    va->hi = 0ll;
}

// a fixed-point value as a double
__device__ __forceinline__ double fx_value(const Fx& v) { return (double)v.hi * 16.0 + (double)v.lo * 0x1p-60; }

// The per-step sums (AccSum): return-less additions of the four limbs, so a
// thread never waits for them.
__device__ __forceinline__ void acc_add_fx(AccSum* a, const Fx& v)
{
    const unsigned long long lo = v.lo, hi = (unsigned long long)v.hi;
    if (lo == 0ull && hi == 0ull) return;
    atomicAdd(&a->limb[0], lo & 0xffffffffull);
    atomicAdd(&a->limb[1], lo >> 32);
    atomicAdd(&a->limb[2], hi & 0xffffffffull);
    atomicAdd(&a->limb[3], hi >> 32);
}

// sum_k limb[k] 2^(32k) modulo 2^128, as a double
__device__ __forceinline__ double acc_read(const AccSum* a)
{
    volatile const unsigned long long* l = a->limb;
    const unsigned long long s0 = l[0], s1 = l[1], s2 = l[2], s3 = l[3];
    const unsigned long long lo = s0 + (s1 << 32);
    const unsigned long long carry = lo < s0 ? 1ull : 0ull;
    const unsigned long long hi = (s1 >> 32) + s2 + (s3 << 32) + carry;
    return (double)(long long)hi * 16.0 + (double)lo * 0x1p-60;
}

__device__ __forceinline__ void acc_clear(AccSum* a)
{
    volatile unsigned long long* l = a->limb;
    l[0] = l[1] = l[2] = l[3] = 0ull;
}

// The stripe a thread adds into: spread over blocks and warps.
__device__ __forceinline__ StepStripe* my_stripe(DevStats* st)
{
    return &st->cur[(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % kStripes];
}

// Totals of one problem's stripes.
struct StatSums {
    unsigned long long e[4], f[4], dir[4], newton, iters, liquid, shifted;
};

// The shift s of a state (FP32 D2Q9 / D2Q5; 0 for the other forms): its tail.
__device__ __forceinline__ float state_shift(const Problem& pb, int parity)
{
    return __ldg(reinterpret_cast<const float*>(static_cast<const char*>(pb.state[parity]) + pb.tail_off));
}

// Read one stripe into `s` and clear it.
__device__ __forceinline__ void stripe_take(StepStripe* stripe, StatSums& s)
{
    volatile StepStripe* c = stripe;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        s.e[j] += c->energy.limb[j];
        s.f[j] += c->flux.limb[j];
        s.dir[j] += c->dir[j];
    }
    s.newton += c->newton;
    s.iters += c->iters;
    s.liquid += c->liquid;
    s.shifted += c->shifted;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c->energy.limb[j] = 0ull;
        c->flux.limb[j] = 0ull;
        c->dir[j] = 0ull;
    }
    c->newton = 0ull;
    c->iters = 0ull;
    c->liquid = 0ull;
    c->shifted = 0ull;
}

// The published step statistics from the stripe totals.
// E = fixed-point sum + (liquid nodes + sum_w Dirichlet nodes of wall w * phi(theta_w)) / Ste.
__device__ __forceinline__ void publish_totals(DevStats* st, const Problem* pb, const StatSums& s)
{
    // every input first, as independent L2 loads (ld.global.cg), so that the
    // publication waits for about one memory round trip, not one per field
    const int have = __ldcg(&st->have_energy);
    const double e_old = __ldcg(&st->energy), imax = __ldcg(&st->imbalance_max);
    const long long steps = __ldcg(&st->steps);
    const int cmax = __ldcg(&st->cur_maxit);
    const unsigned lost = __ldcg(&st->cur_lost);
    double inv_ste = 0.0, wphi[4] = {0.0, 0.0, 0.0, 0.0};
    float shift = 0.0f;
    if (pb) {
        inv_ste = pb->inv_ste;
#pragma unroll
        for (int w = 0; w < 4; ++w) wphi[w] = pb->wall_phi[w];
        if (s.shifted) shift = state_shift(*pb, 0);
    }
    AccSum esum, fsum;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        esum.limb[j] = s.e[j];
        fsum.limb[j] = s.f[j];
    }
    double e = lost & kLostEnergy ? nan_d() : acc_read(&esum);
    const double f = lost & kLostFlux ? nan_d() : acc_read(&fsum);
    if (pb) {
        double c = (double)s.liquid;
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if (s.dir[w]) c += (double)s.dir[w] * wphi[w];
        e += c * inv_ste;
        if (s.shifted) e += (double)s.shifted * (double)shift;
    }
    const double imb = have ? e - e_old - f : 0.0;
    __stcg(&st->imbalance, imb);
    if (have && fabs(imb) > imax) __stcg(&st->imbalance_max, fabs(imb));
    __stcg(&st->energy_prev, e_old);
    __stcg(&st->energy, e);
    __stcg(&st->flux, f);
    __stcg(&st->have_energy, 1);
    __stcg(&st->steps, steps + 1);
    __stcg(&st->newton_nodes, (long long)s.newton);
    __stcg(&st->newton_iters, (long long)s.iters);
    __stcg(&st->newton_max_iter, cmax);
    __stcg(&st->cur_maxit, 0);
    if (lost) __stcg(&st->cur_lost, 0u);
}

// Publish one problem's step statistics and clear its stripes (one thread of
// the last block).
__device__ __forceinline__ void publish_stats(DevStats* st, const Problem* pb)
{
    StatSums s = {};
    for (int k = 0; k < kStripes; ++k) stripe_take(&st->cur[k], s);
    publish_totals(st, pb, s);
}

// The same with one warp: lane k takes stripe k, the warp adds the totals
// (integer sums: the result is the one thread's), lane 0 publishes.
__device__ __forceinline__ void publish_stats_warp(DevStats* st, const Problem* pb, int lane)
{
    static_assert(kStripes == 32, "one stripe per lane");
    StatSums s = {};
    stripe_take(&st->cur[lane], s);
    unsigned long long* v = &s.e[0];   // the 16 fields in order
#pragma unroll
    for (int k = 0; k < 16; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
    if (lane == 0) publish_totals(st, pb, s);
}

// Last-block pattern: every block calls this after its warps have added their
// partial sums; the block that arrives last publishes the statistics of all
// problems (one thread per problem) and resets the ticket.  No block waits.
__device__ __forceinline__ void finish_launch(DevStats* stats, int nprob, unsigned int* ticket, const Problem* probs)
{
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (last) {
        __threadfence();
        for (int p = threadIdx.x; p < nprob; p += blockDim.x) publish_stats(&stats[p], &probs[p]);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) *ticket = 0u;
    }
}

}  // namespace lbm
