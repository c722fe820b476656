// Monte Carlo crystal plasticity (Sec. 2, Eqs. (1)-(3), Table 1) and the
// per-point driving field (Sec. 3, Eq. (4)).  One thread per material point.
//
// Per increment t (Eq. (3), Taylor: every point takes the prescribed strain):
//   eps_c = R^T (t e diag(1,-1/2,-1/2)) R          crystal-frame total strain
//   ee = eps_c - eps_p; s = C : ee                   trial stress (FP32)
//   tau_a = m_a . s . n_a; zeta = {a : |tau_a| > g}  candidates (FP32)
//   per candidate, the single-slip return map |tau_a| - x k = g(gamma + x),
//   k = P:C:P (the same for all twelve), Voce g(gamma + x) = taus - (taus - g)
//   exp(-h0 x/(taus - tau0));
//   energy change of the candidate state  dE_a = -x |tau_a| + x^2 k / 2
//   (E_a = 1/2 ee_a : C : ee_a with ee_a = ee - x sign(tau_a) P_a).  For the
//   selection the candidates use the first Newton iterate from x = 0 in FP32
//   (relative error ~1e-6 for load steps of 1e-4); the chosen system's map is
//   then solved to about 1e-10 (for hr x <= 1e-2 three fixed-point steps on the
//   cubic Taylor form of the Voce term; Newton in FP64 otherwise) and
//   committed, the new resistance from consistency, g = |tau| - k x;
//   p_a = exp(-beta (dE_a - min dE)) / Z (Eq. (1)); R = u0 / 2^32 from
//   Philox(seed; p, t, tag 1); first a with R < sum_{b<=a} p_b (Eq. (2)),
//   all in FP32;
//   commit eps_p += x sign P, gamma += x, g = g(gamma + x).
// After the last increment: sigma = C : (eps_c - eps_p); E_rho = 2 g^2 / G
// (Eq. (4) with sigma_f = g; the Burgers vector cancels); w = 1/2 sigma : ee;
// b = round-half-even(256 scale (w_weight w + E_rho)) clamped to +-2^20.
//
// What bounds it: instructions.  The FP64 pipe, 64 times slower than FP32 here, was
// 62 to 70 % busy with the return map and the conversions around it; the map now
// carries its leading terms as unevaluated sums of two FP32 numbers (relative error
// near 2^-46, where the series it feeds is good to 1e-10).  The resolved shears come
// from one traction per slip plane and component (27 operations) and two operations
// per system instead of nine with the system's vectors from memory; one reciprocal
// serves the twelve divisions by the common k + dg/dgamma; the candidate energies
// run two systems to an operation (packed FP32).  Same bits throughout: 4e6 points,
// two increments: 336 -> 178 us, 1157 -> 730 warp instructions per warp-increment,
// issue 86 % busy; 1e6 points, 20 increments with every output: 734 -> 365 us.
#include <math.h>

#include "common.cuh"

namespace hp {
namespace {

constexpr int kT = 128;

// a double as an unevaluated sum of two floats
struct Pair {
    float hi, lo;
};
__host__ __device__ inline Pair pair_of(double v) {
    Pair p;
    p.hi = (float)v;
    p.lo = (float)(v - (double)p.hi);
    return p;
}

// Constants of the single-slip return map for Voce hardening (taus, tau0, h0).
struct RMConsts {
    double taus, tau0, hr;  // hr = h0 / (taus - tau0); 0 without hardening
    float taus32, hr32, hr2h, hr3s;
    Pair taus2, hr2;
    bool hard;
};

__host__ __device__ inline RMConsts rm_consts(double tau0, double taus, double h0) {
    RMConsts c;
    c.hard = taus - tau0 > 0.0 && h0 > 0.0;
    c.taus = taus;
    c.tau0 = tau0;
    c.hr = c.hard ? h0 / (taus - tau0) : 0.0;
    c.taus32 = (float)taus;
    c.hr32 = (float)c.hr;
    // series coefficients of 1 - exp(-hr x) = hr x - (hr x)^2 / 2 + (hr x)^3 / 6 - ...
    c.hr2h = (float)(0.5 * c.hr * c.hr);
    c.hr3s = (float)(c.hr * c.hr * c.hr / 6.0);
    c.taus2 = pair_of(taus);
    c.hr2 = pair_of(c.hr);
    return c;
}

struct CPArgs {
    float C11, C12, C44;
    RMConsts rm;  // rm_consts(tau0, taus, h0), once per launch on the host
    double k;     // P:C:P, the same for every system of a cubic crystal
    Pair k2;
    float beta;
    float G;
    float e;
    float scale;
    float w_weight;
    uint64_t seed;
    const int32_t* grain;
    const float* quat;
    uint32_t t0;
    int32_t n_incr;
    int64_t P;
    const float* eps_total;  // sample-frame total strain [6][P] per point, or null (Taylor)
    float* eps_p;
    float* gamma;
    float* g;
    float* sigma;
    float* w;
    float* erho;
    int32_t* b;
};

__device__ __forceinline__ void stress(const CPArgs& a, const float ee[6], float s[6]) {
    const float tr = ee[0] + ee[1] + ee[2];
    const float d = a.C11 - a.C12;
    s[0] = d * ee[0] + a.C12 * tr;
    s[1] = d * ee[1] + a.C12 * tr;
    s[2] = d * ee[2] + a.C12 * tr;
    s[3] = 2.0f * a.C44 * ee[3];
    s[4] = 2.0f * a.C44 * ee[4];
    s[5] = 2.0f * a.C44 * ee[5];
}

// exp(-y) for y >= 0: Taylor series for small y, libm otherwise.
__device__ __forceinline__ double exp_neg(double y) {
    if (y < 0.02) {
        // truncation after y^6/720: below 1e-16 relative for y < 0.02
        return 1.0 - y * (1.0 - y * (0.5 - y * (1.0 / 6.0 - y * (1.0 / 24.0 - y * (1.0 / 120.0 - y * (1.0 / 720.0))))));
    }
    return exp(-y);
}

// Newton on the exact FP64 Voce residual at - x k - (taus - sat exp(-hr x)) from
// x; the step uses an FP32 reciprocal of the slope (a relative step error near
// 1e-7 leaves the iteration converging to the same FP64 root, tested on the
// exact residual).  Not inlined: the compiler would otherwise evaluate its
// first residual speculatively on every lane of the common (series) path.
__device__ __noinline__ double newton_slip(double at, double k, double taus, double tau0, double hr, double sat,
                                           double xs) {
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
        const double ey = exp_neg(hr * xs);
        const double f = at - xs * k - (taus - sat * ey);
        if (fabs(f) < 1e-13 * tau0) break;
        const double fp = -k - sat * hr * ey;
        xs -= f * (double)(1.0f / (float)fp);
    }
    return xs;
}

// Slip x >= 0 of one system with resolved shear |tau| = at > g (slip resistance
// g, P:C:P = k): the root of f(x) = (at - g) - k x - sat (1 - exp(-hr x)),
// sat = taus - g, i.e. |tau| - x k = g(gamma + x) for the Voce law; x = (at - g) / k
// without hardening.  *g_new = g(gamma + x), from consistency at - k x.
//
// With y = hr x and q = sat hr / K (K = k + sat hr, q < 1), the exponential's
// cubic Taylor polynomial changes x by at most q y^3 / 24 relative; where that
// is below 4e-10 (q y^3 <= 1e-8, y <= 1e-2) x solves
// x = (a0 + c2 x^2 - c3 x^3) / K with a0 = at - g, c2 = sat hr^2 / 2,
// c3 = sat hr^3 / 6.  a0 (exact), K, the leading term a0 / K and k x are pairs of
// FP32 numbers: error-free sums and products (Dekker 1971, Knuth's two-sum; the
// products by fused multiply-add), the quotient by one correction of its FP32
// value with the exact remainder, relative error near 2^-46.  The correction
// x^2 (c2 - c3 x) / K is at most q y / 2 of x and each fixed-point step shrinks
// its error by a factor q y, so three steps in FP32 leave it below 1e-10.  Other
// slips take Newton on the exact FP64 residual, and so that the committed FP32 slip
// and resistance are those of FP64 arithmetic throughout, with and without hardening, a
// result within 2^-14 of halfway between two FP32 numbers is formed again in FP64 (one
// in 8000).
__device__ __forceinline__ Pair two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair fast_sum(float a, float b) {  // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return Pair{s, __fsub_rn(b, __fsub_rn(s, a))};
}

// v > 0 within 2^-14 of halfway between two FP32 numbers: rounding the sum to FP32 may go
// either way with an error of 2^-46.  Below a power of two the numbers lie half as far
// apart as above it.
__device__ __forceinline__ bool near_half(Pair v) {
    const int below = (int)((uint32_t)__float_as_int(v.lo) >> 31);
    const float half = __int_as_float(((__float_as_int(v.hi) - below) & 0x7F800000) - (24 << 23));
    return fabsf(v.lo) > half * (1.0f - 0x1p-14f);
}
// The map in FP64: the quotient without hardening; with it the series where its bound
// holds, Newton otherwise.  Not inlined (rare; see newton_slip).
__device__ __noinline__ Pair slip_fp64(float at_f, float g, double k, const RMConsts& c, float* g_new) {
    const double at = at_f, sat = c.taus - (double)g, K = k + sat * c.hr;
    if (!c.hard) {
        *g_new = g;
        return pair_of((at - (double)g) / k);
    }
    const float rKf = 1.0f / (float)K;
    double rK = (double)rKf;
    rK = rK * (2.0 - K * rK);
    double xs = (at - (double)g) * rK;
    const float x1f = (float)xs, sr = (c.taus32 - g) * rKf, y = c.hr32 * x1f, q = c.hr32 * sr;
    if (y <= 1e-2f && y * y * y * q <= 1e-8f) {
        const float c2 = c.hr2h * sr, c3 = c.hr3s * sr;
        float d = 0.0f;
        for (int it = 0; it < 3; ++it) {
            const float xf = x1f + d;
            d = xf * xf * (c2 - c3 * xf);
        }
        xs += (double)d;
    } else {
        xs = newton_slip(at, k, c.taus, c.tau0, c.hr, sat, xs);
    }
    *g_new = (float)(at - k * xs);
    return pair_of(xs);
}

__device__ __forceinline__ Pair return_map(float at, float g, Pair k, double kd, const RMConsts& c, float* g_new) {
    const Pair a0 = two_sum(at, -g);
    Pair K = k;
    if (c.hard) {
        const Pair sat = two_sum(c.taus2.hi, -g);
        const float sl = __fadd_rn(sat.lo, c.taus2.lo);
        const float p = __fmul_rn(sat.hi, c.hr2.hi);
        const float e = __fmaf_rn(sat.hi, c.hr2.lo, __fmaf_rn(sl, c.hr2.hi, __fmaf_rn(sat.hi, c.hr2.hi, -p)));
        K = two_sum(k.hi, p);
        K = fast_sum(K.hi, __fadd_rn(K.lo, __fadd_rn(k.lo, e)));
    }
    const float rK = __frcp_rn(K.hi);
    const float q0 = __fmul_rn(a0.hi, rK);
    const float rem = __fadd_rn(__fmaf_rn(-q0, K.hi, a0.hi), __fmaf_rn(-q0, K.lo, a0.lo));
    Pair x = fast_sum(q0, __fmul_rn(rem, rK));
    if (!c.hard) {
        *g_new = g;
        return near_half(x) ? slip_fp64(at, g, kd, c, g_new) : x;
    }
    const float sr = (c.taus32 - g) * rK;  // sat / K
    const float y = c.hr32 * x.hi, q = c.hr32 * sr;
    if (y <= 1e-2f && y * y * y * q <= 1e-8f) {
        const float c2 = c.hr2h * sr, c3 = c.hr3s * sr;
        float d = 0.0f;
#pragma unroll
        for (int it = 0; it < 3; ++it) {
            const float xf = x.hi + d;
            d = xf * xf * (c2 - c3 * xf);
        }
        const Pair s = fast_sum(x.hi, d);
        x = fast_sum(s.hi, __fadd_rn(s.lo, x.lo));
    } else {
        return slip_fp64(at, g, kd, c, g_new);
    }
    const float p = __fmul_rn(k.hi, x.hi);
    const float e = __fmaf_rn(k.hi, x.lo, __fmaf_rn(k.lo, x.hi, __fmaf_rn(k.hi, x.hi, -p)));
    const Pair t = two_sum(at, -p), r = fast_sum(t.hi, __fsub_rn(t.lo, e));
    *g_new = r.hi;
    if (near_half(x) || near_half(r)) return slip_fp64(at, g, kd, c, g_new);
    return x;
}


// The return map as the plasticity kernel evaluates it, for testing.
__global__ void k_rm_eval(const float* __restrict__ at, const float* __restrict__ g, const double* __restrict__ k,
                          int64_t n, RMConsts c, double* __restrict__ x) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gn;
    const Pair v = return_map(at[i], g[i], pair_of(k[i]), k[i], c, &gn);
    x[i] = (double)v.hi + (double)v.lo;
}

// Packed FP32: two numbers in a 64-bit register, each rounded as by itself.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}

// The twelve {111}<110> systems as the kernel lays them out in shared memory: slip
// direction m, plane normal n, and the off-diagonal sums of the Schmid tensor.
constexpr float kCn = 0.57735026918962576f, kCm = 0.70710678118654752f;
__device__ const int8_t kSigns[12][6] = {{0, 1, -1, 1, 1, 1},  {-1, 0, 1, 1, 1, 1},  {1, -1, 0, 1, 1, 1},
                                         {0, 1, -1, -1, 1, 1}, {1, 0, 1, -1, 1, 1},  {1, 1, 0, -1, 1, 1},
                                         {0, 1, 1, 1, -1, 1},  {1, 0, -1, 1, -1, 1}, {1, 1, 0, 1, -1, 1},
                                         {0, 1, 1, 1, 1, -1},  {1, 0, 1, 1, 1, -1},  {1, -1, 0, 1, 1, -1}};

// Resolved shears m_a . s . n_a of all systems from the stress s (Voigt): the
// traction of each plane (normal cn (SX, SY, SZ)), then two components of it per
// system.  The order of every sum is that of the plain expression.
template <int SX, int SY, int SZ>
__device__ __forceinline__ void traction(const float s[6], float a5, float a1, float a3, float t[3]) {
    // a5, a1, a3: cn times s[5], s[1], s[3]
    t[0] = __fmaf_rn(s[4], SZ * kCn, __fmaf_rn(s[0], SX * kCn, SY * a5));
    t[1] = __fmaf_rn(s[3], SZ * kCn, __fmaf_rn(s[5], SX * kCn, SY * a1));
    t[2] = __fmaf_rn(s[2], SZ * kCn, __fmaf_rn(s[4], SX * kCn, SY * a3));
}
template <int M0, int M1, int M2>
__device__ __forceinline__ float along(const float t[3]) {
    if (M2 == 0) return __fmaf_rn(M0 * kCm, t[0], __fmul_rn(M1 * kCm, t[1]));
    return __fmaf_rn(M2 * kCm, t[2], M0 == 0 ? __fmul_rn(M1 * kCm, t[1]) : __fmul_rn(M0 * kCm, t[0]));
}
__device__ __forceinline__ void resolved(const float s[6], float tau[12]) {
    const float a5 = __fmul_rn(s[5], kCn), a1 = __fmul_rn(s[1], kCn), a3 = __fmul_rn(s[3], kCn);
    float t[3];
    traction<1, 1, 1>(s, a5, a1, a3, t);
    tau[0] = along<0, 1, -1>(t); tau[1] = along<-1, 0, 1>(t); tau[2] = along<1, -1, 0>(t);
    traction<-1, 1, 1>(s, a5, a1, a3, t);
    tau[3] = along<0, 1, -1>(t); tau[4] = along<1, 0, 1>(t); tau[5] = along<1, 1, 0>(t);
    traction<1, -1, 1>(s, a5, a1, a3, t);
    tau[6] = along<0, 1, 1>(t); tau[7] = along<1, 0, -1>(t); tau[8] = along<1, 1, 0>(t);
    traction<1, 1, -1>(s, a5, a1, a3, t);
    tau[9] = along<0, 1, 1>(t); tau[10] = along<1, 0, 1>(t); tau[11] = along<1, -1, 0>(t);
}

template <bool STRAIN>
__global__ void __launch_bounds__(kT) k_cp(const __grid_constant__ CPArgs a) {
    __shared__ float sys[12][9];  // m, n, off-diagonal sums (yz, xz, xy); odd pitch: few bank conflicts
    if (threadIdx.x < 12) {
        float* y = sys[threadIdx.x];
        for (int i = 0; i < 3; ++i) y[i] = kSigns[threadIdx.x][i] * kCm;
        for (int i = 3; i < 6; ++i) y[i] = kSigns[threadIdx.x][i] * kCn;
        y[6] = __fmaf_rn(y[2], y[4], __fmul_rn(y[1], y[5]));
        y[7] = __fmaf_rn(y[2], y[3], __fmul_rn(y[0], y[5]));
        y[8] = __fmaf_rn(y[1], y[3], __fmul_rn(y[0], y[4]));
    }
    __syncthreads();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.P) return;
    const float* qq = a.quat + 4 * (int64_t)a.grain[p];
    float qw = qq[0], qx = qq[1], qy = qq[2], qz = qq[3];
    const float inv = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
    qw *= inv; qx *= inv; qy *= inv; qz *= inv;
    float R[3][3];
    R[0][0] = 1.f - 2.f * (qy * qy + qz * qz); R[0][1] = 2.f * (qx * qy - qw * qz); R[0][2] = 2.f * (qx * qz + qw * qy);
    R[1][0] = 2.f * (qx * qy + qw * qz); R[1][1] = 1.f - 2.f * (qx * qx + qz * qz); R[1][2] = 2.f * (qy * qz - qw * qx);
    R[2][0] = 2.f * (qx * qz - qw * qy); R[2][1] = 2.f * (qy * qz + qw * qx); R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
    // unit-strain crystal-frame tensor U = R^T diag(1,-1/2,-1/2) R (Voigt order xx yy zz yz xz xy)
    const int I[6] = {0, 1, 2, 1, 0, 0}, J[6] = {0, 1, 2, 2, 2, 1};
    float U[6];
#pragma unroll
    for (int v = 0; v < 6; ++v)
        U[v] = R[0][I[v]] * R[0][J[v]] - 0.5f * (R[1][I[v]] * R[1][J[v]] + R[2][I[v]] * R[2][J[v]]);
    // a point with its own total strain (elastic-equilibrium coupling): the
    // crystal-frame strain R^T eps R takes the place of t e U
    float Ut[6];
    if (STRAIN) {
        float es[3][3];
        const float e0 = a.eps_total[p], e1 = a.eps_total[a.P + p], e2 = a.eps_total[2 * a.P + p];
        const float e3 = a.eps_total[3 * a.P + p], e4 = a.eps_total[4 * a.P + p], e5 = a.eps_total[5 * a.P + p];
        es[0][0] = e0; es[1][1] = e1; es[2][2] = e2;
        es[1][2] = es[2][1] = e3; es[0][2] = es[2][0] = e4; es[0][1] = es[1][0] = e5;
#pragma unroll
        for (int v = 0; v < 6; ++v) {
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int l = 0; l < 3; ++l) acc += R[k][I[v]] * es[k][l] * R[l][J[v]];
            Ut[v] = acc;
        }
    }
    float ep[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) ep[v] = a.eps_p[(int64_t)v * a.P + p];
    float gam = a.gamma[p];
    float gres = a.g[p];
    const bool hard = a.rm.hard;
    const float hr32 = a.rm.hr32, taus32 = a.rm.taus32, kf = a.k2.hi;
    float ee[6], s[6];
#pragma unroll 1
    for (int32_t inc = 1; inc <= a.n_incr; ++inc) {
        const uint32_t t = a.t0 + (uint32_t)inc;
        const float et = (float)t * a.e;
#pragma unroll
        for (int v = 0; v < 6; ++v) ee[v] = (STRAIN ? Ut[v] : et * U[v]) - ep[v];
        stress(a, ee, s);
        float tau[12];
        resolved(s, tau);
        // candidate energies for the selection (Eq. (1)): the linearised
        // return map x_a = (|tau_a| - g)/(k_a + dg/dgamma), relative error
        // about 1e-6 against the converged one, in FP32.  The common divisor's
        // correctly rounded reciprocal r serves all: q = a r corrected once by
        // its exact remainder is the correctly rounded quotient (Markstein, IBM
        // J. Res. Dev. 34 (1990) 111).
        const float hg = hard ? (taus32 - gres) * hr32 : 0.0f;
        const float den = kf + hg, r = __frcp_rn(den);
        // two systems at a time in the packed FP32 operations
        float wgt[12], dEmin = 3.4e38f;
        bool any = false;
        const uint64_t g2 = pack2(-gres, -gres), r2 = pack2(r, r), d2 = pack2(-den, -den), h2 = pack2(0.5f, 0.5f),
                       kf2 = pack2(kf, kf);
#pragma unroll
        for (int al = 0; al < 12; al += 2) {
            const float t0 = fabsf(tau[al]), t1 = fabsf(tau[al + 1]);
            const uint64_t at = pack2(t0, t1), num = add2(at, g2), q = mul2(num, r2);
            const uint64_t xx = fma2(fma2(q, d2, num), r2, q);
            const uint64_t dE = fma2(mul2(mul2(h2, xx), xx), kf2, mul2(xx, pack2(-t0, -t1)));
            float e0, e1;
            unpack2(dE, e0, e1);
            any |= t0 > gres || t1 > gres;
            wgt[al] = t0 > gres ? e0 : 3.4e38f;
            wgt[al + 1] = t1 > gres ? e1 : 3.4e38f;
            dEmin = fminf(fminf(dEmin, wgt[al]), wgt[al + 1]);
        }
        if (!any) continue;
        // cumulative weights; a system that is no candidate adds nothing
        float Z = 0.0f;
#pragma unroll
        for (int al = 0; al < 12; ++al) {
            const float e = expf(-a.beta * (wgt[al] - dEmin));
            Z += wgt[al] < 3.4e38f ? e : 0.0f;
            wgt[al] = Z;
        }
        uint32_t u;
        if ((uint64_t)p >> 32) {
            u = draw(a.seed, (uint64_t)p, t, kTagMcp, 0).x;
        } else {
            SweepKey key;
            sweep_key(a.seed, t, &key);
            u = sweep_draw(key, (uint32_t)p, (uint32_t)kTagMcp << 24).x;
        }
        // first a with R < sum_{b <= a} w_b / Z, tested as R Z < sum_{b <= a} w_b
        // (no division per candidate; FP32 sums of at most 12 positive terms,
        // relative error near 1e-7, far inside the 1e-5 band around a decision
        // where the FP64 oracle and this kernel may legitimately differ); the
        // last candidate when rounding leaves none
        const float RZ = (float)u * (1.0f / 4294967296.0f) * Z;
        int pick = -1;
        float tau_pick = 0.0f;
#pragma unroll
        for (int al = 11; al >= 0; --al)
            if (RZ < wgt[al]) {
                pick = al;
                tau_pick = tau[al];
            }
        if (pick < 0)
#pragma unroll
            for (int al = 0; al < 12; ++al)
                if (fabsf(tau[al]) > gres) {
                    pick = al;
                    tau_pick = tau[al];
                }
        // the single-slip return map of the chosen system
        float g_next;
        const Pair x = return_map(fabsf(tau_pick), gres, a.k2, a.k, a.rm, &g_next);
        const float sg = tau_pick > 0.f ? 1.f : -1.f;
        const float* y = sys[pick];
        const float m0 = y[0], m1 = y[1], m2 = y[2], n0 = y[3], n1 = y[4], n2 = y[5];
        const float xf = x.hi * sg;
        ep[0] += xf * m0 * n0;
        ep[1] += xf * m1 * n1;
        ep[2] += xf * m2 * n2;
        ep[3] += xf * 0.5f * y[6];
        ep[4] += xf * 0.5f * y[7];
        ep[5] += xf * 0.5f * y[8];
        gam += x.hi;
        gres = g_next;  // g(gamma + x) = |tau| - k x at the solved slip
    }
#pragma unroll
    for (int v = 0; v < 6; ++v) a.eps_p[(int64_t)v * a.P + p] = ep[v];
    a.gamma[p] = gam;
    a.g[p] = gres;
    if (a.sigma || a.w || a.erho || a.b) {
        const uint32_t t = a.t0 + (uint32_t)a.n_incr;
        const float et = (float)t * a.e;
#pragma unroll
        for (int v = 0; v < 6; ++v) ee[v] = (STRAIN ? Ut[v] : et * U[v]) - ep[v];
        stress(a, ee, s);
        if (a.sigma)
#pragma unroll
            for (int v = 0; v < 6; ++v) a.sigma[(int64_t)v * a.P + p] = s[v];
        const float w = 0.5f * (s[0] * ee[0] + s[1] * ee[1] + s[2] * ee[2]) + (s[3] * ee[3] + s[4] * ee[4] + s[5] * ee[5]);
        const float er = 2.0f * gres * gres / a.G;
        if (a.w) a.w[p] = w;
        if (a.erho) a.erho[p] = er;
        if (a.b) {
            float v = rintf(256.0f * a.scale * (a.w_weight * w + er));
            v = fminf(fmaxf(v, -1048576.0f), 1048576.0f);
            a.b[p] = (int32_t)v;
        }
    }
}

__global__ void k_cp_reset(int64_t P, float* eps_p, float* gamma, float* g, float tau0) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
#pragma unroll
    for (int v = 0; v < 6; ++v) eps_p[(int64_t)v * P + p] = 0.0f;
    gamma[p] = 0.0f;
    g[p] = tau0;
}

// P:C:P of a {111}<110> system for cubic moduli (every system's, by symmetry): the
// sum over components of P = (m n^T + n m^T) / 2, m = (0, 1, -1)/sqrt 2, n = (1, 1, 1)/sqrt 3.
double slip_stiffness(const hp_cp_params* prm) {
    const double sn = 1.0 / sqrt(3.0), sm = 1.0 / sqrt(2.0);
    const double m[3] = {0.0, sm, -sm}, n[3] = {sn, sn, sn};
    double P[3][3], v = 0.0;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) P[i][j] = 0.5 * (m[i] * n[j] + n[i] * m[j]);
    const double tr = P[0][0] + P[1][1] + P[2][2];
    for (int i = 0; i < 3; ++i) v += P[i][i] * ((prm->C11 - prm->C12) * P[i][i] + prm->C12 * tr);
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (i != j) v += P[i][j] * 2.0 * prm->C44 * P[i][j];
    return v;
}

}  // namespace
}  // namespace hp

using namespace hp;

extern "C" int hp_debug_return_map(const hp_cp_params* prm, const float* at, const float* g, const double* k,
                                   int64_t n, double* x, void* stream) {
    if (!prm || !at || !g || !k || !x || n < 0) return set_error(HP_ERR_ARG, "hp_debug_return_map: bad arguments");
    if (n == 0) return HP_OK;
    ::hp::count_launch();
    k_rm_eval<<<(unsigned)((n + 255) / 256), 256, 0, as_stream(stream)>>>(at, g, k, n, rm_consts(prm->tau0, prm->taus, prm->h0),
                                                                           x);
    HP_LAUNCH_CHECK("k_rm_eval");
    return HP_OK;
}

extern "C" int hp_cp_reset(const hp_cp_params* prm, hp_cp_state* st, void* stream) {
    if (!prm || !st || st->P < 1 || !st->eps_p || !st->gamma || !st->g)
        return set_error(HP_ERR_ARG, "hp_cp_reset: bad arguments");
    ::hp::count_launch();
    k_cp_reset<<<(unsigned)((st->P + 255) / 256), 256, 0, as_stream(stream)>>>(st->P, st->eps_p, st->gamma, st->g,
                                                                               (float)prm->tau0);
    HP_LAUNCH_CHECK("k_cp_reset");
    return HP_OK;
}

extern "C" int hp_cp_step(const hp_cp_params* prm, uint64_t seed, const int32_t* grain, const float* quat,
                          uint32_t t0, int32_t n_incr, hp_cp_state* st, float* sigma, float* w, float* erho,
                          int32_t* b, void* stream) {
    hp::Range r_("hp_cp_step");
    if (!prm || !st || !grain || !quat || n_incr < 0 || st->P < 1 || !st->eps_p || !st->gamma || !st->g)
        return set_error(HP_ERR_ARG, "hp_cp_step: bad arguments");
    if (!(prm->C11 > prm->C12) || !(prm->C44 > 0) || !(prm->tau0 > 0) || !(prm->G > 0))
        return set_error(HP_ERR_ARG, "hp_cp_step: bad material constants");
    CPArgs a;
    a.k = slip_stiffness(prm);
    a.k2 = pair_of(a.k);
    a.C11 = (float)prm->C11; a.C12 = (float)prm->C12; a.C44 = (float)prm->C44;
    a.rm = rm_consts(prm->tau0, prm->taus, prm->h0);
    a.beta = (float)prm->beta; a.G = (float)prm->G; a.e = (float)prm->e_incr; a.scale = (float)prm->energy_scale;
    a.w_weight = (float)prm->w_weight;
    a.seed = seed; a.grain = grain; a.quat = quat; a.t0 = t0; a.n_incr = n_incr; a.P = st->P;
    a.eps_total = nullptr;
    a.eps_p = st->eps_p; a.gamma = st->gamma; a.g = st->g;
    a.sigma = sigma; a.w = w; a.erho = erho; a.b = b;
    ::hp::count_launch();
    k_cp<false><<<(unsigned)((st->P + kT - 1) / kT), kT, 0, as_stream(stream)>>>(a);
    HP_LAUNCH_CHECK("k_cp");
    return HP_OK;
}

extern "C" int hp_cp_step_strain(const hp_cp_params* prm, uint64_t seed, const int32_t* grain, const float* quat,
                                 uint32_t t, const float* eps_total, hp_cp_state* st, float* sigma, float* w,
                                 float* erho, int32_t* b, void* stream) {
    hp::Range r_("hp_cp_step_strain");
    if (!prm || !st || !grain || !quat || !eps_total || t < 1 || st->P < 1 || !st->eps_p || !st->gamma || !st->g)
        return set_error(HP_ERR_ARG, "hp_cp_step_strain: bad arguments");
    if (!(prm->C11 > prm->C12) || !(prm->C44 > 0) || !(prm->tau0 > 0) || !(prm->G > 0))
        return set_error(HP_ERR_ARG, "hp_cp_step_strain: bad material constants");
    CPArgs a;
    a.k = slip_stiffness(prm);
    a.k2 = pair_of(a.k);
    a.C11 = (float)prm->C11; a.C12 = (float)prm->C12; a.C44 = (float)prm->C44;
    a.rm = rm_consts(prm->tau0, prm->taus, prm->h0);
    a.beta = (float)prm->beta; a.G = (float)prm->G; a.e = (float)prm->e_incr; a.scale = (float)prm->energy_scale;
    a.w_weight = (float)prm->w_weight;
    a.seed = seed; a.grain = grain; a.quat = quat; a.t0 = t - 1; a.n_incr = 1; a.P = st->P;
    a.eps_total = eps_total;
    a.eps_p = st->eps_p; a.gamma = st->gamma; a.g = st->g;
    a.sigma = sigma; a.w = w; a.erho = erho; a.b = b;
    ::hp::count_launch();
    k_cp<true><<<(unsigned)((st->P + kT - 1) / kT), kT, 0, as_stream(stream)>>>(a);
    HP_LAUNCH_CHECK("k_cp");
    return HP_OK;
}
