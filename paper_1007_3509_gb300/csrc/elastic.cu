// Periodic elastic equilibrium of the cubic polycrystal on the lattice grid
// (Sec. 5: the plasticity is coupled to a deformation solver and each load
// increment is iterated to quasi-static equilibrium; here the solver is the
// Lippmann-Schwinger fixed point of Moulinec and Suquet on the voxel grid, one
// material point per voxel).  FP32 throughout.
//
//   sigma(x) = C(x) : (eps(x) - eps_p(x))        evaluated in the crystal frame
//   tau      = sigma - C0 : eps                   C0 isotropic (lambda0, mu0)
//   eps^hat  = -Gamma0 : tau^hat,  xi != 0        Green operator of C0
//   eps^hat(0) = E; zero on the Nyquist planes of even axes
//   Gamma0 : tau = (n (x) a + a (x) n)/(2 mu0) - kappa (n . a) n (x) n,
//   n = xi/|xi|, a = tau n, kappa = (lambda0 + mu0)/(mu0 (lambda0 + 2 mu0))
//
// The fields are real and the strain of the Nyquist planes is zero, so the
// transforms keep kx = 0 .. nx/2 - 1 only: six fields of N/2 complex values.  One
// iteration is four passes over them (three where ny = 1):
//   x    inverse transform along x, strain update, polarisation of the new
//        strain, forward transform along x (k_el_x)
//   y    forward along y (k_el_fft)
//   z    forward along z, Green operator, inverse along z (k_el_z)
//   y    inverse along y
// What bounds it: memory.  An iteration moves 268 bytes per voxel (x 124: spectrum,
// strain, plastic strain and grain in, strain and spectrum out; y, z, y 48 each);
// with complex fields of full size, a pass per axis and direction and one each for
// polarisation, Green operator and update it was 760.  256^3, one iteration: 11.2 ms
// with those passes (radix 2 in shared memory), 1.13 ms now: x 0.58 ms (3.5 TB/s;
// 12 warps an SM, for the shared memory), y 0.14 ms each (5.7 TB/s), z 0.26 ms
// (3.1 TB/s; 16 warps an SM, for the registers).
//
// Every line is transformed in registers, eight points a thread, by the
// self-sorting (Stockham) passes of radix 8 with a last one of 4 or 2, as given by
// Govindaraju et al., "High performance discrete Fourier transforms on graphics
// processors" (SC 2008): a pass reads points t + s n/8 (s = 0 .. 7) of its line and
// the last one leaves them in natural order at the same places, so that global
// memory is read and written straight from registers and shared memory only carries
// the exchange between two passes.  A real line of n values is the complex line of
// its n/2 pairs, unpacked by the usual even/odd identity.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "common.cuh"

namespace hp {
namespace {

constexpr int kET = 256;

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// a times DIR i
template <int DIR>
__device__ __forceinline__ float2 cmuli(float2 a) { return DIR < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x); }
// a times w, or its conjugate for the inverse transform (tables hold exp(-i ...))
template <int DIR>
__device__ __forceinline__ float2 ctw(float2 a, float2 w) { return cmul(a, DIR < 0 ? w : make_float2(w.x, -w.y)); }

// v_r <- sum_q v_q exp(DIR 2 pi i q r / R), in place, natural order
template <int DIR>
__device__ __forceinline__ void dft2(float2& a, float2& b) {
    const float2 t = csub(a, b);
    a = cadd(a, b);
    b = t;
}
template <int DIR>
__device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d) {
    const float2 s = cadd(a, c), t = csub(a, c), u = cadd(b, d), v = cmuli<DIR>(csub(b, d));
    a = cadd(s, u);
    c = csub(s, u);
    b = cadd(t, v);
    d = csub(t, v);
}
template <int DIR>
__device__ __forceinline__ void dft8(float2* v) {
    dft4<DIR>(v[0], v[2], v[4], v[6]);
    dft4<DIR>(v[1], v[3], v[5], v[7]);
    constexpr float h = 0.70710678118654752f;
    // odd terms times exp(DIR 2 pi i k / 8)
    v[3] = make_float2(h * (v[3].x - DIR * v[3].y), h * (v[3].y + DIR * v[3].x));
    v[5] = cmuli<DIR>(v[5]);
    v[7] = make_float2(-h * (v[7].x + DIR * v[7].y), h * (DIR * v[7].x - v[7].y));
    const float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// A line of n = 2^LOGN points held by T threads, E points each: thread t has
// points t + s T in v[s].  tw: exp(-2 pi i k / (n STEP)) for k < n STEP.  X carries
// a pass's results to the next: put(index, value), get(index), wait().
template <int LOGN>
struct Line {
    static constexpr int n = 1 << LOGN, E = n < 8 ? n : 8, T = n / E;
};

template <int LOGN, int DIR, int STEP, int LOGNS, class X>
__device__ __forceinline__ void fft_from(float2* v, int t, const float2* tw, X& x) {
    constexpr int n = 1 << LOGN, E = Line<LOGN>::E, T = Line<LOGN>::T, Ns = 1 << LOGNS;
    constexpr int L = LOGN - LOGNS, LR = L > 3 ? 3 : L, R = 1 << LR, G = E / R;
    if constexpr (L > 0) {
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const int jm = (t + q * T) & (Ns - 1);
            if (LOGNS)
#pragma unroll
                for (int r = 1; r < R; ++r) v[q + G * r] = ctw<DIR>(v[q + G * r], tw[jm * r * (n / (Ns * R)) * STEP]);
            if constexpr (R == 2) dft2<DIR>(v[q], v[q + G]);
            if constexpr (R == 4) dft4<DIR>(v[q], v[q + G], v[q + 2 * G], v[q + 3 * G]);
            if constexpr (R == 8) dft8<DIR>(v);
        }
        if constexpr (L > LR) {
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int j = t + q * T, d = ((j >> LOGNS) << (LOGNS + LR)) + (j & (Ns - 1));
#pragma unroll
                for (int r = 0; r < R; ++r) x.put(d + r * Ns, v[q + G * r]);
            }
            x.wait();
#pragma unroll
            for (int s = 0; s < E; ++s) v[s] = x.get(t + s * T);
            x.done();
            fft_from<LOGN, DIR, STEP, LOGNS + LR>(v, t, tw, x);
        }
    }
}

template <int N_>
__device__ __forceinline__ void fill_twiddles(float2* tw, int threads) {
    for (int k = threadIdx.x; k < N_; k += threads) {
        float s, c;
        sincospif(2.0f * (float)k / (float)N_, &s, &c);
        tw[k] = make_float2(c, -s);
    }
}

// Exchange across a block whose lines lie side by side (line w of W fastest), so
// that no two lanes of a half-warp meet in a bank; BUFS = 2 takes turns with two
// buffers and saves the barrier after the reads.  A line by itself has a gap after
// every eighth point instead.
template <int W, int N_, int BUFS>
struct XBlock {
    float2* sm;
    int w;
    __device__ __forceinline__ static int at(int i) { return W == 1 ? i + (i >> 3) : i * W; }
    __device__ __forceinline__ void put(int i, float2 v) { sm[at(i) + w] = v; }
    __device__ __forceinline__ float2 get(int i) const { return sm[at(i) + w]; }
    __device__ __forceinline__ void wait() { __syncthreads(); }
    __device__ __forceinline__ void done() {
        if (BUFS == 1) __syncthreads();
        else sm = flip(sm);
    }
    float2* other;
    __device__ __forceinline__ float2* flip(float2* p) { float2* o = other; other = p; return o; }
};

// lines per block of the transforms along y and z: as wide in x as the threads
// allow (16 adjacent complex values are a 128-byte line)
template <int LOGN>
struct YCfg {
    static constexpr int n = 1 << LOGN;
    static constexpr int W = LOGN >= 9 ? 8 : LOGN >= 7 ? 16 : 2048 / (n < 8 ? 8 : n);
    static constexpr int threads = W * Line<LOGN>::T;
    static constexpr size_t smem = sizeof(float2) * ((size_t)n * W + n);
};
template <int LOGN, bool ONE>
struct ZCfg {
    static constexpr int n = 1 << LOGN;
    static constexpr int W = ONE ? 1 : LOGN >= 10 ? 4 : LOGN >= 8 ? 8 : 1024 / (n < 8 ? 8 : n);
    static constexpr int threads = W * Line<LOGN>::T;
    static constexpr int buf = W == 1 ? n + n / 8 : n * W;
    static constexpr size_t smem = sizeof(float2) * (2 * (size_t)buf + n);
};

// Transform along y of all six fields: lines (x, z, field), x fastest.
template <int LOGN, int DIR>
__global__ void __launch_bounds__(YCfg<LOGN>::threads) k_el_fft(float2* __restrict__ data, int nxh, int64_t lines) {
    using C = YCfg<LOGN>;
    constexpr int n = C::n, W = C::W, E = Line<LOGN>::E, T = Line<LOGN>::T;
    extern __shared__ __align__(16) float2 esm[];
    float2* tw = esm + n * W;
    fill_twiddles<n>(tw, C::threads);
    const int w = threadIdx.x % W, t = threadIdx.x / W;
    const int64_t L = (int64_t)blockIdx.x * W + w;
    const bool on = L < lines;
    const int64_t r = L / nxh;
    float2* p = data + r * ((int64_t)n * nxh) + (L - r * nxh) + (int64_t)t * nxh;
    const int64_t st = (int64_t)T * nxh;
    float2 v[E];
#pragma unroll
    for (int s = 0; s < E; ++s) v[s] = on ? p[s * st] : make_float2(0.f, 0.f);
    __syncthreads();
    XBlock<W, n, 1> x{esm, w, nullptr};
    fft_from<LOGN, DIR, 1, 0>(v, t, tw, x);
    if (on)
#pragma unroll
        for (int s = 0; s < E; ++s) p[s * st] = v[s];
}

struct ElArgs {
    int nx, ny, nz;
    int64_t N;
    float C11, C12, C44, lam0, mu0;
    const int32_t* grain;
    const float* quat;
    const float* eps_p;  // crystal frame, [6][N], or null
    float E[6];
    int nxh;             // kx kept: nx / 2 (1 for nx = 1)
    int64_t Nh;          // complex values per field: nxh ny nz
    int mean;            // the strain of the voxels is E throughout (not yet in eps)
    float* eps;
    float* sigma;        // stress wanted with the last update, or null
    unsigned* change;    // largest strain change (bits of a non-negative float)
};

__device__ __forceinline__ void rot_of(const float* qq, float R[3][3]) {
    float w = qq[0], x = qq[1], y = qq[2], z = qq[3];
    const float inv = rsqrtf(w * w + x * x + y * y + z * z);
    w *= inv; x *= inv; y *= inv; z *= inv;
    R[0][0] = 1.f - 2.f * (y * y + z * z); R[0][1] = 2.f * (x * y - w * z); R[0][2] = 2.f * (x * z + w * y);
    R[1][0] = 2.f * (x * y + w * z); R[1][1] = 1.f - 2.f * (x * x + z * z); R[1][2] = 2.f * (y * z - w * x);
    R[2][0] = 2.f * (x * z - w * y); R[2][1] = 2.f * (y * z + w * x); R[2][2] = 1.f - 2.f * (x * x + y * y);
}

__device__ __forceinline__ void sym(const float v[6], float t[3][3]) {
    t[0][0] = v[0]; t[1][1] = v[1]; t[2][2] = v[2];
    t[1][2] = t[2][1] = v[3]; t[0][2] = t[2][0] = v[4]; t[0][1] = t[1][0] = v[5];
}

// sample-frame stress at sample-frame strain e (Voigt) of a crystal with
// orientation qq and crystal-frame plastic strain ep
__device__ __forceinline__ void crystal_stress(const ElArgs& a, const float* qq, const float ep[6], const float e[6],
                                               float s_out[6]) {
    float R[3][3], es[3][3], ec[3][3], sc[3][3], tmp[3][3], et[3][3];
    rot_of(qq, R);
    sym(e, es);
    // ec = R^T es R - ep
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) tmp[p][q] = es[p][0] * R[0][q] + es[p][1] * R[1][q] + es[p][2] * R[2][q];
    sym(ep, et);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q)
            ec[p][q] = R[0][p] * tmp[0][q] + R[1][p] * tmp[1][q] + R[2][p] * tmp[2][q] - et[p][q];
    const float tr = ec[0][0] + ec[1][1] + ec[2][2];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) sc[p][q] = 2.f * a.C44 * ec[p][q];
#pragma unroll
    for (int p = 0; p < 3; ++p) sc[p][p] = (a.C11 - a.C12) * ec[p][p] + a.C12 * tr;
    // s = R sc R^T
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) tmp[p][q] = sc[p][0] * R[q][0] + sc[p][1] * R[q][1] + sc[p][2] * R[q][2];
    float s[3][3];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) s[p][q] = R[p][0] * tmp[0][q] + R[p][1] * tmp[1][q] + R[p][2] * tmp[2][q];
    s_out[0] = s[0][0]; s_out[1] = s[1][1]; s_out[2] = s[2][2];
    s_out[3] = s[1][2]; s_out[4] = s[0][2]; s_out[5] = s[0][1];
}

// eps^hat = -Gamma0 : tau^hat at frequency (kx, ky, kz), six components in place
// (E N at 0, zero on the Nyquist planes of y and z; that of x is not kept)
__device__ __forceinline__ void green(const ElArgs& a, int kx, int ky, int kz, float2* t) {
    if ((kx | ky | kz) == 0) {
#pragma unroll
        for (int c = 0; c < 6; ++c) t[c] = make_float2(a.E[c] * (float)a.N, 0.f);
        return;
    }
    if ((a.ny > 1 && ky == -a.ny / 2) || (a.nz > 1 && kz == -a.nz / 2)) {
#pragma unroll
        for (int c = 0; c < 6; ++c) t[c] = make_float2(0.f, 0.f);
        return;
    }
    const float inv = rsqrtf((float)kx * kx + (float)ky * ky + (float)kz * kz);
    const float n[3] = {kx * inv, ky * inv, kz * inv};
    // a = tau n (complex), tau symmetric: rows (xx xy xz), (xy yy yz), (xz yz zz)
    const float2 av[3] = {
        make_float2(t[0].x * n[0] + t[5].x * n[1] + t[4].x * n[2], t[0].y * n[0] + t[5].y * n[1] + t[4].y * n[2]),
        make_float2(t[5].x * n[0] + t[1].x * n[1] + t[3].x * n[2], t[5].y * n[0] + t[1].y * n[1] + t[3].y * n[2]),
        make_float2(t[4].x * n[0] + t[3].x * n[1] + t[2].x * n[2], t[4].y * n[0] + t[3].y * n[1] + t[2].y * n[2])};
    const float2 cc = make_float2(n[0] * av[0].x + n[1] * av[1].x + n[2] * av[2].x,
                                  n[0] * av[0].y + n[1] * av[1].y + n[2] * av[2].y);
    const float h = 0.5f / a.mu0, kap = (a.lam0 + a.mu0) / (a.mu0 * (a.lam0 + 2.f * a.mu0));
    const int I[6] = {0, 1, 2, 1, 0, 0}, J[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const int p = I[c], q = J[c];
        t[c].x = -(h * (n[p] * av[q].x + av[p].x * n[q]) - kap * cc.x * n[p] * n[q]);
        t[c].y = -(h * (n[p] * av[q].y + av[p].y * n[q]) - kap * cc.y * n[p] * n[q]);
    }
}

// Forward along z, Green operator, inverse along z.  A thread keeps its eight
// points of all six components in registers (96), so that the operator, which
// mixes the components of one frequency, needs no exchange.  ONE: a line to a block, for
// grids of fewer columns than a block has lines: the others' threads would only lengthen
// every exchange (1 x 1 x 1024, six iterations: 375 -> 298 us).
template <int LOGN, bool ONE>
__global__ void __launch_bounds__(ZCfg<LOGN, ONE>::threads, 512 / ZCfg<LOGN, ONE>::threads)
    k_el_z(const __grid_constant__ ElArgs a, float2* __restrict__ data) {
    using C = ZCfg<LOGN, ONE>;
    constexpr int n = C::n, W = C::W, E = Line<LOGN>::E, T = Line<LOGN>::T;
    extern __shared__ __align__(16) float2 esm[];
    float2* tw = esm + 2 * C::buf;
    fill_twiddles<n>(tw, C::threads);
    const int w = threadIdx.x % W, t = threadIdx.x / W;
    const int64_t plane = (int64_t)a.nxh * a.ny, L = (int64_t)blockIdx.x * W + w;
    const bool on = L < plane;
    float2* p = data + L + (int64_t)t * plane;
    const int64_t st = (int64_t)T * plane;
    float2 v[6][E];
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int s = 0; s < E; ++s) v[c][s] = on ? p[c * a.Nh + s * st] : make_float2(0.f, 0.f);
    __syncthreads();
    XBlock<W, n, 2> x{esm, w, esm + C::buf};
#pragma unroll
    for (int c = 0; c < 6; ++c) fft_from<LOGN, -1, 1, 0>(v[c], t, tw, x);
    const int kx = (int)(L % a.nxh), y = (int)(L / a.nxh), ky = y < (a.ny + 1) / 2 ? y : y - a.ny;
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int z = t + s * T, kz = z < (n + 1) / 2 ? z : z - n;
        float2 f[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) f[c] = v[c][s];
        green(a, kx, ky, kz, f);
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c][s] = f[c];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        fft_from<LOGN, 1, 1, 0>(v[c], t, tw, x);
        if (on)
#pragma unroll
            for (int s = 0; s < E; ++s) p[c * a.Nh + s * st] = v[c][s];
    }
}

// The x pass.  A block takes whole lines of x, 16 voxels (eight pairs) a thread;
// the six real components of its voxels meet in shared memory between the inverse
// and the forward transform, where they are updated voxel by voxel.  A line's
// threads lie in one warp up to nx = 512, so its exchanges need no block barrier.
constexpr int kXT = 128;
template <int LOGNX>
struct XCfg {
    static constexpr int nx = 1 << LOGNX, LOGM = LOGNX > 0 ? LOGNX - 1 : 0, m = 1 << LOGM;  // pairs (kx kept) per line
    static constexpr int E = Line<LOGM>::E, T = Line<LOGM>::T, lines = kXT / T, vox = lines * nx;
    static constexpr int padded = m + m / 8;
    static constexpr size_t smem = sizeof(float2) * ((size_t)lines * padded + nx) + sizeof(float) * 6 * (size_t)vox;
};
template <int LOGNX>
struct XLine {
    float2* sm;  // this line's
    __device__ __forceinline__ static int at(int i) { return i + (i >> 3); }
    __device__ __forceinline__ void put(int i, float2 v) { sm[at(i)] = v; }
    __device__ __forceinline__ float2 get(int i) const { return sm[at(i)]; }
    __device__ __forceinline__ void wait() {
        if (XCfg<LOGNX>::T > 32) __syncthreads(); else __syncwarp();
    }
    __device__ __forceinline__ void done() { wait(); }
};

// INV: inverse transform and strain update (with the largest change, and the stress
// when a.sigma is set); FWD: polarisation of the strain and forward transform.
template <int LOGNX, bool INV, bool FWD>
__global__ void __launch_bounds__(kXT) k_el_x(const __grid_constant__ ElArgs a, float2* __restrict__ data) {
    using C = XCfg<LOGNX>;
    constexpr int nx = C::nx, m = C::m, E = C::E, T = C::T, LOGM = C::LOGM;
    extern __shared__ __align__(16) float2 esm[];
    float2* tw = esm + C::lines * C::padded;                       // exp(-2 pi i k / nx)
    float* f = reinterpret_cast<float*>(tw + nx);                  // [6][voxels of the block]
    const int w = threadIdx.x / T, t = threadIdx.x % T;
    const int64_t nl = (int64_t)a.ny * a.nz, l0 = (int64_t)blockIdx.x * C::lines, l = l0 + w;
    const bool on = l < nl;
    fill_twiddles<nx>(tw, kXT);
    XLine<LOGNX> x{esm + w * C::padded};
    float2* p = data + l * m + t;
    __syncthreads();
    if (INV) {
        float2 nxt[E];
#pragma unroll
        for (int s = 0; s < E; ++s) nxt[s] = on ? p[s * T] : make_float2(0.f, 0.f);
#pragma unroll 1
        for (int c = 0; c < 6; ++c) {
            float2 v[E];
#pragma unroll
            for (int s = 0; s < E; ++s) v[s] = nxt[s];
            if (c < 5)
#pragma unroll
                for (int s = 0; s < E; ++s) nxt[s] = on ? p[(c + 1) * a.Nh + s * T] : make_float2(0.f, 0.f);
            if (LOGNX > 0) {
                // Z_k = (X_k + conj X_{m-k}) + i exp(2 pi i k / nx) (X_k - conj X_{m-k}); X_m = 0, X_0 real
                if (t == 0) v[0].y = 0.f;
                if (m > 1) {
#pragma unroll
                    for (int s = 0; s < E; ++s) x.put(t + s * T, v[s]);
                    x.wait();
                }
#pragma unroll
                for (int s = 0; s < E; ++s) {
                    const int k = t + s * T;
                    float2 o = make_float2(0.f, 0.f);
                    if (m > 1 && k) o = x.get(m - k);
                    o.y = -o.y;
                    const float2 d = cmuli<1>(ctw<1>(csub(v[s], o), tw[k]));
                    v[s] = cadd(cadd(v[s], o), d);
                }
                if (m > 1) x.done();
                fft_from<LOGM, 1, 2, 0>(v, t, tw, x);
#pragma unroll
                for (int s = 0; s < E; ++s)
                    *reinterpret_cast<float2*>(f + c * C::vox + w * nx + 2 * (t + s * T)) = v[s];
            } else {
                f[c * C::vox + w] = v[0].x;
            }
        }
        __syncthreads();
    }
    // ---- voxels: update, change, stress or polarisation ------------------------
    // Four voxels of a thread at a time, everything they read fetched first (the
    // strain is overwritten in place, so no later read may pass an earlier write).
    constexpr int U = C::vox / kXT < 4 ? C::vox / kXT : 4;
    float big = 0.f;
    const int64_t v0 = l0 * nx;
    const int count = (int)(nl - l0 < C::lines ? (nl - l0) * nx : C::vox);
    const float invN = 1.0f / (float)a.N;
    const bool need = FWD || a.sigma;
    for (int k0 = threadIdx.x; k0 < count; k0 += U * kXT) {
        float e[U][6], ep[U][6], qq[U][4];
        int32_t gr[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = v0 + min(k0 + u * kXT, count - 1);
            gr[u] = need ? __ldg(a.grain + i) : 0;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                e[u][c] = a.mean ? a.E[c] : __ldcg(a.eps + (int64_t)c * a.N + i);
                ep[u][c] = need && a.eps_p ? __ldg(a.eps_p + (int64_t)c * a.N + i) : 0.f;
            }
        }
        if (need)
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int c = 0; c < 4; ++c) qq[u][c] = __ldg(a.quat + 4 * (int64_t)gr[u] + c);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = k0 + u * kXT;
            const int64_t i = v0 + k;
            if (k >= count) break;
            if (INV)
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    const float v = f[c * C::vox + k] * invN;
                    big = fmaxf(big, fabsf(v - e[u][c]));
                    e[u][c] = v;
                    a.eps[(int64_t)c * a.N + i] = v;
                }
            if (!need) continue;
            float s[6];
            crystal_stress(a, qq[u], ep[u], e[u], s);
            if (FWD) {
                const float tr = e[u][0] + e[u][1] + e[u][2];
#pragma unroll
                for (int c = 0; c < 6; ++c)
                    f[c * C::vox + k] = s[c] - 2.f * a.mu0 * e[u][c] - (c < 3 ? a.lam0 * tr : 0.f);
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) a.sigma[(int64_t)c * a.N + i] = s[c];
            }
        }
    }
    if (INV) {
#pragma unroll
        for (int o = 16; o; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xFFFFFFFFu, big, o));
        // one atomic per warp, and only while it would raise the maximum
        if ((threadIdx.x & 31) == 0 && __float_as_uint(big) > *(volatile unsigned*)a.change)
            atomicMax(a.change, __float_as_uint(big));
    }
    if (FWD) {
        __syncthreads();
#pragma unroll 1
        for (int c = 0; c < 6; ++c) {
            float2 v[E];
            if (LOGNX > 0) {
#pragma unroll
                for (int s = 0; s < E; ++s)
                    v[s] = on ? *reinterpret_cast<const float2*>(f + c * C::vox + w * nx + 2 * (t + s * T)) : make_float2(0.f, 0.f);
                fft_from<LOGM, -1, 2, 0>(v, t, tw, x);
                // X_k = (Z_k + conj Z_{m-k}) / 2 - i exp(-2 pi i k / nx) (Z_k - conj Z_{m-k}) / 2; Z_m = Z_0
                if (m > 1) {
#pragma unroll
                    for (int s = 0; s < E; ++s) x.put(t + s * T, v[s]);
                    x.wait();
                }
#pragma unroll
                for (int s = 0; s < E; ++s) {
                    const int k = t + s * T;
                    float2 o = m > 1 ? x.get((m - k) & (m - 1)) : v[s];
                    o.y = -o.y;
                    const float2 d = cmuli<-1>(ctw<-1>(csub(v[s], o), tw[k]));
                    const float2 sum = cadd(cadd(v[s], o), d);
                    v[s] = make_float2(0.5f * sum.x, 0.5f * sum.y);
                }
                if (m > 1) x.done();
            } else {
                v[0] = make_float2(on ? f[c * C::vox + w] : 0.f, 0.f);
            }
            if (on)
#pragma unroll
                for (int s = 0; s < E; ++s) p[c * a.Nh + s * T] = v[s];
        }
    }
}

__global__ void k_el_stress(ElArgs a, const float* __restrict__ eps, float* __restrict__ sig) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    float e[6], ep[6], s[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        e[c] = eps[(int64_t)c * a.N + i];
        ep[c] = a.eps_p ? a.eps_p[(int64_t)c * a.N + i] : 0.f;
    }
    crystal_stress(a, a.quat + 4 * (int64_t)a.grain[i], ep, e, s);
#pragma unroll
    for (int c = 0; c < 6; ++c) sig[(int64_t)c * a.N + i] = s[c];
}

int log2_exact(int n) {
    int l = 0;
    while ((1 << l) < n) ++l;
    return (1 << l) == n ? l : -1;
}

// Raise a kernel's dynamic shared memory limit (every call: the limit belongs to the
// current device) and launch it.
template <class K, class... A>
int launch_dyn(K kernel, const char* what, int64_t grid, int threads, size_t smem, cudaStream_t s, A... args) {
    if (smem > 48 * 1024) HP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    count_launch();
    kernel<<<(unsigned)grid, threads, smem, s>>>(args...);
    HP_LAUNCH_CHECK(what);
    return HP_OK;
}

// Call f with the compile-time logarithm of a power-of-two edge (1 .. 1024).
template <class F>
int with_log(int n, F f) {
    switch (log2_exact(n)) {
        case 0: return f(std::integral_constant<int, 0>());
        case 1: return f(std::integral_constant<int, 1>());
        case 2: return f(std::integral_constant<int, 2>());
        case 3: return f(std::integral_constant<int, 3>());
        case 4: return f(std::integral_constant<int, 4>());
        case 5: return f(std::integral_constant<int, 5>());
        case 6: return f(std::integral_constant<int, 6>());
        case 7: return f(std::integral_constant<int, 7>());
        case 8: return f(std::integral_constant<int, 8>());
        case 9: return f(std::integral_constant<int, 9>());
        default: return f(std::integral_constant<int, 10>());
    }
}

template <bool INV, bool FWD>
int x_pass(const ElArgs& a, float2* W, cudaStream_t s) {
    return with_log(a.nx, [&](auto lg) {
        using C = XCfg<decltype(lg)::value>;
        const int64_t grid = ((int64_t)a.ny * a.nz + C::lines - 1) / C::lines;
        return launch_dyn(k_el_x<decltype(lg)::value, INV, FWD>, "k_el_x", grid, kXT, C::smem, s, a, W);
    });
}

template <int DIR>
int y_pass(const ElArgs& a, float2* W, cudaStream_t s) {
    if (a.ny == 1) return HP_OK;
    return with_log(a.ny, [&](auto lg) {
        using C = YCfg<decltype(lg)::value>;
        const int64_t lines = 6 * (int64_t)a.nxh * a.nz;
        return launch_dyn(k_el_fft<decltype(lg)::value, DIR>, "k_el_fft", (lines + C::W - 1) / C::W, C::threads, C::smem, s,
                          W, a.nxh, lines);
    });
}

int z_pass(const ElArgs& a, float2* W, cudaStream_t s) {
    return with_log(a.nz, [&](auto lg) {
        constexpr int LOGN = decltype(lg)::value;
        using C = ZCfg<LOGN, false>;
        const int64_t lines = (int64_t)a.nxh * a.ny;
        if constexpr (LOGN >= 8)
            if (lines < C::W) {
                using D = ZCfg<LOGN, true>;
                return launch_dyn(k_el_z<LOGN, true>, "k_el_z", lines, D::threads, D::smem, s, a, W);
            }
        return launch_dyn(k_el_z<LOGN, false>, "k_el_z", (lines + C::W - 1) / C::W, C::threads, C::smem, s, a, W);
    });
}

}  // namespace
}  // namespace hp

using namespace hp;

extern "C" int hp_elastic_solve(const hp_cp_params* prm, const hp_elastic_params* ep, const int32_t* grain,
                                const float* quat, const float* eps_p, const double E[6], float* eps, float* sigma,
                                int32_t* iters, double* change_out, void* stream) {
    hp::Range r_("hp_elastic_solve");
    if (!prm || !ep || !grain || !quat || !E || !eps) return set_error(HP_ERR_ARG, "hp_elastic_solve: bad arguments");
    for (int d = 0; d < 3; ++d)
        if (ep->n[d] < 1 || ep->n[d] > 1024 || log2_exact(ep->n[d]) < 0)
            return set_error(HP_ERR_ARG, "hp_elastic_solve: grid edges must be powers of two up to 1024");
    if (!(ep->tol > 0.0) || ep->max_iter < 1) return set_error(HP_ERR_ARG, "hp_elastic_solve: bad tolerance");
    cudaStream_t s = as_stream(stream);
    ElArgs a;
    a.nx = ep->n[0]; a.ny = ep->n[1]; a.nz = ep->n[2];
    a.N = (int64_t)a.nx * a.ny * a.nz;
    a.C11 = (float)prm->C11; a.C12 = (float)prm->C12; a.C44 = (float)prm->C44;
    // isotropic reference: the mean of the two shear moduli, the crystal's bulk modulus
    const double mu0 = 0.5 * (prm->C44 + 0.5 * (prm->C11 - prm->C12));
    const double K = (prm->C11 + 2.0 * prm->C12) / 3.0;
    a.mu0 = (float)mu0;
    a.lam0 = (float)(K - 2.0 * mu0 / 3.0);
    a.grain = grain; a.quat = quat; a.eps_p = eps_p;
    double emax = 0.0;
    for (int c = 0; c < 6; ++c) {
        a.E[c] = (float)E[c];
        emax = fabs(E[c]) > emax ? fabs(E[c]) : emax;
    }
    if (!(emax > 0.0)) return set_error(HP_ERR_ARG, "hp_elastic_solve: zero mean strain");
    a.nxh = a.nx > 1 ? a.nx / 2 : 1;
    a.Nh = (int64_t)a.nxh * a.ny * a.nz;
    a.eps = eps;
    a.sigma = nullptr;
    a.mean = ep->start_from_mean ? 1 : 0;
    float2* W = nullptr;
    unsigned* d_change = nullptr;
    if (cudaMallocAsync((void**)&W, sizeof(float2) * 6 * (size_t)a.Nh, s) != cudaSuccess ||
        cudaMallocAsync((void**)&d_change, sizeof(unsigned), s) != cudaSuccess) {
        cudaFreeAsync(W, s);
        cudaFreeAsync(d_change, s);
        return set_error(HP_ERR_OOM, "hp_elastic_solve: work buffer allocation failed");
    }
    a.change = d_change;
    int it = 0;
    double ch = INFINITY;
    // an update starts the next iteration on its way out (polarisation, transform
    // along x) unless it is the last one allowed, which writes the stress instead
    int rc = x_pass<false, true>(a, W, s);
    bool have_sigma = false;
    for (it = 1; it <= ep->max_iter && rc == HP_OK; ++it) {
        if ((rc = y_pass<-1>(a, W, s)) || (rc = z_pass(a, W, s)) || (rc = y_pass<1>(a, W, s))) break;
        cudaMemsetAsync(d_change, 0, sizeof(unsigned), s);
        if (it < ep->max_iter) {
            rc = x_pass<true, true>(a, W, s);
        } else {
            a.sigma = sigma;
            have_sigma = true;
            rc = x_pass<true, false>(a, W, s);
        }
        if (rc) break;
        a.mean = 0;
        unsigned hc = 0;
        cudaError_t e = cudaMemcpyAsync(&hc, d_change, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { rc = cuda_error(e, "hp_elastic_solve"); break; }
        float hf;
        memcpy(&hf, &hc, sizeof hf);
        ch = (double)hf / emax;
        if (ch < ep->tol) break;
    }
    if (it > ep->max_iter) it = ep->max_iter;
    if (rc == HP_OK && sigma && !have_sigma) {
        count_launch();
        k_el_stress<<<(unsigned)((a.N + kET - 1) / kET), kET, 0, s>>>(a, eps, sigma);
    }
    if (rc == HP_OK) {
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_error(e, "hp_elastic_solve");
    }
    cudaFreeAsync(W, s);
    cudaFreeAsync(d_change, s);
    if (iters) *iters = it;
    if (change_out) *change_out = ch;
    return rc;
}
