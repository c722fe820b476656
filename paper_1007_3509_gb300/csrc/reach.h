// Distances of a Voronoi seed to a box of sites, one axis at a time, and the rule that
// says which lattices are assigned by boxes (voronoi.cu).  Plain C++ as well as device
// code, so that both can be checked on the host.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define HP_HD __host__ __device__ __forceinline__
#else
#define HP_HD inline
#endif

namespace hp {

// least and largest distance of a seed to the sites of a box
struct Reach {
    int lo, hi;
};

// Along a periodic axis of (even, or 1) length L: coordinate s against the interval
// [b, b + len], len < L.
HP_HD Reach reach(int s, int b, int len, int L) {
    int u = s - b;
    u += u < 0 ? L : 0;  // 0 <= u < L
    const int v = u > len ? u - len : len - u;
    int h = u + (L >> 1);
    h -= h >= L ? L : 0;  // offset of the point opposite to s
    const int au = u < L - u ? u : L - u, av = v < L - v ? v : L - v, below = u - len < L - u ? u - len : L - u;
    Reach r;
    r.lo = u <= len ? 0 : below;
    r.hi = h <= len ? L >> 1 : (au > av ? au : av);
    return r;
}

// The same for a coordinate already moved to the image that is closest to every
// site of the interval.
HP_HD Reach reach_near(int s, int b, int len) {
    const int u = b - s, v = s - b - len;  // past either end where positive
    const int out = u > v ? u : v, in = u < v ? u : v;
    return Reach{out > 0 ? out : 0, -in};
}

// Bricks of the assignment, and the seeds that a brick's list holds.
constexpr int kBrick3[3] = {32, 8, 8}, kBrick2[3] = {64, 32, 1};
constexpr int kNear = 1024;

struct BrickLists {
    double seeds;    // expected length of a brick's list (3D: 10 to 20 % high)
    bool near;       // every seed of it has one image closest to the whole brick
    int64_t bricks;
};
// G seeds at random on the lattice: those within U of a brick, U the least over the
// seeds of the largest distance to it -- half its diagonal and a part of the spacing.
inline BrickLists brick_lists(int dim, const int* L, int64_t G) {
    const int* ext = dim == 3 ? kBrick3 : kBrick2;
    double N = 1.0, half = 0.0;
    BrickLists r{0.0, true, 1};
    for (int d = 0; d < dim; ++d) {
        const double e = ext[d] < L[d] ? ext[d] : L[d];
        N *= L[d];
        half += 0.25 * e * e;
        r.bricks *= (L[d] + ext[d] - 1) / ext[d];
    }
    const double U = sqrt(half) + 0.35 * pow(N / (double)G, 1.0 / dim);
    // the brick grown by U on all sides; an axis that it wraps counts whole
    double a[3], whole = 1.0, vol = 1.0;
    int n = 0;
    for (int d = 0; d < dim; ++d) {
        const double e = ext[d] < L[d] ? ext[d] : L[d];
        r.near = r.near && U + e <= 0.5 * L[d];
        if (e + 2.0 * U >= L[d]) whole *= L[d];
        else a[n++] = e;
    }
    const double pi = 3.14159265358979323846;
    if (n == 1) vol = a[0] + 2.0 * U;
    if (n == 2) vol = a[0] * a[1] + 2.0 * (a[0] + a[1]) * U + pi * U * U;
    if (n == 3)
        vol = a[0] * a[1] * a[2] + 2.0 * (a[0] * a[1] + a[1] * a[2] + a[0] * a[2]) * U + pi * (a[0] + a[1] + a[2]) * U * U +
              4.0 / 3.0 * pi * U * U * U;
    r.seeds = vol * whole * (double)G / N;
    return r;
}

// Bricks where their lists fit and pay; single sites where grains are so small that a
// list would overflow (its brick is then scanned site by site, by one block), or long
// against what the chip has to do otherwise, and on axes whose squared distances do
// not fit 32 bits.  us per call, single sites -> bricks: 128^3, 110 sites a grain 557
// -> 344, 80 sites 577 -> 670, 8 sites 859 -> 1668; 1024^2, 14 sites 286 -> 276, 12
// sites 320 -> 372.  Folded distances (a brick's reach past half an axis) cost some 2.5
// times as much per seed: 512 x 512 x 8, 32 sites 650 -> 486, 24 sites 695 -> 965.  A
// few bricks leave the chip idle: 30^3 (16 bricks), 80 sites 115 -> 116, 48 sites
// 115 -> 161; 48^3 (72), 110 sites 131 -> 128, 90 sites 128 -> 164.
inline bool assign_by_bricks(int dim, const int* L, int64_t G) {
    for (int d = 0; d < dim; ++d)
        if (L[d] > 32768) return false;
    const BrickLists b = brick_lists(dim, L, G);
    double most = b.near || b.bricks < 512 ? (double)kNear : 700.0;
    if (250.0 + 8.0 * (double)b.bricks < most) most = 250.0 + 8.0 * (double)b.bricks;
    return b.seeds <= most;
}

}  // namespace hp
