// Distances of a Voronoi seed to a box of sites, one axis at a time (voronoi.cu).
// Plain C++ as well as device code, so that the bounds can be checked on the host.
#pragma once

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

}  // namespace hp
