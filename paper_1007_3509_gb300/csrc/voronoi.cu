// Initial polycrystal: Voronoi tessellation of G seeds on the periodic lattice
// and per-grain orientations (the set-up of the polycrystal runs, Sec. 4-5).
//
// Seeds: in round a every unplaced seed g draws site floor(u0 * N / 2^32) from
// Philox(seed; g, a, tag 2 | 0).  A site drawn by several seeds in one round
// goes to the lowest g; a site owned since an earlier round stays with its
// owner; losers redraw in round a+1.  The q buffer doubles as the claim array
// (free = 0x7F7F7F7F, tentative claim = g, placed = -1 - g).
//
// Assignment: each site takes the seed at the smallest periodic minimum-image
// squared distance, ties to the lowest index.  Seeds are bucketed into a grid
// of cells (about two seeds per cell); any seed outside the cells within Chebyshev
// radius r of a set of cells is at least r * wmin + 1 (wmin = narrowest cell width)
// away from every site in them.
//
// A block takes a brick of sites (k_assign_bricks).  With D(s) the largest distance
// of seed s to any site of the brick, no site of it is further than U = min D(s)
// from its nearest seed, so only seeds whose least distance to the brick is at most
// U can be anyone's; rings of cells are added until U is below the bound above.
// Every warp narrows the brick's list down in the same way to its runs of 32
// adjacent sites, and its lanes then compare a handful of seeds each.  What bounds
// it: integer instructions; the scan of the 27 cells around every site that it
// replaces (54 seeds, 64-bit distances) took about 6000 per site.
#include <math.h>


#include "common.cuh"
#include "reach.h"

namespace hp {
namespace {

constexpr int kT = 256;

__global__ void k_seed_claim(int32_t* claim, const int64_t* pos, int32_t G, uint64_t seed, uint32_t round,
                             int64_t N) {
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G || pos[g] >= 0) return;
    const uint4 u = draw(seed, (uint64_t)g, round, kTagVoronoi, 0);
    const int64_t s = (int64_t)(((uint64_t)u.x * (uint64_t)N) >> 32);
    atomicMin(claim + s, g);
}

__global__ void k_seed_resolve(int32_t* claim, int64_t* pos, int32_t G, uint64_t seed, uint32_t round, int64_t N,
                               int32_t* n_left) {
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G || pos[g] >= 0) return;
    const uint4 u = draw(seed, (uint64_t)g, round, kTagVoronoi, 0);
    const int64_t s = (int64_t)(((uint64_t)u.x * (uint64_t)N) >> 32);
    if (claim[s] == g) {
        pos[g] = s;
        claim[s] = -1 - g;
    } else {
        atomicAdd(n_left, 1);
    }
}

struct Cells {
    int L[3];
    int nc[3];
    int wmin;
    int dim;
};

__device__ __forceinline__ int cell_of(int x, int L, int nc) { return (int)(((int64_t)x * nc) / L); }

__global__ void k_cell_count(const int64_t* pos, int32_t G, Cells c, int32_t* cnt, int4* xyz) {
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    const int64_t p = pos[g];
    const int x = (int)(p % c.L[0]);
    const int y = (int)((p / c.L[0]) % c.L[1]);
    const int z = (int)(p / ((int64_t)c.L[0] * c.L[1]));
    const int cid = cell_of(x, c.L[0], c.nc[0]) + c.nc[0] * (cell_of(y, c.L[1], c.nc[1]) + c.nc[1] * cell_of(z, c.L[2], c.nc[2]));
    xyz[g] = make_int4(x, y, z, cid);
    atomicAdd(cnt + cid, 1);
}

// exclusive scan of n ints by one block (n is at most a few million)
__global__ void k_scan(const int32_t* in, int32_t* out, int32_t n) {
    __shared__ int32_t part[1024];
    const int t = threadIdx.x;
    const int per = (n + 1023) / 1024;
    const int b = t * per, e = min(n, b + per);
    int32_t s = 0;
    for (int i = b; i < e; ++i) s += in[i];
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const int32_t v = t >= off ? part[t - off] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int32_t run = t ? part[t - 1] : 0;
    for (int i = b; i < e; ++i) {
        out[i] = run;
        run += in[i];
    }
    if (t == 1023) out[n] = part[1023];
}

__global__ void k_cell_scatter(const int4* xyz, int32_t G, const int32_t* start, int32_t* cursor, int4* list) {
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    const int4 v = xyz[g];
    const int32_t k = atomicAdd(cursor + v.w, 1);
    list[start[v.w] + k] = make_int4(v.x, v.y, v.z, g);
}

__device__ __forceinline__ int64_t mi(int d, int L) {
    d = d < 0 ? -d : d;
    return (int64_t)(d < L - d ? d : L - d);
}

__device__ __forceinline__ int wrapc(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}

// Nearest seed of one site by its own rings of cells: for lattices that are not
// assigned by bricks, and for a brick with more seeds nearby than its list holds.
__device__ __noinline__ int32_t assign_site(int x, int y, int z, const Cells& c, const int32_t* start, const int4* list) {
    const int cx = cell_of(x, c.L[0], c.nc[0]), cy = cell_of(y, c.L[1], c.nc[1]), cz = cell_of(z, c.L[2], c.nc[2]);
    int64_t best = INT64_MAX;
    int32_t arg = INT32_MAX;
    for (int r = 0;; ++r) {
        const int rz = c.dim == 3 ? r : 0;
        for (int dz = -rz; dz <= rz; ++dz) {
            for (int dy = -r; dy <= r; ++dy) {
                const bool face = (dz == -rz || dz == rz) && c.dim == 3;
                const bool yface = dy == -r || dy == r;
                // on an inner row only the two end cells belong to the ring
                const int step = (face || yface) ? 1 : (r > 0 ? 2 * r : 1);
                for (int dx = -r; dx <= r; dx += step) {
                    const int ccx = wrapc(cx + dx, c.nc[0]), ccy = wrapc(cy + dy, c.nc[1]), ccz = wrapc(cz + dz, c.nc[2]);
                    const int cid = ccx + c.nc[0] * (ccy + c.nc[1] * ccz);
                    const int b = start[cid], e = start[cid + 1];
                    for (int k = b; k < e; ++k) {
                        const int4 s = list[k];
                        const int64_t ddx = mi(x - s.x, c.L[0]), ddy = mi(y - s.y, c.L[1]), ddz = mi(z - s.z, c.L[2]);
                        const int64_t d2 = ddx * ddx + ddy * ddy + ddz * ddz;
                        if (d2 < best || (d2 == best && s.w < arg)) {
                            best = d2;
                            arg = s.w;
                        }
                    }
                }
            }
        }
        const int64_t bound = (int64_t)r * c.wmin + 1;
        const bool all = (2 * r + 1 >= c.nc[0]) && (2 * r + 1 >= c.nc[1]) && (c.dim == 2 || 2 * r + 1 >= c.nc[2]);
        if ((arg != INT32_MAX && best < bound * bound) || all) break;
    }
    return arg;
}

__global__ void __launch_bounds__(kT) k_assign(int32_t* q, int32_t* mp, int64_t N, Cells c, const int32_t* start,
                                               const int4* list) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int x = (int)(i % c.L[0]);
    const int y = (int)((i / c.L[0]) % c.L[1]);
    const int z = (int)(i / ((int64_t)c.L[0] * c.L[1]));
    q[i] = assign_site(x, y, z, c, start, list);
    if (mp) mp[i] = (int32_t)i;
}

struct Box {
    int b[3], len[3];
};
// squared least and largest distances of seed s to the box
__device__ __forceinline__ Reach reach2(const int4 s, const Box& k, const Cells& c) {
    const Reach x = reach(s.x, k.b[0], k.len[0], c.L[0]), y = reach(s.y, k.b[1], k.len[1], c.L[1]),
                z = reach(s.z, k.b[2], k.len[2], c.L[2]);
    return Reach{x.lo * x.lo + y.lo * y.lo + z.lo * z.lo, x.hi * x.hi + y.hi * y.hi + z.hi * z.hi};
}

// Bricks of 32 x 8 x 8 sites (2D: 64 x 32), one warp run 8 x 4 x 2 (8 x 8), two sites
// to a lane: compact, for a short list, and 32 bytes of a row, for whole sectors.
// kNear seeds per brick and kRun per run; beyond, a run tests the brick's list and a
// brick its sites' own rings.  256^3, 16000 seeds, whole call: 3.1 ms with the rings
// per site, 0.34 ms with bricks (0.45 ms while a run's upper bound exceeded the largest
// distance by its length and some 25 seeds of a run's list stood for six).
constexpr int kRun = 64;

template <int DIM>
struct Brick {
    static constexpr int X = DIM == 3 ? kBrick3[0] : kBrick2[0], Y = DIM == 3 ? kBrick3[1] : kBrick2[1],
                         Z = DIM == 3 ? kBrick3[2] : kBrick2[2];
    static constexpr int RX = 8, RY = DIM == 3 ? 4 : 8, RZ = DIM == 3 ? 2 : 1;  // lanes: 8 x 4, twice (in z; in y)
    static constexpr int NX = X / RX, NY = Y / RY, RUNS = NX * NY * (Z / RZ);
};

// The runs of a brick.  NEAR: the brick's seeds are given by the image closest to it,
// which is the closest to each of its sites (the brick and its reach span no more than
// half of any axis); otherwise every distance is folded.
template <int DIM, bool NEAR>
__device__ __forceinline__ void brick_runs(const Box& k, const Cells& c, const int4* near_, int n, int4* run,
                                           int32_t* __restrict__ q, int32_t* __restrict__ mp) {
    using B = Brick<DIM>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int t = warp; t < B::RUNS; t += kT / 32) {
        Box m;
        m.b[0] = k.b[0] + (t % B::NX) * B::RX;
        m.b[1] = k.b[1] + (t / B::NX % B::NY) * B::RY;
        m.b[2] = k.b[2] + (t / (B::NX * B::NY)) * B::RZ;
        if (m.b[0] >= c.L[0] || m.b[1] >= c.L[1] || m.b[2] >= c.L[2]) continue;
        const int full[3] = {B::RX, B::RY, B::RZ};
#pragma unroll
        for (int d = 0; d < 3; ++d) m.len[d] = min(full[d], c.L[d] - m.b[d]) - 1;
        auto reach_of = [&](const int4 s) {
            if (!NEAR) return reach2(s, m, c);
            const int sd[3] = {s.x, s.y, s.z};
            Reach r{0, 0};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (DIM == 2 && d == 2) continue;
                const Reach a = reach_near(sd[d], m.b[d], m.len[d]);
                r.lo += a.lo * a.lo;
                r.hi += a.hi * a.hi;
            }
            return r;
        };
        // the first 64 seeds stay in registers between the two looks at them
        int lo0 = INT32_MAX, lo1 = INT32_MAX, best = INT32_MAX;
        if (lane < n) {
            const Reach r = reach_of(near_[lane]);
            lo0 = r.lo;
            best = r.hi;
        }
        if (lane + 32 < n) {
            const Reach r = reach_of(near_[lane + 32]);
            lo1 = r.lo;
            best = min(best, r.hi);
        }
        for (int i = lane + 64; i < n; i += 32) best = min(best, reach_of(near_[i]).hi);
        best = __reduce_min_sync(0xFFFFFFFFu, best);
        int nr = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            int lo = i0 == 0 ? lo0 : lo1;
            if (i0 >= 64) lo = i < n ? reach_of(near_[i]).lo : INT32_MAX;
            const bool keep = lo <= best && i < n;
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
            const int at = nr + __popc(bal & lt);
            if (keep && at < kRun) run[at] = near_[i];
            nr += __popc(bal);
        }
        __syncwarp();
        const int4* src = nr <= kRun ? run : near_;
        const int ns = nr <= kRun ? nr : n;
        // lane's sites (x, y, z) and one further along z (3D) or four along y (2D)
        const int x = m.b[0] + (lane & 7), y = m.b[1] + (lane >> 3), z = m.b[2];
        const int y1 = DIM == 3 ? y : y + 4, z1 = DIM == 3 ? z + 1 : z;
        int d0 = INT32_MAX, d1 = INT32_MAX, g0 = INT32_MAX, g1 = INT32_MAX;
        for (int i = 0; i < ns; ++i) {
            const int4 s = src[i];
            int dx = x - s.x, dy = y - s.y, dz = z - s.z, ey = y1 - s.y, ez = z1 - s.z;
            if (!NEAR) {
                dx = abs(dx); dy = abs(dy); dz = abs(dz); ey = abs(ey); ez = abs(ez);
                dx = min(dx, c.L[0] - dx);
                dy = min(dy, c.L[1] - dy);
                dz = min(dz, c.L[2] - dz);
                ey = min(ey, c.L[1] - ey);
                ez = min(ez, c.L[2] - ez);
            }
            const int a = dx * dx + (DIM == 3 ? dy * dy : 0), u = a + (DIM == 3 ? dz * dz : dy * dy),
                      v = a + (DIM == 3 ? ez * ez : ey * ey);
            if (u < d0 || (u == d0 && s.w < g0)) { d0 = u; g0 = s.w; }
            if (v < d1 || (v == d1 && s.w < g1)) { d1 = v; g1 = s.w; }
        }
        __syncwarp();
        if (x < c.L[0] && y < c.L[1]) {
            const int64_t i = x + (int64_t)c.L[0] * (y + (int64_t)c.L[1] * z);
            q[i] = g0;
            if (mp) mp[i] = (int32_t)i;
        }
        if (x < c.L[0] && y1 < c.L[1] && z1 < c.L[2]) {
            const int64_t i = x + (int64_t)c.L[0] * (y1 + (int64_t)c.L[1] * z1);
            q[i] = g1;
            if (mp) mp[i] = (int32_t)i;
        }
    }
}

template <int DIM>
__global__ void __launch_bounds__(kT) k_assign_bricks(int32_t* __restrict__ q, int32_t* __restrict__ mp,
                                                      const __grid_constant__ Cells c,
                                                      const int32_t* __restrict__ start, const int4* __restrict__ list,
                                                      int nbx, int nby) {
    using B = Brick<DIM>;
    __shared__ int4 near_[kNear];
    __shared__ int4 run[kT / 32][kRun];
    __shared__ int s_best, s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bx = (int)(blockIdx.x % (unsigned)nbx), br = (int)(blockIdx.x / (unsigned)nbx);
    Box k;
    k.b[0] = bx * B::X;
    k.b[1] = (br % nby) * B::Y;
    k.b[2] = (br / nby) * B::Z;
    const int ext[3] = {B::X, B::Y, B::Z};
    int c0[3], nc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        k.len[d] = min(ext[d], c.L[d] - k.b[d]) - 1;
        c0[d] = cell_of(k.b[d], c.L[d], c.nc[d]);
        nc[d] = cell_of(k.b[d] + k.len[d], c.L[d], c.nc[d]) - c0[d] + 1;
    }
    // seeds of the cells within radius r of the brick's, by rows of cells along x (one
    // or, across the edge, two runs of the list): f(seed) for every one of them
    auto scan = [&](int r, auto f) {
        int n[3], f0[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int rr = d == 2 && DIM == 2 ? 0 : r;
            n[d] = min(nc[d] + 2 * rr, c.nc[d]);
            f0[d] = n[d] == c.nc[d] ? 0 : c0[d] - rr;  // rr < nc: at most one period below 0
            f0[d] += f0[d] < 0 ? c.nc[d] : 0;
        }
        const int first = min(n[0], c.nc[0] - f0[0]);  // cells before the edge
        for (int row = warp; row < n[1] * n[2]; row += kT / 32) {
            const int rz = DIM == 3 ? (int)((unsigned)row / (unsigned)n[1]) : 0;
            int cy = f0[1] + row - rz * n[1], cz = f0[2] + rz;
            cy -= cy >= c.nc[1] ? c.nc[1] : 0;
            cz -= cz >= c.nc[2] ? c.nc[2] : 0;
            const int32_t* st = start + (int64_t)c.nc[0] * (cy + (int64_t)c.nc[1] * cz);
            int s0 = st[f0[0]], s1 = st[f0[0] + first];
            for (int i = s0 + lane; i < s1; i += 32) f(list[i]);
            if (first < n[0]) {
                s0 = st[0];
                s1 = st[n[0] - first];
                for (int i = s0 + lane; i < s1; i += 32) f(list[i]);
            }
        }
        return n[0] == c.nc[0] && n[1] == c.nc[1] && n[2] == c.nc[2];
    };
    if (tid == 0) {
        s_best = INT32_MAX;
        s_n = 0;
    }
    __syncthreads();
    int r = 1, far2;
    for (;; ++r) {
        int best = INT32_MAX;
        const bool all = scan(r, [&](const int4 s) { best = min(best, reach2(s, k, c).hi); });
        best = __reduce_min_sync(0xFFFFFFFFu, best);
        if (lane == 0) atomicMin(&s_best, best);
        __syncthreads();
        far2 = s_best;
        const int64_t bound = (int64_t)r * c.wmin + 1;
        if (all || (int64_t)far2 < bound * bound) break;
        __syncthreads();
    }
    // no distance looked at below exceeds U + the brick's length, U = sqrt(far2)
    const int U = (int)sqrtf((float)far2) + 2;
    bool near = true;
#pragma unroll
    for (int d = 0; d < DIM; ++d) near &= U + k.len[d] <= c.L[d] / 2;
    scan(r, [&](int4 s) {
        if (reach2(s, k, c).lo > far2) return;
        if (near) {  // the image closest to the brick
            int* sd[3] = {&s.x, &s.y, &s.z};
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                int u = *sd[d] - k.b[d];
                u += u < 0 ? c.L[d] : 0;
                *sd[d] = k.b[d] + (u > k.len[d] && u - k.len[d] > c.L[d] - u ? u - c.L[d] : u);
            }
        }
        const int i = atomicAdd(&s_n, 1);
        if (i < kNear) near_[i] = s;
    });
    __syncthreads();
    const int n = s_n;
    if (n <= kNear) {
        if (near) brick_runs<DIM, true>(k, c, near_, n, run[warp], q, mp);
        else brick_runs<DIM, false>(k, c, near_, n, run[warp], q, mp);
        return;
    }
    for (int t = tid; t < B::X * B::Y * B::Z; t += kT) {
        const int x = k.b[0] + t % B::X, y = k.b[1] + t / B::X % B::Y, z = k.b[2] + t / (B::X * B::Y);
        if (x >= c.L[0] || y >= c.L[1] || z >= c.L[2]) continue;
        const int64_t i = x + (int64_t)c.L[0] * (y + (int64_t)c.L[1] * z);
        q[i] = assign_site(x, y, z, c, start, list);
        if (mp) mp[i] = (int32_t)i;
    }
}

// Bricks or single sites, see assign_by_bricks.
void launch_assign(int32_t* q, int32_t* mp, int64_t N, const Cells& c, int32_t G, const int32_t* start, const int4* list,
                   cudaStream_t s) {
    ::hp::count_launch();
    if (!assign_by_bricks(c.dim, c.L, G)) {
        k_assign<<<(unsigned)((N + kT - 1) / kT), kT, 0, s>>>(q, mp, N, c, start, list);
    } else if (c.dim == 3) {
        using B = Brick<3>;
        const int nx = (c.L[0] + B::X - 1) / B::X, ny = (c.L[1] + B::Y - 1) / B::Y, nz = (c.L[2] + B::Z - 1) / B::Z;
        k_assign_bricks<3><<<(unsigned)nx * ny * nz, kT, 0, s>>>(q, mp, c, start, list, nx, ny);
    } else {
        using B = Brick<2>;
        const int nx = (c.L[0] + B::X - 1) / B::X, ny = (c.L[1] + B::Y - 1) / B::Y;
        k_assign_bricks<2><<<(unsigned)nx * ny, kT, 0, s>>>(q, mp, c, start, list, nx, ny);
    }
}

__global__ void k_orient(int32_t G, uint64_t seed, int32_t kind, float* out) {
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    const uint4 u = draw(seed, (uint64_t)g, 0, kTagVoronoi, 1);
    const double two32 = 4294967296.0, pi = 3.14159265358979323846;
    if (kind == HP_ORIENT_ANGLE) {
        out[g] = (float)(((double)u.x / two32) * (pi / 2.0));
    } else if (kind == HP_ORIENT_ZROT) {
        const double t = ((double)u.x / two32) * (pi / 2.0);
        double sh, ch;
        sincos(0.5 * t, &sh, &ch);
        out[4 * g + 0] = (float)ch;
        out[4 * g + 1] = 0.0f;
        out[4 * g + 2] = 0.0f;
        out[4 * g + 3] = (float)sh;
    } else {
        const double u1 = (double)u.x / two32, u2 = (double)u.y / two32, u3 = (double)u.z / two32;
        const double a = sqrt(1.0 - u1), b = sqrt(u1);
        double s2, c2, s3, c3;
        sincos(2.0 * pi * u2, &s2, &c2);
        sincos(2.0 * pi * u3, &s3, &c3);
        out[4 * g + 0] = (float)(a * s2);
        out[4 * g + 1] = (float)(a * c2);
        out[4 * g + 2] = (float)(b * s3);
        out[4 * g + 3] = (float)(b * c3);
    }
}

}  // namespace

int orientations_run(int32_t G, uint64_t seed, int32_t kind, float* orient, cudaStream_t s) {
    if (G < 1 || !orient || kind < HP_ORIENT_ANGLE || kind > HP_ORIENT_ZROT)
        return set_error(HP_ERR_ARG, "hp_orientations: bad arguments");
    ::hp::count_launch();
    k_orient<<<(G + kT - 1) / kT, kT, 0, s>>>(G, seed, kind, orient);
    HP_LAUNCH_CHECK("k_orient");
    return HP_OK;
}

int voronoi_run(hp_handle* h, int32_t orient_kind, float* orient, int64_t* seed_pos, cudaStream_t s) {
    const int32_t G = h->desc.n_grains;
    const int64_t N = h->lat.N;
    if (G < 1 || G > N) return set_error(HP_ERR_ARG, "hp_init_voronoi: need 1 <= G <= N");
    if (N >= (int64_t)1 << 32) return set_error(HP_ERR_ARG, "hp_init_voronoi: lattice too large (N >= 2^32)");
    // scratch: seed positions, per-seed coordinates, cell arrays
    Cells c;
    c.dim = h->lat.dim;
    for (int d = 0; d < 3; ++d) c.L[d] = (int)h->lat.L[d];
    const double per = pow(2.0 * (double)N / (double)G, 1.0 / c.dim);  // cell edge for ~2 seeds per cell
    int64_t ncell = 1;
    c.wmin = INT32_MAX;
    for (int d = 0; d < 3; ++d) {
        if (d >= c.dim) { c.nc[d] = 1; continue; }
        int n = (int)floor((double)c.L[d] / per);
        n = n < 1 ? 1 : n;
        c.nc[d] = n;
        ncell *= n;
        const int w = c.L[d] / n;  // narrowest cell width along d
        c.wmin = w < c.wmin ? w : c.wmin;
    }
    // one allocation, carved (seven of them cost more than the kernels of a small call)
    size_t bytes = 0;
    auto take = [&](size_t n) { const size_t at = bytes; bytes += (n + 255) & ~(size_t)255; return at; };
    const size_t o_xyz = take(sizeof(int4) * G), o_list = take(sizeof(int4) * G), o_cnt = take(sizeof(int32_t) * ncell),
                 o_start = take(sizeof(int32_t) * (ncell + 1)), o_cursor = take(sizeof(int32_t) * ncell),
                 o_left = take(sizeof(int32_t)), o_pos = take(seed_pos ? 0 : sizeof(int64_t) * G);
    unsigned char* buf = nullptr;
    cudaError_t e = cudaMallocAsync((void**)&buf, bytes, s);
    auto cleanup = [&]() { cudaFreeAsync(buf, s); };
    if (e != cudaSuccess) return set_error(HP_ERR_OOM, "hp_init_voronoi: scratch allocation failed");
    int64_t* pos = seed_pos ? seed_pos : (int64_t*)(buf + o_pos);
    int4 *xyz = (int4*)(buf + o_xyz), *list = (int4*)(buf + o_list);
    int32_t *cnt = (int32_t*)(buf + o_cnt), *start = (int32_t*)(buf + o_start), *cursor = (int32_t*)(buf + o_cursor),
            *n_left = (int32_t*)(buf + o_left);

    int rc = HP_OK;
    do {
        if ((e = cudaMemsetAsync(h->q, 0x7F, sizeof(int32_t) * N, s))) break;
        if ((e = cudaMemsetAsync(pos, 0xFF, sizeof(int64_t) * G, s))) break;
        const int gb = (G + kT - 1) / kT;
        for (uint32_t round = 0;; ++round) {
            if ((e = cudaMemsetAsync(n_left, 0, sizeof(int32_t), s))) break;
            ::hp::count_launch();
            k_seed_claim<<<gb, kT, 0, s>>>(h->q, pos, G, h->desc.seed, round, N);
            ::hp::count_launch();
            k_seed_resolve<<<gb, kT, 0, s>>>(h->q, pos, G, h->desc.seed, round, N, n_left);
            int32_t left = 0;
            if ((e = cudaMemcpyAsync(&left, n_left, sizeof(int32_t), cudaMemcpyDeviceToHost, s))) break;
            if ((e = cudaStreamSynchronize(s))) break;
            if (left == 0) break;
            if (round > (1u << 20)) { rc = set_error(HP_ERR_STATE, "hp_init_voronoi: seeding did not converge"); break; }
        }
        if (e || rc) break;
        if ((e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * ncell, s))) break;
        if ((e = cudaMemsetAsync(cursor, 0, sizeof(int32_t) * ncell, s))) break;
        ::hp::count_launch();
        k_cell_count<<<gb, kT, 0, s>>>(pos, G, c, cnt, xyz);
        ::hp::count_launch();
        k_scan<<<1, 1024, 0, s>>>(cnt, start, (int32_t)ncell);
        ::hp::count_launch();
        k_cell_scatter<<<gb, kT, 0, s>>>(xyz, G, start, cursor, list);
        launch_assign(h->q, h->mp, N, c, G, start, list, s);
        if ((e = cudaGetLastError())) break;
        if (orient) {
            ::hp::count_launch();
            k_orient<<<gb, kT, 0, s>>>(G, h->desc.seed, orient_kind, orient);
            if ((e = cudaGetLastError())) break;
        }
    } while (0);
    cleanup();
    if (e) return cuda_error(e, "hp_init_voronoi");
    return rc;
}

}  // namespace hp

// ---------------------------------------------------------------------------
// Voronoi initialisation without any device allocation.
//
// For callers that cannot allocate device memory while they run -- e.g. a
// process whose device memory is entirely pre-reserved by another allocator,
// or a steady-state loop that must never enter cudaMalloc/cudaFree -- the
// scratch of the tessellation (seed coordinates, cell lists, cell counters,
// the round counter) lives in one file-scope device array of fixed size.
// The array exists on every GPU that loads this library, until exit.
// ---------------------------------------------------------------------------
namespace hp {
namespace {

constexpr size_t kStaticScratchBytes = (size_t)HP_VORONOI_STATIC_BYTES;
static __device__ __align__(256) unsigned char g_vor_scratch[kStaticScratchBytes];

// Worst case of the carve below at HP_VORONOI_STATIC_MAX_GRAINS on a square or
// cubic lattice: int64 seed sites (8 G), int4 seed coordinates and the int4
// cell list (16 G each), and three int32 cell arrays of at most G/2 + 1 cells
// (the cell edge is (2N/G)^(1/dim)), each carve rounded up to 256 bytes.
// Thin lattices whose cell count rounds up past G/2 are caught at run time.
static_assert((size_t)HP_VORONOI_STATIC_MAX_GRAINS * (8 + 16 + 16) +
                      3 * ((size_t)HP_VORONOI_STATIC_MAX_GRAINS / 2 + 2) * 4 + 7 * 256 <=
                  kStaticScratchBytes,
              "static Voronoi scratch too small for HP_VORONOI_STATIC_MAX_GRAINS");

// Device address of the static scratch on the current device.  The array's
// name is only a host-side stand-in; its device address comes from
// cudaGetSymbolAddress, taken on every call with the caller's device current
// (nothing is cached, so a context torn down and created again between calls
// never leaves a stale address behind).
int static_scratch(void** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_vor_scratch);
    if (e != cudaSuccess) return cuda_error(e, "hp_init_voronoi_static: cudaGetSymbolAddress");
    *out = p;
    return HP_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace
}  // namespace hp

extern "C" int hp_init_voronoi_static(hp_handle* h, int32_t orient_kind, float* orient, int64_t* seed_pos,
                                      void* stream) {
    using namespace hp;
    if (!h) return set_error(HP_ERR_ARG, "hp_init_voronoi_static: null handle");
    if (!h->q) return set_error(HP_ERR_STATE, "hp_init_voronoi_static: no lattice bound");
    if (orient && (orient_kind < HP_ORIENT_ANGLE || orient_kind > HP_ORIENT_ZROT))
        return set_error(HP_ERR_ARG, "hp_init_voronoi_static: bad orient_kind");
    const int32_t G = h->desc.n_grains;
    const int64_t N = h->lat.N;
    if (G < 1 || G > N) return set_error(HP_ERR_ARG, "hp_init_voronoi_static: need 1 <= G <= N");
    if (G > HP_VORONOI_STATIC_MAX_GRAINS)
        return set_error(HP_ERR_ARG, "hp_init_voronoi_static: more grains than the static scratch holds "
                                     "(HP_VORONOI_STATIC_MAX_GRAINS); use hp_init_voronoi");
    if (N >= (int64_t)1 << 32) return set_error(HP_ERR_ARG, "hp_init_voronoi_static: lattice too large (N >= 2^32)");
    cudaStream_t s = as_stream(stream);
    Cells c;
    c.dim = h->lat.dim;
    for (int d = 0; d < 3; ++d) c.L[d] = (int)h->lat.L[d];
    const double per = pow(2.0 * (double)N / (double)G, 1.0 / c.dim);
    int64_t ncell = 1;
    c.wmin = INT32_MAX;
    for (int d = 0; d < 3; ++d) {
        if (d >= c.dim) { c.nc[d] = 1; continue; }
        int n = (int)floor((double)c.L[d] / per);
        n = n < 1 ? 1 : n;
        c.nc[d] = n;
        ncell *= n;
        const int w = c.L[d] / n;
        c.wmin = w < c.wmin ? w : c.wmin;
    }
    // carve the static scratch
    void* base = nullptr;
    int rc = static_scratch(&base);
    if (rc) return rc;
    size_t off = 0;
    auto take = [&](size_t bytes) { void* p = (unsigned char*)base + off; off += align256(bytes); return p; };
    int64_t* pos = seed_pos ? seed_pos : (int64_t*)take(sizeof(int64_t) * G);
    int4* xyz = (int4*)take(sizeof(int4) * G);
    int4* list = (int4*)take(sizeof(int4) * G);
    int32_t* cnt = (int32_t*)take(sizeof(int32_t) * ncell);
    int32_t* start = (int32_t*)take(sizeof(int32_t) * (ncell + 1));
    int32_t* cursor = (int32_t*)take(sizeof(int32_t) * ncell);
    int32_t* n_left = (int32_t*)take(sizeof(int32_t));
    if (off > kStaticScratchBytes)
        return set_error(HP_ERR_ARG, "hp_init_voronoi_static: scratch layout exceeds the static array");

    // everything that must start at zero (or -1) is cleared here on every call
    HP_CUDA(cudaMemsetAsync(h->q, 0x7F, sizeof(int32_t) * N, s));
    HP_CUDA(cudaMemsetAsync(pos, 0xFF, sizeof(int64_t) * G, s));
    const int gb = (G + kT - 1) / kT;
    for (uint32_t round = 0;; ++round) {
        HP_CUDA(cudaMemsetAsync(n_left, 0, sizeof(int32_t), s));
        ::hp::count_launch();
        k_seed_claim<<<gb, kT, 0, s>>>(h->q, pos, G, h->desc.seed, round, N);
        ::hp::count_launch();
        k_seed_resolve<<<gb, kT, 0, s>>>(h->q, pos, G, h->desc.seed, round, N, n_left);
        int32_t left = 0;
        HP_CUDA(cudaMemcpyAsync(&left, n_left, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        HP_CUDA(cudaStreamSynchronize(s));
        if (left == 0) break;
        if (round > (1u << 20)) return set_error(HP_ERR_STATE, "hp_init_voronoi_static: seeding did not converge");
    }
    HP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * ncell, s));
    HP_CUDA(cudaMemsetAsync(cursor, 0, sizeof(int32_t) * ncell, s));
    ::hp::count_launch();
    k_cell_count<<<gb, kT, 0, s>>>(pos, G, c, cnt, xyz);
    ::hp::count_launch();
    k_scan<<<1, 1024, 0, s>>>(cnt, start, (int32_t)ncell);
    ::hp::count_launch();
    k_cell_scatter<<<gb, kT, 0, s>>>(xyz, G, start, cursor, list);
    launch_assign(h->q, h->mp, N, c, G, start, list, s);
    if (orient) {
        ::hp::count_launch();
        k_orient<<<gb, kT, 0, s>>>(G, h->desc.seed, orient_kind, orient);
    }
    HP_LAUNCH_CHECK("hp_init_voronoi_static");
    return HP_OK;
}
