// Rules that choose among the sweep kernels by size and shape, and the geometry that
// they need.  Plain C++ as well as device code, so that they can be checked on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define HP_HD __host__ __device__ __forceinline__
#else
#define HP_HD inline
#endif

namespace hp {

constexpr int kSMs = 152;

// Warps of a 64 x 32 window of the 26-neighbour kernel (lean.cu), by the windows of
// the launch: eight up to three windows an SM, where material points are carried and in
// the launches of an ensemble, which are not chained.  Such a launch is a chain of
// latencies -- draws, proposals, the gathers of a test -- and with twice the warps each
// goes through half as many rows; with more windows in flight the instructions count,
// and four warps issue fewer.  us per MCS, point field, four warps -> eight: 44 x 76 x 32
// (96 windows) 27.0 -> 18.6, 76 x 64 x 40 22.8 -> 15.8, 112^3 (448) 29.4 -> 23.4, but
// 128 x 128 x 64 (480) 30.0 -> 32.5; ensembles of two 48^3, grain field 22.4 -> 15.2.
inline int lean_warps(int64_t windows) { return windows <= 3 * kSMs ? 8 : 4; }

// ---- 2D tiles (tile.cu): cores of 120 x 28 (variant 3) and 120 x 60 (variant 4) ------
inline int64_t tiles_2d(int64_t Lx, int64_t Ly, int core) { return ((Lx + 119) / 120) * ((Ly + core - 1) / core); }

// One lattice on the tall tiles rather than the short ones?  The short ones have the
// shorter chain per launch, but once they come in two waves the tall ones, half as many,
// still come in one.  8 neighbours: five short tiles an SM.  us per MCS, short / tall:
// 1502^2 (702 tiles) 19.6 / 21.0, 1602 x 1700 (854) 27.0 / 21.2, 1600 x 1700 18.7 /
// 18.0, 2046 x 1500 27.7 / 23.1, 2400^2 31.3 / 29.0.  4 neighbours: six an SM, and the
// short tiles' second wave is the cheaper one where rows come in 16-byte pieces (1800^2
// 15.9 / 15.3, 2048^2 18.2 / 25.0, 4096^2 60.2 / 65.4), not where each element is
// fetched by itself (1702^2 23.3 / 20.9, 1922 x 1960 26.7 / 23.2; 722 x 3600, one wave,
// 17.9 / 20.9).  With material points the short ones up to 2^22 sites.
inline bool tall_tiles(int nbr, int64_t Lx, int64_t Ly, bool hasmp) {
    if (hasmp) return nbr == 8 && Lx * Ly >= (int64_t)1 << 22;
    if (nbr == 8) return tiles_2d(Lx, Ly, 28) > 5 * kSMs;
    return Lx % 4 != 0 && tiles_2d(Lx, Ly, 28) > 6 * kSMs && tiles_2d(Lx, Ly, 60) <= 4 * kSMs;
}

}  // namespace hp
