// Rules that choose among kernels and their splits by size and shape, and the geometry
// that they need.  Plain C++ as well as device code, so that they can be checked on the host.
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
// So is a second wave of four-warp windows that comes to no more than a third of the
// first (`wave`: how many an SM holds; 0 with material points, where it does not pay):
// ensembles of 200-site grains, 64^3, 128^3 and 64^3 (1344 windows) 67.0 -> 55.9, 2 x 96^3
// and 2 x 64^3 (1152) 55.3 -> 49.8, 160^3 (1440) 59.5 -> 58.0, but 8 x 64^3 (1536) 59.3 ->
// 64.1.
inline int lean_warps(int64_t windows, int wave = 0) {
    if (windows <= 3 * kSMs) return 8;
    const int64_t first = (int64_t)wave * kSMs;
    return windows > first && 100 * windows <= 136 * first ? 8 : 4;
}

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

// 2D lattices that the per-colour kernel sweeps faster than the tiles: chained launches of
// one site a thread against a window's fill and halo.  us per MCS, per colour / tiles, 50
// and 500 sites a grain:
//  * 4 neighbours, two launches: 256^2 3.8 and 3.8 / 8.4 and 6.8, 700^2 5.9 and 5.7 / 8.5
//    and 6.9, with material points 6.6 and 6.4 / 11.0 and 9.3, 1500^2 18.0 and 17.5 / 15.3
//    and 11.1; with misorientation tables 300^2 9.4 and 7.5 / 13.0 and 9.0, 360^2 11.5 and
//    10.0 / 13.0 and 9.0;
//  * 8 neighbours, four launches: lattices that the cluster kernel would take but for
//    their long strips (one_resident): 2000 x 30 7.3 / 8.0, 64 x 1000 7.2 / 12.4;
//  * lattices narrower than a window of 128 columns, which goes through theirs twice and
//    more: 4 neighbours 16 x 60000 7.1 / 33.1, 126 x 8000 9.2 / 14.7, with tables 16 x 8000
//    8.9 and 6.7 / 21.8 and 15.9, 100 x 4000 12.1 and 11.2 / 17.9 and 13.2; 8 neighbours up
//    to 64 columns, 16 x 60000 11.4 / 38.6, 64 x 20000 15.3 / 21.0, with tables 16 x 60000
//    36.5 and 24.6 / 181 and 90, but 100 x 4000 32.3 and 23.0 / 31.2 and 19.4.
inline bool per_colour_2d(int nbr, int64_t Lx, int64_t N, bool tables, bool hasmp) {
    if (nbr == 4) return Lx < 128 || N < (tables ? 100000 : (int64_t)1 << 19);
    return Lx <= 64 || (!tables && !hasmp && N <= 65536);
}

// ---- Resident 2D sweep (res2d.cu): one thread-block cluster per lattice ---------------
// CTAs per cluster, from `cs` down: at least eight rows a strip.
inline int res_cluster(int cs, int64_t Ly) {
    while (cs > 1 && Ly < 8 * cs) cs /= 2;
    return cs;
}
// Strips: row pairs are dealt out as evenly as they go, the first ones larger.
HP_HD int strip_rows(int Ly, int cs, int r) {
    const int pairs = Ly / 2;
    return 2 * (pairs / cs + (r < pairs % cs ? 1 : 0));
}
// Lines of a strip that are worked at the same time (8 neighbours: row pairs), and the
// lines each warp of at most 32 goes through.
HP_HD int strip_lines(int nbr, int rows) { return nbr == 8 ? rows / 2 : rows; }
inline int lines_per_warp(int lines) { return (lines + 31) / 32; }

// Estimated us per MCS of one lattice on its cluster, `sharing` CTAs to an SM: the
// barriers, a chain per line of a warp and pass over 128 columns, and the instructions
// of all passes of the SM.  Fitted to lattices of 50-site grains at kT = 1, 64^2 to 600^2
// and 16 x 2000 to 2048 x 64: within 15 % (some coarse ones run 10 % below it).
inline double res_us(int nbr, int64_t Lx, int64_t Ly, int cs, int sharing = 1) {
    const int lines = strip_lines(nbr, strip_rows((int)Ly, cs, 0)), passes = (int)((Lx + 127) / 128);
    const int chain = lines_per_warp(lines) * (1 + passes), work = lines * passes * sharing;
    return nbr == 8 ? 1.0 + chain + 0.11 * work : 1.3 + 0.3 * chain + 0.07 * work;
}

// One lattice on its cluster?  Against the per-colour kernel's 3.7 us per MCS (4
// neighbours, two launches) and 7.2 to 7.4 us (8 neighbours, four) on lattices of this
// size: 4 neighbours by the passes of a strip, 8 neighbours by the estimate.  Per MCS on
// the cluster / per colour: 4 neighbours 128^2 (16 passes) 2.9 / 3.7, 190 x 86 (24) 3.4 /
// 3.6, 128 x 200 (26) 3.8 / 3.6, 120 x 240 4.3 / 3.6, 512 x 32 4.3 / 3.6, 2048 x 8 12.0 /
// 3.6; 8 neighbours 256^2 6.8 / 7.3, 512 x 64 6.9 / 7.3, 128 x 500 7.3 / 7.3, 512 x 128
// 7.9 / 7.4, 300 x 200 8.6 / 7.3, 64 x 1000 12.7 / 7.2, 2000 x 30 25.1 / 7.3, 16 x 4000
// 33.1 / 7.2.
inline bool one_resident(int nbr, int64_t Lx, int64_t Ly, int cs) {
    if (nbr == 4) return strip_rows((int)Ly, cs, 0) * (int)((Lx + 127) / 128) <= 24;
    return res_us(nbr, Lx, Ly, cs) <= 8.0;
}

// An ensemble's launches of short tiles, us per MCS: a floor (longer where a window is
// wider than a lattice) and so much per tile, a fifth more where a window is not fetched
// by bulk copies.  `built`: the field mode has these tiles; the plane kernel otherwise.
struct TileCost {
    double tiles = 0.0;
    bool narrow = false;
    void add(int64_t Lx, int64_t Ly) {
        const bool slow = Lx % 4 != 0 || Lx < 128 || Ly < 32;
        tiles += (double)tiles_2d(Lx, Ly, 28) * (slow ? 1.2 : 1.0);
        narrow = narrow || Lx < 128;
    }
    double us(int nbr, bool built) const {
        const double floor = (built ? (nbr == 8 ? 12.0 : 11.2) : (nbr == 8 ? 24.0 : 22.0)) * (narrow ? 1.4 : 1.0);
        const double t = built ? (nbr == 8 ? 6.0 + 0.024 * tiles : 5.0 + 0.0192 * tiles)
                               : (nbr == 8 ? 15.0 + 0.029 * tiles : 12.0 + 0.026 * tiles);
        return t > floor ? t : floor;
    }
};

// ---- Grain counts (field.cu) ---------------------------------------------------------------
// Sites that a warp goes through, 128 at a step: 2048 where the chip is full of warps
// anyhow (64 an SM), down to 128 where they are few and each step is a wait for memory.
// hp_measure, us, 2048 sites throughout / now / 32 sites a thread: 500^2 77 / 65 / 74,
// 250^2 62 / 52 / 61, 64^2 54 / 44 / 58.
inline int counts_seg(int64_t N) {
    int seg = 128;
    while (seg < 2048 && N > (int64_t)seg * 64 * kSMs) seg *= 2;
    return seg;
}

}  // namespace hp
