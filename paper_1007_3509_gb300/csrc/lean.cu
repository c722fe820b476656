// Lean 3D kernel of the fused checkerboard sweep (Eq. (7), Sec. 4) for the
// 26-neighbour simple cubic lattice, built to spend few instructions per
// site-update and to keep a warp from waiting for others.
//
// Colours c = (x&1) + 2(y&1) + 4(z&1): one MCS is two launches, the even planes
// (colours 0-3, their z-neighbours the odd planes as they were) and then the odd
// planes (colours 4-7, their z-neighbours the even planes as just updated).  One
// CTA = one 64 x WY window of one plane: q of the plane and of its two
// z-neighbours and, with material points, mp of the plane.  The window keeps a
// halo of four columns and two rows on each side (the exact region of the four
// in-plane phases, as in the 2D Moore tiles), so the core is (64 - 8) x (WY - 4).
//
// What the kernel is bound by: instructions and the latency of the few dependent
// loads of a test, not memory.  What keeps both down:
//  * every random number of the launch is drawn while the window is in flight and
//    stays in registers (lane = column of the colour sub-grid);
//  * there is no interior test: a site proposes its k-th neighbour's grain, and
//    only proposals of another grain (about a fifth of the sites in a
//    polycrystal) are tested;
//  * a warp owns whole rows.  Phases 0 and 1 (even rows) see the odd rows only as
//    they arrived, and phases 2 and 3 the even rows only as phases 0 and 1 left
//    them, so a warp queues and tests its own proposals phase after phase with no
//    more than warp-level synchronisation; the block meets once, between phases 1
//    and 2.  A block-wide queue (two block barriers per phase, half of the warps
//    idle in every test) spent 3.7 of 10 stall cycles per instruction there;
//  * four warps of WY / 8 row pairs each: about 28 of the 128 sites a warp looks
//    at per phase go on to its test, one per lane, so a pass runs nearly full.
//    With eight warps (14 proposals, two lanes to each) the same window took 66 %
//    more instructions and 138 us where this takes 100.  A launch of few windows
//    waits rather than issues and takes eight (lean_warps);
//  * the neighbour planes' material points are gathered for the proposals that
//    point there instead of being staged: 37 KB of shared memory a block, six
//    blocks on an SM (staged, 53 KB and four).
// Measured on 512^3 (two launches per MCS), site-updates/s: point field 7.9e10 ->
// 9.2e10, grain field 1.10e11 -> 1.25e11; 512 x 512 x 64, one launch, ncu: 113.6
// -> 100.7 us and 10.0 -> 7.7 warp instructions per site-update with the point
// field, 87.2 -> 77.8 us with the grain field.
#include <string.h>

#include <cudaTypedefs.h>

#include "routes.h"
#include "sweep.cuh"

namespace hp {
namespace {

__device__ int g_lean_err;

// Tiled TMA descriptors of the launch's source arrays (3D, Lx x Ly x Lz int32,
// box 64 x WY x 1); zeroed when a window is never copied by TMA.  `tab` maps a
// per-material-point field table laid out like the lattice (entry p belongs to
// the point that started at site p).
struct alignas(64) LeanMaps {
    CUtensorMap q_in, q_nb, mp_in, mp_nb, tab;
    int ok;   // 1: the q (and mp_in) descriptors are valid
    int pfm;  // 1: `mp_nb` is valid (the neighbour planes' material points are prefetched into L2)
    int pf;   // 1: `tab` is valid (the field table is prefetched into L2)
};

__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(mbar) : "memory");
}

// Bring one box of a mapped array into L2 (a hint: nothing lands in shared
// memory and nothing is waited for).
__device__ __forceinline__ void tma_prefetch_l2(const CUtensorMap* map, int x, int y, int z) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z) : "memory");
}


template <int WY, int FIELD, bool HASMP, int NW_ = 4>
struct LeanCfg {
    static constexpr int NW = NW_, kLT = 32 * NW;
    static constexpr int WX = 64, HX = 4, HY = 2, TX = WX - 2 * HX, TY = WY - 2 * HY;
    static constexpr int PS = WX * WY;             // one plane window, sites
    static constexpr int NA = HASMP ? 4 : 3;       // window arrays: q(z-1) q(z) q(z+1) [mp(z)]
    static constexpr int SX = WX / 2, SY = WY / 2;                   // one colour's sites in the window
    static constexpr int PER = (SY + NW - 1) / NW;                   // row pairs per warp
    static constexpr int CAP = 32 * PER;                             // sites of one colour per warp
    static_assert(SX == 32 && WY % 2 == 0 && TY % 2 == 0, "lean window shape");
    // 64 x 32 is the fastest on every lattice measured (512^3, point field: 5.83
    // ms for 4 MCS against 6.8, 7.0 and 7.5 ms of 36, 40 and 44 rows, whose row
    // pairs do not share out evenly among four warps)
    // shared memory: the window arrays | a proposal queue per warp | neighbour
    // offsets | mbarrier
    static constexpr size_t smem() { return 128 + 4 * (size_t)NA * PS + 8 * (size_t)(NW * CAP) + 4 * 28 + 8; }
    // blocks per SM that the shared memory allows (228 KB, 1 KB of it per block taken)
    static constexpr int FIT = (int)(228 * 1024 / (smem() + 1024));
    static constexpr int MINB = NW > 4 ? 3 : FIT > 7 ? 7 : FIT;
    __host__ __device__ static constexpr int ylo(int p) { return 1 + (p >> 1); }
};

// One block, nothing in flight: an mbarrier that expects one arrival, waited
// on by the whole block with a short limit.  With `late` the arrival comes from
// thread 32 after two limits (the first wait gives up, the drain sees it: flag
// 1); otherwise it never comes (the drain runs out as well: flag 2).
__global__ void k_wait_probe(long long limit, int late) {
    __shared__ unsigned long long bar;
    const uint32_t mb = s_addr(&bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (late && threadIdx.x == 32) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2 * limit) {
        }
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
    }
    wait_or_drain(mb, &g_lean_err, limit);
}

// a wrapped into [0, L), however far off (windows wider than the lattice)
__device__ __noinline__ int wrap_any(int a, int L) { return wrapi(a, L); }

// One window (tile `tile` of plane 2 zidx + a.zpar) of one lattice; maps NULL
// when no window of this launch is copied by TMA boxes.
template <int WY, int FIELD, bool HASMP, int NW>
struct Lean {
    using Cfg = LeanCfg<WY, FIELD, HASMP, NW>;
    static constexpr int WX = Cfg::WX, PS = Cfg::PS;
    const PlaneArgs& a;
    int32_t* Q;         // q of plane z (z-1 at -PS, z+1 at +PS)
    int32_t* MP;        // mp of plane z
    int x0, y0;
    uint32_t lobase, hibase;  // first site of planes z-1, z+1
    uint32_t tab_last;        // last index of the field table
    bool fast;    // the window fits the lattice
    bool inside;  // and does not cross its edge in x or y

    __device__ __forceinline__ Lean(const PlaneArgs& a_) : a(a_) {}
    __device__ __forceinline__ int gx_of(int col) const {
        int v = x0 - 4 + col;
        if (!inside) v = fast ? wrap1(v, a.Lx) : wrap_any(v, a.Lx);
        return v;
    }
    __device__ __forceinline__ int gy_of(int r) const {
        int v = y0 - 2 + r;
        if (!inside) v = fast ? wrap1(v, a.Ly) : wrap_any(v, a.Ly);
        return v;
    }
    // field table entry, the index clamped into the table
    __device__ __forceinline__ int32_t field(int32_t i) const { return __ldg(a.table + min((uint32_t)i, tab_last)); }
    // material point of the neighbour at offset o: of planes z-1 and z+1, which
    // this launch does not change, from global memory
    __device__ __forceinline__ int32_t mp_of(int pos, int o) const {
        if (o >= -(PS / 2) && o <= PS / 2) return MP[pos + o];
        const int n = pos + o + (o < 0 ? PS : -PS);
        return a.mp_nb[(o < 0 ? lobase : hibase) + (uint32_t)gx_of(n & (WX - 1)) +
                       (uint32_t)a.Lx * (uint32_t)gy_of(n / WX)];
    }
    // The Metropolis test of the proposal at pos (offset o, acceptance draw u1).
    __device__ __forceinline__ void test(int pos, int o, uint32_t u1) const {
        const int32_t* c = Q + pos;
        const int32_t qi = c[0], qj = c[o];
        int32_t mj = 0, bi = 0, bj = 0;
        if (HASMP) mj = mp_of(pos, o);
        if (FIELD) {
            bi = field(FIELD == 2 ? MP[pos] : qi);
            bj = field(FIELD == 2 ? mj : qj);
        }
        // all 27 sites of the neighbourhood: of each row the aligned pair with the
        // site's column and the column on its other side; the site itself counts
        // once among those of its own grain
        const int32_t* pr = Q + (pos & ~1);
        const int32_t* sg = c + ((pos & 1) ? 1 : -1);
        int ni[3] = {0, -1, 0}, nj[3] = {0, 0, 0};  // per plane: six short chains of adds
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dz = 0; dz < 3; ++dz) {
                const int2 v = *reinterpret_cast<const int2*>(pr + (dz - 1) * PS + dy * WX);
                const int32_t w = sg[(dz - 1) * PS + dy * WX];
                if (v.x == qi) ++ni[dz];
                if (v.x == qj) ++nj[dz];
                if (v.y == qi) ++ni[dz];
                if (v.y == qj) ++nj[dz];
                if (w == qi) ++ni[dz];
                if (w == qj) ++nj[dz];
            }
        const int dn = (ni[0] + ni[1] + ni[2]) - (nj[0] + nj[1] + nj[2]);
        if (metropolis(a.J * dn + (bj - bi), a.D, a.thr, u1)) {
            Q[pos] = qj;
            if (HASMP) MP[pos] = mj;
        }
    }
};

template <int WY, int FIELD, bool HASMP, int NW>
__device__ __forceinline__ void lean_body(const PlaneArgs& a, const LeanMaps* maps, const int tile, const int zidx,
                                          unsigned char* raw) {
    using L = Lean<WY, FIELD, HASMP, NW>;
    using Cfg = typename L::Cfg;
    constexpr int WX = Cfg::WX, PS = Cfg::PS, NA = Cfg::NA, PER = Cfg::PER, CAP = Cfg::CAP;
    constexpr int kLT = Cfg::kLT;
    constexpr bool EVEN = Cfg::SY % NW == 0;  // every warp has PER row pairs
    int32_t* base = reinterpret_cast<int32_t*>(raw + ((128u - (s_addr(raw) & 127u)) & 127u));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    L w(a);
    w.Q = base + PS;
    w.MP = base + 3 * PS;
    uint2* queue = reinterpret_cast<uint2*>(base + NA * PS) + CAP * warp;  // this warp's: pos | offset << 16, u1
    int* off = reinterpret_cast<int*>(base + NA * PS + 2 * CAP * NW);      // offset of neighbour k at [k + 1], 0 at [0]
    unsigned long long* mbar = reinterpret_cast<unsigned long long*>(off + 28);

    const int ty = tile / a.tiles_x, tx = tile - ty * a.tiles_x;
    w.x0 = tx * Cfg::TX;
    w.y0 = ty * Cfg::TY;
    const int x0 = w.x0, y0 = w.y0;
    const int z = 2 * zidx + a.zpar;
    const int zlo = z > 0 ? z - 1 : a.Lz - 1, zhi = z < a.Lz - 1 ? z + 1 : 0;
    const uint32_t sxy = (uint32_t)a.Lx * (uint32_t)a.Ly;
    const uint32_t zbase = sxy * (uint32_t)z;
    w.lobase = sxy * (uint32_t)zlo;
    w.hibase = sxy * (uint32_t)zhi;
    w.tab_last = a.table_n - 1u;
    w.fast = a.fast != 0;
    w.inside = x0 >= 4 && x0 - 4 + WX <= a.Lx && y0 >= 2 && y0 - 2 + WY <= a.Ly;

    // ---- window in flight ----------------------------------------------------
    // A window inside the lattice arrives as one tiled TMA box per array (64 x WY
    // of plane z, one request each, completing on an mbarrier that warp 0 polls).
    // A window that crosses the periodic edge is filled with asynchronous copies
    // issued by every thread, 16 bytes where rows keep 16-byte boundaries (Lx % 4
    // == 0) and 8 bytes otherwise (edges are even: x0 - 4 and Lx are multiples of
    // the chunk, so no chunk straddles the edge; 250 x 198 x 130 with material
    // points, 10 MCS: 3.28 ms with 4-byte loads and a modulo per coordinate, 1.20
    // ms with this kernel).  Either way the copies land while the draws below run.
    const uintptr_t low = (uintptr_t)a.q_in | (uintptr_t)a.q_nb | (HASMP ? (uintptr_t)a.mp_in : 0);
    const bool v16 = a.Lx % 4 == 0 && (low & 15u) == 0, v8 = !v16 && (low & 7u) == 0;
    const bool boxed = v16 && maps && maps->ok && w.inside;
    if (tid < 27) {
        const int k = tid - 1, kk = k + (k >= 13);
        off[tid] = tid ? (kk / 9 - 1) * PS + ((kk / 3) % 3 - 1) * WX + (kk % 3 - 1) : 0;
    }
    const bool chained = maps != nullptr, early = chained && chain_early();  // batched launches are not chained
    if (early) chain_open();
    if (chained) chain_wait();
    const uint32_t mb = s_addr(mbar);
    auto src = [&](int arr) -> const int32_t* {
        return arr == 0 ? a.q_nb + w.lobase : arr == 1 ? a.q_in + zbase : arr == 2 ? a.q_nb + w.hibase : a.mp_in + zbase;
    };
    if (boxed) {
        if (tid == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb),
                         "r"((uint32_t)(NA * PS * 4)) : "memory");
            const int xs = x0 - 4, ys = y0 - 2;
            tma_box(s_addr(base), &maps->q_nb, xs, ys, zlo, mb);
            tma_box(s_addr(base + PS), &maps->q_in, xs, ys, z, mb);
            tma_box(s_addr(base + 2 * PS), &maps->q_nb, xs, ys, zhi, mb);
            if (HASMP) tma_box(s_addr(base + 3 * PS), &maps->mp_in, xs, ys, z, mb);
            // The proposals look up the material points of the neighbour planes
            // and the field of the window's material points.  A point moves only a
            // few sites under grain growth, so most of them lie in the table's
            // boxes at the window's own coordinates: start these towards L2 now.
            if (HASMP && maps->pfm) {
                tma_prefetch_l2(&maps->mp_nb, xs, ys, zlo);
                tma_prefetch_l2(&maps->mp_nb, xs, ys, zhi);
            }
            if (FIELD == 2 && maps->pf) {
                tma_prefetch_l2(&maps->tab, xs, ys, zlo);
                tma_prefetch_l2(&maps->tab, xs, ys, z);
                tma_prefetch_l2(&maps->tab, xs, ys, zhi);
            }
        }
    } else if (v16) {
        const int c = 4 * (tid & 15), gx = w.gx_of(c);
#pragma unroll
        for (int r = tid >> 4; r < WY; r += kLT / 16) {
            const uint32_t g = (uint32_t)gx + (uint32_t)a.Lx * (uint32_t)w.gy_of(r);
#pragma unroll
            for (int arr = 0; arr < NA; ++arr)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s_addr(base + arr * PS + r * WX + c)),
                             "l"(src(arr) + g) : "memory");
        }
    } else if (v8) {
        const int c = 2 * lane, gx = w.gx_of(c);
        for (int r = warp; r < WY; r += NW) {
            const uint32_t g = (uint32_t)gx + (uint32_t)a.Lx * (uint32_t)w.gy_of(r);
#pragma unroll
            for (int arr = 0; arr < NA; ++arr)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s_addr(base + arr * PS + r * WX + c)),
                             "l"(src(arr) + g) : "memory");
        }
    } else {
        for (int i = tid; i < PS; i += kLT) {
            const uint32_t g = (uint32_t)w.gx_of(i & (WX - 1)) + (uint32_t)a.Lx * (uint32_t)w.gy_of(i / WX);
#pragma unroll
            for (int arr = 0; arr < NA; ++arr) base[arr * PS + i] = src(arr)[g];
        }
    }
    // every thread sees the barrier initialised (and the offsets) before it waits
    __syncthreads();

    // ---- every draw of the launch, while the copies land -------------------
    // Warp v owns the row pairs (2j, 2j + 1), j = v + NW m; lane = column of the
    // colour sub-grid, so that the lane's sites of the pair are the four window
    // positions (2 lane, 2 lane + 1) x (2j, 2j + 1), one of each phase.  A site's
    // Philox unit is a row base plus a column, each wrapped once per thread.
    // Whether the row lies in the phase's region is the same for the whole warp
    // (a branch); whether the column does is a select.  A slot without a site
    // gets choice 0 (offset 0): it proposes itself, which is no proposal.
    const uint32_t cz = 4u * (uint32_t)a.zpar;
    const uint32_t gxc[2] = {(uint32_t)w.gx_of(2 * lane), (uint32_t)w.gx_of(2 * lane + 1)};
    const int pos0 = 2 * warp * WX + 2 * lane;
    uint32_t u1[4][PER];
    uint32_t kk[2][PER];  // choices + 1 of phases 2r, 2r + 1 in bytes 0 and 1
#pragma unroll
    for (int m = 0; m < PER; ++m) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int y = 2 * (warp + NW * m) + r;
            kk[r][m] = 0;
            u1[2 * r][m] = u1[2 * r + 1][m] = 0;
            if (y >= Cfg::ylo(2 * r) && y < WY - Cfg::ylo(2 * r)) {
                const uint32_t rowb = zbase + (uint32_t)a.Lx * (uint32_t)w.gy_of(y);
#pragma unroll
                for (int px = 0; px < 2; ++px) {
                    const int p = 2 * r + px, x = 2 * lane + px;
                    const uint2 u = sweep_draw(a.key, rowb + gxc[px], cz + (uint32_t)p);
                    u1[p][m] = u.y;
                    kk[r][m] |= (x >= p + 1 && x < WX - p - 1 ? __umulhi(u.x, 26u) + 1u : 0u) << (8 * px);
                }
            }
        }
    }

    if (boxed) {
        if (!wait_or_drain(mb, &g_lean_err)) return;
    } else {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }

    // ---- phases.  Sites of phases 0 and 1 share the even rows and meet phase 2's
    // and 3's, in the odd rows, only as unchanged neighbours (and the other way
    // round), so a warp runs phases 0 and 1 of its own rows on its own, and after
    // one block barrier phases 2 and 3.
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
        const int at = pos0 + (p >> 1) * WX + (p & 1), sh = 8 * (p & 1);
        int n = 0;
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            if (!EVEN && warp + NW * m >= Cfg::SY) continue;
            const uint32_t kc = ((p & 2 ? kk[1][m] : kk[0][m]) >> sh) & 255u;
            const uint32_t u = p & 2 ? (p & 1 ? u1[3][m] : u1[2][m]) : (p & 1 ? u1[1][m] : u1[0][m]);
            const int pos = at + 2 * NW * m * WX, o = off[kc];
            const bool pr = w.Q[pos + o] != w.Q[pos];
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, pr);
            if (pr) queue[n + __popc(bal & lt)] = make_uint2((uint32_t)pos | ((uint32_t)o << 16), u);
            n += __popc(bal);
        }
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const uint2 e = queue[i];
            w.test((int)(e.x & 0xFFFFu), (int)e.x >> 16, e.y);
        }
        if (p == 1) __syncthreads(); else __syncwarp();
    }

    if (chained && !early) chain_open();
    // ---- write the warp's rows of the core: rows [2, WY - 2), columns [4, WX - 4)
    int32_t* qo = a.q_out + zbase;
    int32_t* mpo = HASMP ? a.mp_out + zbase : nullptr;
    const uintptr_t lowo = (uintptr_t)a.q_out | (HASMP ? (uintptr_t)a.mp_out : 0);
    const int wv = a.Lx % 4 == 0 && (lowo & 15u) == 0 ? 4 : (lowo & 7u) == 0 ? 2 : 1;
#pragma unroll
    for (int m = 0; m < PER; ++m) {
        const int y = 2 * (warp + NW * m);  // 16-byte chunks: a half-warp per row; else a row after the other
        if (wv == 4) {
            const int yy = y + (lane >> 4), c = 4 * (lane & 15), gx = x0 + c - 4, gy = y0 + yy - 2;
            if (yy < 2 || yy >= WY - 2 || c < 4 || c >= WX - 4 || gx >= a.Lx || gy >= a.Ly) continue;
            const uint32_t o = (uint32_t)gx + (uint32_t)a.Lx * (uint32_t)gy;
            *reinterpret_cast<int4*>(qo + o) = *reinterpret_cast<const int4*>(w.Q + yy * WX + c);
            if (HASMP) *reinterpret_cast<int4*>(mpo + o) = *reinterpret_cast<const int4*>(w.MP + yy * WX + c);
        } else {
            const int c = 2 * lane, gx = x0 + c - 4;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int yy = y + r, gy = y0 + yy - 2, li = yy * WX + c;
                if (yy < 2 || yy >= WY - 2 || c < 4 || c >= WX - 4 || gx >= a.Lx || gy >= a.Ly) continue;
                const uint32_t o = (uint32_t)gx + (uint32_t)a.Lx * (uint32_t)gy;
                if (wv == 2) {
                    *reinterpret_cast<int2*>(qo + o) = *reinterpret_cast<const int2*>(w.Q + li);
                    if (HASMP) *reinterpret_cast<int2*>(mpo + o) = *reinterpret_cast<const int2*>(w.MP + li);
                } else {
                    qo[o] = w.Q[li];
                    qo[o + 1] = w.Q[li + 1];
                    if (HASMP) {
                        mpo[o] = w.MP[li];
                        mpo[o + 1] = w.MP[li + 1];
                    }
                }
            }
        }
    }
}

template <int WY, int FIELD, bool HASMP, int NW>
__global__ void __launch_bounds__(LeanCfg<WY, FIELD, HASMP, NW>::kLT, LeanCfg<WY, FIELD, HASMP, NW>::MINB)
    k_lean26(const __grid_constant__ PlaneArgs a, const __grid_constant__ LeanMaps maps) {
    extern __shared__ __align__(16) unsigned char raw[];
    lean_body<WY, FIELD, HASMP, NW>(a, &maps, (int)blockIdx.x, (int)blockIdx.y, raw);
}

// Many independent lattices in one launch: block b belongs to the replica r
// with start[r] <= b < start[r+1]; within it b - start[r] = zidx * tiles + tile.
// Windows are filled by the asynchronous copies, 16 or 8 bytes, or by single loads.
template <int WY, int FIELD, bool HASMP, int NW>
__global__ void __launch_bounds__(LeanCfg<WY, FIELD, HASMP, NW>::kLT, LeanCfg<WY, FIELD, HASMP, NW>::MINB)
    k_lean26_batch(const PlaneArgs* __restrict__ args, const int64_t* __restrict__ start, int R, uint32_t sweep_add) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ PlaneArgs sa;
    __shared__ int s_tile, s_zidx;
    if (threadIdx.x == 0) {
        const int64_t blk = blockIdx.x;
        int lo = 0, hi = R - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (start[mid] <= blk) lo = mid; else hi = mid - 1;
        }
        sa = args[lo];
        sa.sweep += sweep_add;
        sweep_key(sa.seed, sa.sweep, &sa.key);
        const int64_t local = blk - start[lo];
        s_zidx = (int)(local / sa.tiles);
        s_tile = (int)(local - (int64_t)s_zidx * sa.tiles);
    }
    __syncthreads();
    lean_body<WY, FIELD, HASMP, NW>(sa, nullptr, s_tile, s_zidx, raw);
}

PFN_cuTensorMapEncodeTiled_v12000 map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Descriptor of one int32 lattice array (Lx x Ly x Lz) with a 64 x WY x 1 box;
// false when it cannot be encoded (the kernel then copies every window with
// asynchronous copies, or single loads, instead).
bool encode_box(CUtensorMap* m, const void* base, const PlaneArgs& a, int WY) {
    memset(m, 0, sizeof(*m));
    PFN_cuTensorMapEncodeTiled_v12000 enc = map_encoder();
    if (!enc || !base || a.Lx % 4 != 0 || ((uintptr_t)base & 15u) != 0) return false;
    cuuint64_t dims[3] = {(cuuint64_t)a.Lx, (cuuint64_t)a.Ly, (cuuint64_t)a.Lz};
    cuuint64_t strides[2] = {(cuuint64_t)a.Lx * 4, (cuuint64_t)a.Lx * (cuuint64_t)a.Ly * 4};
    cuuint32_t box[3] = {64u, (cuuint32_t)WY, 1u};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_INT32, 3u, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int WY, int FIELD, bool HASMP, int NW>
int launch_lean_nw(const PlaneArgs& a, int planes, cudaStream_t s) {
    using Cfg = LeanCfg<WY, FIELD, HASMP, NW>;
    constexpr size_t smem = Cfg::smem();
    static bool configured = false;  // per template instance
    if (!configured) {
        HP_CUDA(cudaFuncSetAttribute(k_lean26<WY, FIELD, HASMP, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
        configured = true;
    }
    if (a.tiles == 0 || planes == 0) return HP_OK;
    LeanMaps maps;
    memset(&maps, 0, sizeof(maps));
    bool ok = a.Lx >= 64 && encode_box(&maps.q_in, a.q_in, a, WY) && encode_box(&maps.q_nb, a.q_nb, a, WY);
    if (ok && HASMP) ok = encode_box(&maps.mp_in, a.mp_in, a, WY);
    maps.ok = ok ? 1 : 0;
    if (ok && HASMP) maps.pfm = encode_box(&maps.mp_nb, a.mp_nb, a, WY) ? 1 : 0;
    // a per-point field table of one entry per site shares the lattice's layout
    if (ok && FIELD == 2 && a.table_n == (uint32_t)((uint64_t)a.Lx * a.Ly * a.Lz) &&
        (uint64_t)a.Lx * a.Ly * a.Lz <= 0xFFFFFFFFull)
        maps.pf = encode_box(&maps.tab, a.table, a, WY) ? 1 : 0;
    count_launch();
    HP_CUDA(launch_chained(k_lean26<WY, FIELD, HASMP, NW>, dim3((unsigned)a.tiles, (unsigned)planes), Cfg::kLT, smem, s,
                           a.chain != 0, a, maps));
    return HP_OK;
}

template <int WY, int FIELD, bool HASMP>
int launch_lean(const PlaneArgs& a, int planes, cudaStream_t s) {
    if constexpr (HASMP && WY == 32)
        if (lean_warps((int64_t)a.tiles * planes) == 8) return launch_lean_nw<WY, FIELD, HASMP, 8>(a, planes, s);
    return launch_lean_nw<WY, FIELD, HASMP, 4>(a, planes, s);
}

template <int WY, int FIELD, bool HASMP, int NW>
int launch_lean_batch_nw(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add,
                         cudaStream_t s) {
    using Cfg = LeanCfg<WY, FIELD, HASMP, NW>;
    constexpr size_t smem = Cfg::smem();
    static bool configured = false;  // per template instance
    if (!configured) {
        HP_CUDA(cudaFuncSetAttribute(k_lean26_batch<WY, FIELD, HASMP, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
        configured = true;
    }
    if (blocks == 0) return HP_OK;  // configure only (outside a graph capture)
    count_launch();
    k_lean26_batch<WY, FIELD, HASMP, NW><<<(unsigned)blocks, Cfg::kLT, smem, s>>>(d_args, d_start, R, sweep_add);
    HP_LAUNCH_CHECK("k_lean26_batch");
    return HP_OK;
}

template <int WY, int FIELD, bool HASMP>
int launch_lean_batch(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add,
                      cudaStream_t s) {
    if constexpr (WY == 32) {
        if (blocks == 0) {  // either may be launched
            const int rc = launch_lean_batch_nw<WY, FIELD, HASMP, 8>(d_args, d_start, R, 0, sweep_add, s);
            if (rc) return rc;
        } else if (lean_warps(blocks, HASMP ? 0 : LeanCfg<WY, FIELD, HASMP>::MINB) == 8) {
            return launch_lean_batch_nw<WY, FIELD, HASMP, 8>(d_args, d_start, R, blocks, sweep_add, s);
        }
    }
    return launch_lean_batch_nw<WY, FIELD, HASMP, 4>(d_args, d_start, R, blocks, sweep_add, s);
}

template <int WY>
int lean_fm_batch(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add, int field,
                  bool m, cudaStream_t s) {
    if (field == HP_FIELD_POINT) return launch_lean_batch<WY, 2, true>(d_args, d_start, R, blocks, sweep_add, s);
    if (field == HP_FIELD_GRAIN)
        return m ? launch_lean_batch<WY, 1, true>(d_args, d_start, R, blocks, sweep_add, s)
                 : launch_lean_batch<WY, 1, false>(d_args, d_start, R, blocks, sweep_add, s);
    return m ? launch_lean_batch<WY, 0, true>(d_args, d_start, R, blocks, sweep_add, s)
             : launch_lean_batch<WY, 0, false>(d_args, d_start, R, blocks, sweep_add, s);
}

template <int WY>
int lean_fm(const PlaneArgs& a, int field, bool m, int planes, cudaStream_t s) {
    if (field == HP_FIELD_POINT) return launch_lean<WY, 2, true>(a, planes, s);
    if (field == HP_FIELD_GRAIN) return m ? launch_lean<WY, 1, true>(a, planes, s) : launch_lean<WY, 1, false>(a, planes, s);
    return m ? launch_lean<WY, 0, true>(a, planes, s) : launch_lean<WY, 0, false>(a, planes, s);
}

}  // namespace

int lean_launch(const PlaneArgs& a, int field, bool hasmp, int planes, int WY, cudaStream_t s) {
    if (WY == 44) return lean_fm<44>(a, field, hasmp, planes, s);
    if (WY == 40) return lean_fm<40>(a, field, hasmp, planes, s);
    if (WY == 36) return lean_fm<36>(a, field, hasmp, planes, s);
    if (WY == 32) return lean_fm<32>(a, field, hasmp, planes, s);
    return set_error(HP_ERR_ARG, "sweep: no lean kernel of this shape");
}

int lean_launch_batch(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add,
                      int field, bool hasmp, int WY, cudaStream_t s) {
    if (WY == 44) return lean_fm_batch<44>(d_args, d_start, R, blocks, sweep_add, field, hasmp, s);
    if (WY == 40) return lean_fm_batch<40>(d_args, d_start, R, blocks, sweep_add, field, hasmp, s);
    if (WY == 36) return lean_fm_batch<36>(d_args, d_start, R, blocks, sweep_add, field, hasmp, s);
    if (WY == 32) return lean_fm_batch<32>(d_args, d_start, R, blocks, sweep_add, field, hasmp, s);
    return set_error(HP_ERR_ARG, "sweep: no lean kernel of this shape");
}

int lean_wait_probe(long long limit, int late, cudaStream_t s) {
    if (limit < 1 || limit > kWaitCycles) return set_error(HP_ERR_ARG, "wait probe: limit out of range");
    count_launch();
    k_wait_probe<<<1, 64, 0, s>>>(limit, late);
    HP_LAUNCH_CHECK("k_wait_probe");
    return HP_OK;
}

int lean_status(int* timed_out) {
    int v = 0, zero = 0;
    HP_CUDA(cudaMemcpyFromSymbol(&v, g_lean_err, sizeof(int)));
    if (v) HP_CUDA(cudaMemcpyToSymbol(g_lean_err, &zero, sizeof(int)));
    *timed_out = v;
    return HP_OK;
}

}  // namespace hp
