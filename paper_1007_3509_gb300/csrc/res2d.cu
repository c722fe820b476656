// Resident 2D sweep: the whole lattice stays in the shared memory of one
// thread-block cluster for many MCS (Eq. (7), Sec. 4; 4- and 8-neighbour lattices,
// no field or a per-grain one, no material points).
//
// A small lattice is bound by latency: one launch per MCS, a window fill, a handful
// of barriers and the drain of a nearly empty chip cost 7 to 14 us however few the
// sites.  Here CTA r of a cluster of `cs` keeps a strip of whole row pairs with one
// ghost row above and below, and one launch runs all the MCS asked for:
//  * a flip in a strip's first or last row is also stored into the neighbour
//    strip's ghost row (distributed shared memory); flips are few, so nothing else
//    is exchanged;
//  * a warp owns whole rows.  8 neighbours: colours 0 and 1 (even rows) meet the
//    odd rows only as unchanged neighbours, so a warp runs both on its rows, then
//    the cluster meets, then colours 2 and 3: two cluster barriers per MCS.
//    4 neighbours: one barrier per colour, two per MCS as well;
//  * per row and colour a warp draws for every site, queues the proposals of another
//    grain and tests 32 of them at a time.  An interior test before the draw costs
//    as much as it saves (159 against 84 operations per site-update on a lattice of
//    50-site grains at kT = 1);
//  * the first draws after a barrier are made between arriving and waiting;
//  * rows carry one ghost column on either side, so no address is wrapped.
// The barriers are the hardware's (barrier.cluster), over CTAs that are scheduled
// together by construction; there is no spin.
// Measured, per MCS: 128^2, 4 neighbours 14.4 -> 2.9 us (one launch per MCS before);
// 32 lattices of 500^2, 8 neighbours, kT = 1: 90.6 -> 60.3 us (one launch of plane
// tiles before).  The first is bound by latency (two barriers, two rounds of a draw
// and a test), the second by instructions: 124 per site-update, 37 of them the draw.
#include <string.h>

#include <atomic>

#include "routes.h"
#include "sweep.cuh"

namespace hp {
namespace {

constexpr int kMembers = 60;             // lattices per launch (their arguments are launch parameters)
constexpr int kMcsPerLaunch = 4096;      // keeps one launch within a fraction of a second
constexpr int kSmemMax = 227 * 1024;

struct ResArgs {
    int32_t* q;
    const int32_t* table;
    const uint32_t* thr;
    uint64_t seed;
    uint32_t table_n, sweep;
    int32_t D, J;
    int32_t Lx, Ly;
};
struct ResBatch {
    ResArgs m[kMembers];
    int cs;        // CTAs per lattice (the cluster size)
    int n_mcs;
    int smem;      // dynamic shared memory of the launch, bytes
};

__host__ __device__ inline int strip_start(int Ly, int cs, int r) {
    const int pairs = Ly / 2, rem = pairs % cs;
    return 2 * (r * (pairs / cs) + (r < rem ? r : rem));
}
// A strip row: two ints of padding, of which the second is the ghost of column
// Lx - 1, the row, and the ghost of column 0 (even sites lie on 8-byte boundaries).
__host__ __device__ inline int pitch(int Lx) { return Lx + 4; }
// shared memory: rows with their ghosts | proposal queue (kQueue per warp) |
// neighbour offsets | thresholds and field table, each where it fits
constexpr int kQueue = 96;
__host__ __device__ inline size_t res_bytes(int rows, int Lx, int warps) {
    return ((4 * (size_t)(rows + 2) * pitch(Lx) + 15) & ~(size_t)15) + 8 * kQueue * (size_t)warps + 32;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// store into another CTA's shared memory, at the address that p has in this one
__device__ __forceinline__ void store_remote(int32_t* p, uint32_t rank, int32_t v) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(s_addr(p)), "r"(rank));
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// what a lane drew for its sites of two adjacent runs of 32 columns of one colour
struct Draws {
    uint32_t k[2], u[2];
};

template <int NBR, int FIELD>
struct Res {
    int32_t* Q;      // rows 0 .. rows + 1 of the strip (column 0), 0 and rows + 1 ghosts
    int Lx, half, P;  // half = Lx / 2, P = pitch
    int rows, up_rows;
    uint32_t up, down;
    int y0;          // lattice row of strip row 1
    const int32_t* tab;
    uint32_t tab_last;
    const uint32_t* thr;
    int32_t D, J;
    uint2* queue;    // this warp's: column | neighbour << 24, acceptance draw
    const int* off;  // offset of each neighbour
    SweepKey key;

    // Metropolis test of queued proposal e in strip row `row`
    __device__ __forceinline__ void test(int row, uint2 e) const {
        const int x = (int)(e.x & 0xFFFFFFu);
        int32_t* c = Q + row * P + x;
        const int32_t qi = c[0], qj = c[off[e.x >> 24]];
        const int odd = x & 1;
        const int32_t* pr = c - odd;                 // the aligned pair with the site's column
        const int32_t* sg = c + 2 * odd - 1;         // the column on its other side
        int ni = -1, nj = 0;                         // the site itself counts once among its own
        if (NBR == 8) {
#pragma unroll
            for (int r = -1; r <= 1; ++r) {
                const int2 v = *reinterpret_cast<const int2*>(pr + r * P);
                const int32_t w = sg[r * P];
                if (v.x == qi) ++ni;
                if (v.x == qj) ++nj;
                if (v.y == qi) ++ni;
                if (v.y == qj) ++nj;
                if (w == qi) ++ni;
                if (w == qj) ++nj;
            }
        } else {
            const int2 v = *reinterpret_cast<const int2*>(pr);
            const int32_t w = sg[0], u = c[-P], d = c[P];
            ni += (v.x == qi) + (v.y == qi) + (w == qi) + (u == qi) + (d == qi);
            nj += (v.x == qj) + (v.y == qj) + (w == qj) + (u == qj) + (d == qj);
        }
        int32_t db = 0;
        if (FIELD) db = tab[min((uint32_t)qj, tab_last)] - tab[min((uint32_t)qi, tab_last)];
        const int32_t d = J * (ni - nj) + db;
        if (d > D) return;
        if (d >= 0) {
            const uint32_t t = thr[d];
            if (!(t == 0xFFFFFFFFu || e.y < t)) return;
        }
        c[0] = qj;
        const int wrap = x == 0 ? Lx : (x == Lx - 1 ? -Lx : 0);  // the column's ghost
        if (wrap) c[wrap] = qj;
        if (row == 1 || row == rows) {                           // the neighbour strips' ghost rows
            if (row == 1) {
                int32_t* g = Q + (up_rows + 1) * P + x;
                store_remote(g, up, qj);
                if (wrap) store_remote(g + wrap, up, qj);
            }
            if (row == rows) {
                store_remote(Q + x, down, qj);
                if (wrap) store_remote(Q + x + wrap, down, qj);
            }
        }
    }
    __device__ __forceinline__ Draws draw2(int row, int px, uint32_t colour, int c) const {
        const uint32_t unit = (uint32_t)Lx * (uint32_t)(y0 + row - 1) + (uint32_t)(2 * (c + (int)(threadIdx.x & 31)) + px);
        Draws d;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint2 u = sweep_draw(key, unit + 64u * (uint32_t)i, colour);
            d.k[i] = __umulhi(u.x, (uint32_t)NBR);
            d.u[i] = u.y;
        }
        return d;
    }
    // one colour of one strip row (sites 2 s + px), by one warp; d: the draws of its
    // first two runs
    __device__ __forceinline__ void line(int row, int px, uint32_t colour, Draws d) const {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        const int32_t* b = Q + row * P;
        int n = 0;
        for (int c = 0;;) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int s = c + 32 * i + lane;
                const bool in = s < half;
                const int x = in ? 2 * s + px : px;
                const bool pr = in && b[x + off[d.k[i]]] != b[x];
                const unsigned bal = __ballot_sync(0xFFFFFFFFu, pr);
                if (pr) queue[n + __popc(bal & lt)] = make_uint2((uint32_t)x | (d.k[i] << 24), d.u[i]);
                n += __popc(bal);
            }
            __syncwarp();
            while (n >= 32) {
                n -= 32;
                test(row, queue[n + lane]);
            }
            c += 64;
            if (c >= half) break;
            d = draw2(row, px, colour, c);
            __syncwarp();
        }
        if (lane < n) test(row, queue[lane]);
        __syncwarp();
    }
    __device__ __forceinline__ void line(int row, int px, uint32_t colour) const {
        line(row, px, colour, draw2(row, px, colour, 0));
    }
};

template <int NBR, int FIELD>
__global__ void __launch_bounds__(1024, 1) k_res2d(const __grid_constant__ ResBatch a) {
    extern __shared__ __align__(16) int32_t rsm[];
    const ResArgs& m = a.m[blockIdx.x / a.cs];
    const int tid = threadIdx.x, warp = tid >> 5, nw = (int)blockDim.x >> 5, nt = (int)blockDim.x;
    Res<NBR, FIELD> r;
    const uint32_t rank = a.cs > 1 ? cluster_rank() : 0u;
    r.up = rank == 0 ? (uint32_t)a.cs - 1u : rank - 1u;
    r.down = rank + 1u == (uint32_t)a.cs ? 0u : rank + 1u;
    r.Q = rsm;
    r.Lx = m.Lx;
    r.half = m.Lx / 2;
    r.rows = strip_rows(m.Ly, a.cs, (int)rank);
    r.up_rows = strip_rows(m.Ly, a.cs, (int)r.up);
    r.y0 = strip_start(m.Ly, a.cs, (int)rank);
    r.D = m.D;
    r.J = m.J;
    // every strip of a lattice lays its rows out from the same address
    const int most = strip_rows(m.Ly, a.cs, 0), P = pitch(m.Lx);
    r.P = P;
    r.Q = rsm + 2;
    char* at = reinterpret_cast<char*>(rsm) + ((4 * (size_t)(most + 2) * P + 15) & ~(size_t)15);
    r.queue = reinterpret_cast<uint2*>(at) + kQueue * warp;
    int* off = reinterpret_cast<int*>(at + 8 * kQueue * nw);
    r.off = off;
    if (tid < NBR) {
        int dx, dy, dz;
        Geo<2, NBR>::off(tid, dx, dy, dz);
        off[tid] = dy * P + dx;
    }
    char* end = reinterpret_cast<char*>(rsm) + a.smem;
    char* room = reinterpret_cast<char*>(off + 8);
    r.thr = m.thr;
    if (room + 4 * (int64_t)(m.D + 1) <= end) {
        uint32_t* t = reinterpret_cast<uint32_t*>(room);
        for (int i = tid; i <= m.D; i += nt) t[i] = m.thr[i];
        r.thr = t;
        room += 4 * (int64_t)(m.D + 1);
    }
    r.tab = m.table;
    r.tab_last = m.table_n - 1u;
    if (FIELD && room + 4 * (int64_t)m.table_n <= end) {
        int32_t* t = reinterpret_cast<int32_t*>(room);
        for (uint32_t i = tid; i < m.table_n; i += nt) t[i] = m.table[i];
        r.tab = t;
    }
    // rows y0 - 1 .. y0 + rows of the lattice, with their ghost columns
    for (int y = warp; y < r.rows + 2; y += nw) {
        const int g = r.y0 + y - 1, gy = g < 0 ? m.Ly - 1 : (g >= m.Ly ? 0 : g);
        const int32_t* src = m.q + (int64_t)m.Lx * gy;
        int32_t* dst = r.Q + y * P;
        for (int x = tid & 31; x < m.Lx; x += 32) dst[x] = src[x];
        if ((tid & 31) == 0) dst[-1] = src[m.Lx - 1];
        if ((tid & 31) == 1) dst[m.Lx] = src[0];
    }
    const bool cluster = a.cs > 1;
    // first row and column parity of this warp in half h of an MCS
    const int row0 = NBR == 8 ? 1 + 2 * warp : 1 + warp;
    if (cluster) cluster_arrive(); else __syncthreads();
    for (int t = 0; t < a.n_mcs; ++t) {
        sweep_key(m.seed, m.sweep + (uint32_t)t, &r.key);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (NBR == 8) {
                Draws d = r.draw2(row0 + h, 0, 2u * (uint32_t)h, 0);
                if (cluster) cluster_wait();
                for (int row = row0 + h; row <= r.rows; row += 2 * nw) {
                    if (row != row0 + h) d = r.draw2(row, 0, 2u * (uint32_t)h, 0);
                    r.line(row, 0, 2u * (uint32_t)h, d);
                    r.line(row, 1, 2u * (uint32_t)h + 1u);
                }
            } else {
                Draws d = r.draw2(row0, (h + row0 - 1) & 1, (uint32_t)h, 0);
                if (cluster) cluster_wait();
                for (int row = row0; row <= r.rows; row += nw) {
                    const int px = (h + row - 1) & 1;
                    if (row != row0) d = r.draw2(row, px, (uint32_t)h, 0);
                    r.line(row, px, (uint32_t)h, d);
                }
            }
            if (cluster) cluster_arrive(); else __syncthreads();
        }
    }
    if (cluster) cluster_wait();
    for (int y = 1 + warp; y <= r.rows; y += nw) {
        int32_t* dst = m.q + (int64_t)m.Lx * (r.y0 + y - 1);
        for (int x = tid & 31; x < m.Lx; x += 32) dst[x] = r.Q[y * P + x];
    }
}

int warps_for(int nbr, int rows) {
    const int lines = strip_lines(nbr, rows), per = lines_per_warp(lines);
    return (lines + per - 1) / per;
}

// Warps a block needs for the largest strip among the members.
int res_warps(hp_handle* const* m, int R, int cs) {
    int w = 1;
    for (int r = 0; r < R; ++r) {
        const int v = warps_for(m[r]->lat.nbr, strip_rows((int)m[r]->lat.L[1], cs, 0));
        w = v > w ? v : w;
    }
    return w;
}

// Shared memory of one member's largest strip: rows and queues, and everything.
size_t res_rows(const hp_handle* h, int cs, int warps) {
    return res_bytes(strip_rows((int)h->lat.L[1], cs, 0), (int)h->lat.L[0], warps);
}
size_t res_all(const hp_handle* h, int cs, int warps) {
    const size_t all = res_rows(h, cs, warps) + 4 * ((size_t)h->D + 1) +
                       (h->desc.field_mode == HP_FIELD_GRAIN ? 4 * (size_t)h->table_n : 0);
    return all < (size_t)kSmemMax ? all : (size_t)kSmemMax;
}

// Launch of `members` clusters; at: room for its one attribute.
template <int NBR, int FIELD>
int config_res(int members, int cs, int warps, int smem, cudaStream_t s, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
    HP_CUDA(cudaFuncSetAttribute(k_res2d<NBR, FIELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
    memset(cfg, 0, sizeof *cfg);
    cfg->gridDim = dim3((unsigned)(members * cs));
    cfg->blockDim = dim3((unsigned)(32 * warps));
    cfg->dynamicSmemBytes = (size_t)smem;
    cfg->stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cs;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = cs > 1 ? 1 : 0;
    return HP_OK;
}

template <int NBR, int FIELD>
int launch_res(const ResBatch& b, int members, int warps, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    const int rc = config_res<NBR, FIELD>(members, b.cs, warps, b.smem, s, &cfg, &at);
    if (rc) return rc;
    count_launch();
    HP_CUDA(cudaLaunchKernelEx(&cfg, k_res2d<NBR, FIELD>, b));
    return HP_OK;
}

// Clusters of a launch that run at the same time (0: the query failed).
template <int NBR, int FIELD>
int active_res(int members, int cs, int warps, int smem) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    int n = 0;
    if (config_res<NBR, FIELD>(members, cs, warps, smem, nullptr, &cfg, &at)) return 0;
    if (cs == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_res2d<NBR, FIELD>, 32 * warps, (size_t)smem) != cudaSuccess) n = 0;
        n *= kSMs;
    } else if (cudaOccupancyMaxActiveClusters(&n, k_res2d<NBR, FIELD>, &cfg) != cudaSuccess) {
        n = 0;
    }
    if (n <= 0) cudaGetLastError();
    return n;
}

size_t res_smem(hp_handle* const* m, int R, int cs, int warps) {
    size_t smem = 0;
    for (int r = 0; r < R; ++r) {
        const size_t want = res_all(m[r], cs, warps);
        smem = want > smem ? want : smem;
    }
    return smem;
}

}  // namespace

int res2d_cluster(hp_handle* const* m, int R) {
    int cs = 8;
    for (int r = 0; r < R; ++r) {
        const hp_handle* h = m[r];
        const int64_t Lx = h->lat.L[0], Ly = h->lat.L[1];
        if (h->lat.dim != 2 || h->mp || h->an_J || h->desc.field_mode == HP_FIELD_POINT || Lx > 2048 || Ly > 4096) return 0;
        cs = res_cluster(cs, Ly);
    }
    const int warps = res_warps(m, R, cs);
    for (int r = 0; r < R; ++r)
        if (res_rows(m[r], cs, warps) > (size_t)kSmemMax) return 0;
    return cs;
}

// Estimated us per MCS of R lattices on clusters of cs, launch after launch: in each, the
// members taken in order by the clusters that run at the same time.  -1: unknown.
double res2d_us(hp_handle* const* m, int R, int cs) {
    const int nbr = m[0]->lat.nbr, field = m[0]->desc.field_mode == HP_FIELD_GRAIN ? 1 : 0;
    double total = 0.0;
    for (int r0 = 0; r0 < R; r0 += kMembers) {
        const int k = R - r0 < kMembers ? R - r0 : kMembers;
        const int warps = res_warps(m + r0, k, cs), smem = (int)res_smem(m + r0, k, cs, warps);
        int active = nbr == 8 ? (field ? active_res<8, 1>(k, cs, warps, smem) : active_res<8, 0>(k, cs, warps, smem))
                              : (field ? active_res<4, 1>(k, cs, warps, smem) : active_res<4, 0>(k, cs, warps, smem));
        if (active < 1) return -1.0;
        const int per_sm = active * cs < kSMs ? 1 : (active * cs + kSMs / 2) / kSMs;  // CTAs an SM takes
        if (active > k) active = k;
        double busy[kMembers] = {}, most = 0.0;
        for (int i = 0; i < k; ++i) {
            int at = 0;
            for (int c = 1; c < active; ++c)
                if (busy[c] < busy[at]) at = c;
            const int first = i / active * active, wave = k - first < active ? k - first : active;
            const int asked = (wave * cs + kSMs - 1) / kSMs;  // CTAs an SM has in this member's wave
            busy[at] += res_us(nbr, m[r0 + i]->lat.L[0], m[r0 + i]->lat.L[1], cs, asked < per_sm ? asked : per_sm);
            most = busy[at] > most ? busy[at] : most;
        }
        total += most;
    }
    return total;
}

int res2d_run(hp_handle* const* m, int R, int cs, int32_t n_mcs, cudaStream_t s) {
    const int nbr = m[0]->lat.nbr, field = m[0]->desc.field_mode == HP_FIELD_GRAIN ? 1 : 0;
    for (int32_t done = 0; done < n_mcs; done += kMcsPerLaunch) {
        const int32_t n = n_mcs - done < kMcsPerLaunch ? n_mcs - done : kMcsPerLaunch;
        for (int r0 = 0; r0 < R; r0 += kMembers) {
            const int k = R - r0 < kMembers ? R - r0 : kMembers;
            ResBatch b;
            memset(&b, 0, sizeof b);
            b.cs = cs;
            b.n_mcs = n;
            const int warps = res_warps(m + r0, k, cs);
            for (int i = 0; i < k; ++i) {
                const hp_handle* h = m[r0 + i];
                ResArgs& a = b.m[i];
                a.q = h->q;
                a.table = h->table;
                a.thr = h->thr;
                a.seed = h->desc.seed;
                a.table_n = (uint32_t)h->table_n;
                a.sweep = (uint32_t)(h->sweep + (uint64_t)done);
                a.D = h->D;
                a.J = h->desc.J_fix;
                a.Lx = (int)h->lat.L[0];
                a.Ly = (int)h->lat.L[1];
            }
            b.smem = (int)res_smem(m + r0, k, cs, warps);
            const int rc = nbr == 8 ? (field ? launch_res<8, 1>(b, k, warps, s) : launch_res<8, 0>(b, k, warps, s))
                                    : (field ? launch_res<4, 1>(b, k, warps, s) : launch_res<4, 0>(b, k, warps, s));
            if (rc) return rc;
        }
    }
    return HP_OK;
}

}  // namespace hp
