// Device helpers shared by the sweep kernels (sweep.cu, tile.cu, lean.cu): lattice
// neighbourhoods and colourings (Sec. 4), the integer Metropolis test (Eq. (7)
// with the acceptance table of Sec. 4), periodic wrapping, the launch
// arguments of one fused sweep launch, and the mbarrier wait used by the
// TMA-fed kernels.  Internal; not part of the public ABI.
#pragma once

#include "common.cuh"

namespace hp {

// Arguments of one fused sweep launch over the planes of one parity.
struct PlaneArgs {
    const int32_t* q_in;    // own plane, previous state
    const int32_t* mp_in;
    const int32_t* q_nb;    // z-neighbour planes (3D)
    const int32_t* mp_nb;
    int32_t* q_out;
    int32_t* mp_out;
    const int32_t* table;
    uint32_t table_n;
    const uint32_t* thr;
    int32_t D, J;
    uint64_t seed;
    uint32_t sweep;
    int Lx, Ly, Lz;
    int zpar;               // 3D: parity of the planes handled by this launch
    int tiles_x;
    int tiles;              // tiles per plane
    int fast;               // 1: window narrower than the lattice (wrap by one add)
    int vec;                // 1: fast, Lx % 4 == 0 and every buffer on 16 bytes (16-byte row chunks)
    SweepKey key;           // what the draws of (seed, sweep) share
    int chain;              // 1: the launch before on the stream is this call's (launch_chained)
};

// Misorientation tables of hp_set_anisotropy: bin of grains a and b = |ang_a -
// ang_b| folded by the angle's symmetry period, divided by the bin width, clamped
// to the last bin.  The division is a multiplication (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994): floor(d / bin) =
// (t + ((d - t) >> 1)) >> shift, t = mul d / 2^32, for every 32-bit d.
struct Aniso {
    const int32_t* ang;   // grain angles (borrowed, G entries)
    const int32_t* jtab;  // energy per misorientation bin (256 = 1 J)
    const uint32_t* mob;  // relative mobility per bin (all ones = 1), or null
    uint32_t period, bin, mul, shift, last_bin, last_grain;
};
inline Aniso aniso_of(const hp_handle* h) {
    Aniso a;
    a.ang = h->an_ang;
    a.jtab = h->an_J;
    a.mob = h->an_mob;
    a.period = (uint32_t)h->an_period;
    a.bin = (uint32_t)h->an_bin;
    a.last_bin = (uint32_t)h->an_nbins - 1u;
    a.last_grain = (uint32_t)h->desc.n_grains - 1u;
    uint32_t l = 0;
    while (l < 32 && ((uint64_t)1 << l) < a.bin) ++l;
    a.mul = a.bin ? (uint32_t)(((((uint64_t)1 << l) - a.bin) << 32) / a.bin + 1) : 0u;
    a.shift = l ? l - 1 : 0;
    return a;
}

namespace {

// a grain's angle (the id clamped into the table: it comes from a caller buffer)
__device__ __forceinline__ int32_t mis_angle(const Aniso& a, int32_t q) { return __ldg(a.ang + min((uint32_t)q, a.last_grain)); }
__device__ __forceinline__ uint32_t mis_bin(const Aniso& a, int32_t ua, int32_t ub) {
    uint32_t d = ua > ub ? (uint32_t)ua - (uint32_t)ub : (uint32_t)ub - (uint32_t)ua;
    if (d >= a.period) d %= a.period;  // angles outside [0, period)
    d = min(d, a.period - d);
    const uint32_t t = __umulhi(a.mul, d);
    const uint32_t k = a.bin == 1u ? d : (t + ((d - t) >> 1)) >> a.shift;
    return min(k, a.last_bin);
}
// Trial with the mobility of the (q_i, q_j) boundary: eff = thr[d] (all ones for d <
// 0) when the mobility m is all ones, m when thr is all ones, else floor(thr m /
// 2^32); accept iff d <= D and (eff is all ones or u < eff).
__device__ __forceinline__ bool metropolis_mob(const Aniso& an, int32_t d, int32_t D, const uint32_t* __restrict__ thr,
                                               uint32_t u, int32_t ai, int32_t aj) {
    if (d > D) return false;
    const uint32_t th = d < 0 ? 0xFFFFFFFFu : __ldg(thr + d);
    const uint32_t m = an.mob ? __ldg(an.mob + mis_bin(an, ai, aj)) : 0xFFFFFFFFu;
    const uint32_t eff = m == 0xFFFFFFFFu ? th : (th == 0xFFFFFFFFu ? m : __umulhi(th, m));
    return eff == 0xFFFFFFFFu || u < eff;
}

template <int DIM, int NBR>
struct Geo;

// 2D-4: +x, -x, +y, -y ; colours (x+y)&1
template <>
struct Geo<2, 4> {
    static constexpr int M = 4, C = 2;
    __device__ static void off(int k, int& dx, int& dy, int& dz) {
        dx = k == 0 ? 1 : (k == 1 ? -1 : 0);
        dy = k == 2 ? 1 : (k == 3 ? -1 : 0);
        dz = 0;
    }
};
// 2D-8: (dy,dx) row-major without (0,0) ; colours (x&1) + 2(y&1)
template <>
struct Geo<2, 8> {
    static constexpr int M = 8, C = 4;
    __device__ static void off(int k, int& dx, int& dy, int& dz) {
        const int kk = k + (k >= 4);
        dy = kk / 3 - 1;
        dx = kk % 3 - 1;
        dz = 0;
    }
};
// 3D-6: +x, -x, +y, -y, +z, -z ; colours (x+y+z)&1
template <>
struct Geo<3, 6> {
    static constexpr int M = 6, C = 2;
    __device__ static void off(int k, int& dx, int& dy, int& dz) {
        dx = k == 0 ? 1 : (k == 1 ? -1 : 0);
        dy = k == 2 ? 1 : (k == 3 ? -1 : 0);
        dz = k == 4 ? 1 : (k == 5 ? -1 : 0);
    }
};
// 3D-26: (dz,dy,dx) lexicographic without (0,0,0) ; colours (x&1)+2(y&1)+4(z&1)
template <>
struct Geo<3, 26> {
    static constexpr int M = 26, C = 8;
    __device__ static void off(int k, int& dx, int& dy, int& dz) {
        const int kk = k + (k >= 13);
        dz = kk / 9 - 1;
        dy = (kk / 3) % 3 - 1;
        dx = kk % 3 - 1;
    }
};

__device__ __forceinline__ int wrapi(int a, int L) {
    a %= L;
    return a < 0 ? a + L : a;
}

// a in [-L, 2L)
__device__ __forceinline__ int wrap1(int a, int L) {
    a += a < 0 ? L : 0;
    return a - (a >= L ? L : 0);
}

__device__ __forceinline__ bool metropolis(int32_t d, int32_t D, const uint32_t* __restrict__ thr, uint32_t u) {
    if (d < 0) return true;
    if (d > D) return false;
    const uint32_t t = __ldg(thr + d);
    return t == 0xFFFFFFFFu || u < t;
}

// Field-table lookup with the index clamped into the table (ids come from
// caller buffers; an out-of-range id must not read outside the table).
__device__ __forceinline__ int32_t tab(const int32_t* __restrict__ t, uint32_t n, int32_t i) {
    const uint32_t u = (uint32_t)i;
    return __ldg(t + (u < n ? u : n - 1));
}

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Wait for an mbarrier phase with a clock limit (default about two seconds at
// the boost clock); false on timeout.  Each try_wait may suspend the thread for
// up to 20 us (it wakes as soon as the phase completes), so a waiting warp
// issues few instructions.
constexpr long long kWaitCycles = 1ll << 32;
__device__ __forceinline__ bool wait_parity(uint32_t mbar, uint32_t parity, long long limit = kWaitCycles) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(mbar), "r"(parity), "r"(20000u) : "memory");
        if (done) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// Block-wide wait for a window's bulk copies (every thread calls it).  Warp 0
// polls the barrier while the other warps wait at the block barrier (issuing
// nothing); once the copies have landed every thread observes the completed
// phase itself (a try_wait that succeeds at once), which orders its reads
// after the copies.  On a timeout every thread of the block keeps waiting, up
// to four more limits, so that no copy is still landing in this block's shared
// memory when it leaves; *flag becomes 1, or 2 if even that drain ran out
// (copies may still have been in flight at exit: the context must not be
// trusted).  False after a timeout.
__device__ __forceinline__ bool wait_or_drain(uint32_t mbar, int* flag, long long limit = kWaitCycles) {
    bool ok = true;
    if (threadIdx.x < 32) ok = wait_parity(mbar, 0u, limit);
    if (!__syncthreads_or(!ok)) {
        if (threadIdx.x >= 32) wait_parity(mbar, 0u, limit);
        return true;
    }
    bool drained = false;
    for (int i = 0; i < 5 && !drained; ++i) drained = wait_parity(mbar, 0u, limit);
    const bool all = !__syncthreads_or(!drained);
    if (threadIdx.x == 0) atomicMax(flag, all ? 1 : 2);
    return false;
}

// Launches of one call chained without a drain between them (programmatic dependent
// launch): a kernel lets the next one's blocks in (chain_open), and those set up and
// then wait (chain_wait) until it has finished and its stores are visible.  They are
// let in once every block of the kernel has got that far, so they only take slots
// that nobody waits for, and the wait is the hardware's.  Whatever a chained kernel
// reads before chain_wait, or through the read-only path, no kernel of the chain
// writes.  A grid of many waves opens at its start, so that the next one fills the
// slots that its last wave leaves; one of about a wave opens before it writes back:
// opened at its start, the next grid is packed onto whatever SMs have room, three
// blocks here and none there (1024^2 with misorientation tables: 28 us per MCS; 20.7
// with a drain between launches, 18.7 as it is).  Per MCS, drained -> chained: 700^2, 8
// neighbours 10.4 -> 8.1 us; 1500^2, 4 neighbours 14.7 -> 11.4; 4096^2, 8 neighbours
// 63.5 -> 61.6; 3D 64^3 20.7 -> 16.3, 256^3 217 -> 212.  The batched launches of an
// ensemble are not chained: 24 uneven replicas of 64^3 to 256^3 took 8.7 ms so, 8.4
// without.
__device__ __forceinline__ void chain_open() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ bool chain_early() { return gridDim.x * gridDim.y > 2048u; }  // some three waves

template <class... P, class... A>
cudaError_t launch_chained(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, bool chain, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<A&&>(args)...);
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const int32_t* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}

// Copy window columns [xs, xs + W) of one lattice row (xs >= -4, W <= Lx,
// all multiples of 4 ints) into dst, wrapping periodically.
__device__ __forceinline__ void copy_row(int32_t* dst, const int32_t* row, int xs, int W, int Lx, uint32_t mb) {
    if (xs < 0) {
        bulk_g2s(s_addr(dst), row + Lx + xs, (uint32_t)(-xs) * 4u, mb);
        bulk_g2s(s_addr(dst - xs), row, (uint32_t)(W + xs) * 4u, mb);
    } else if (xs + W > Lx) {
        bulk_g2s(s_addr(dst), row + xs, (uint32_t)(Lx - xs) * 4u, mb);
        bulk_g2s(s_addr(dst + (Lx - xs)), row, (uint32_t)(xs + W - Lx) * 4u, mb);
    } else {
        bulk_g2s(s_addr(dst), row + xs, (uint32_t)W * 4u, mb);
    }
}

}  // namespace

// Tile kernel (tile.cu): one launch over the planes of one parity; WX x WY
// window (core (WX - 8) x (WY - 8)), a.tiles_x / a.tiles set for that core.
int tile_launch(const PlaneArgs& a, int field, bool hasmp, int nbr, int planes, int WX, int WY, cudaStream_t s);
// The same over many lattices: d_args[R] (device), block offsets d_start[R+1];
// blocks == 0 only configures the kernel (outside a graph capture).
int tile_launch_batch(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add,
                      int field, bool hasmp, int nbr, int WX, int WY, cudaStream_t s);
// One launch over a 2D lattice with misorientation tables (128 x 32 windows).
int tile_launch_aniso(const PlaneArgs& a, const Aniso& an, int field, bool hasmp, int nbr, cudaStream_t s);
// Reads and clears the tile kernel's timeout flag.
int tile_status(int* timed_out);

// Lean 3D kernel (lean.cu): one launch over the planes of one parity; 64 x WY
// windows (WY 32, 36, 40 or 44), draws made while the window is in flight.
int lean_launch(const PlaneArgs& a, int field, bool hasmp, int planes, int WY, cudaStream_t s);
// The same over many lattices (see tile_launch_batch).
int lean_launch_batch(const PlaneArgs* d_args, const int64_t* d_start, int R, int64_t blocks, uint32_t sweep_add,
                      int field, bool hasmp, int WY, cudaStream_t s);
// Reads and clears the lean kernel's timeout flag (2: a drain ran out too).
int lean_status(int* timed_out);

// Resident 2D sweep (res2d.cu): cluster size for these lattices (all of one dim, nbr,
// field mode), 0 when one of them does not fit or is of another kind.
int res2d_cluster(hp_handle* const* m, int R);
// Estimated us per MCS of an ensemble there, -1 when unknown.
double res2d_us(hp_handle* const* m, int R, int cs);
// n_mcs MCS of every lattice, in place, from each handle's sweep counter (not
// advanced here).
int res2d_run(hp_handle* const* m, int R, int cs, int32_t n_mcs, cudaStream_t s);


}  // namespace hp
