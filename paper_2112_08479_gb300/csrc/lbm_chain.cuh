// lbm_chain.cuh -- many time steps in one launch: a persistent kernel whose
// SMs take (step, rows) items in a fixed order and start each as soon as the
// rows around it have finished the step before.
//
// Why.  One launch per step costs a box that fits the 129 MB L2 a launch gap
// and an unfilled last wave per step (4 us of 17 at 256x32x64), and makes a
// larger box read and write its whole state in HBM every step.  In the AA
// pattern a step of plane z needs the step before on planes z - 1 .. z + 1
// only, and every element is touched by one node per step, so steps can follow
// each other through the box as a wave, T of them a few planes apart, and the
// state passes through HBM once per T steps.  An in-place copy of 26 rows runs
// at 13.4 TB/s on a working set of up to 64 MB in L2, 11.9 at 80 MB, 9.4 at
// 96 MB, against 7.0 in HBM.
//
// Items.  A tile is R rows (y) of a plane, M tiles to a plane; an item is U
// warp units (a warp's segment of a row) of a tile at one step.  Tickets are
// drawn from one counter.  Position v = z M + k counts tiles plane by plane;
// ticket W (T bpt) + s bpt + b is item b of step slot s at position W - s lag,
// slot s taking tile (k + s) mod M of its plane so that the periodic
// neighbours of its first and last tile are done in time.  Large planes are
// cut into slabs along x, slot s shifted by s segments to the left (a step
// reaches one node further), one slab's sweep through all planes after the
// other.  With periodic x ends the slots turn like the tiles do: place i of slot
// s is segment (i + s) mod ns, two places behind slot s - 1.
//
// Dependencies.  done[z][tile] counts the finished items of a tile; item
// groups (slab, slot) follow each other on a tile in ticket order, so before
// group nu the 3 x 3 tiles around must count nu bpt.  All these have smaller
// tickets (lag >= M + 3; nz M >= (T - 1) lag + 2 M), and every ticket drawn is
// held by a running block, so the wait always ends, whatever else runs on the
// GPU; it is bounded all the same (ChainParams::limit_ns, LBM_DEVFLAG_TIMEOUT): a
// feeding warp that gives up sets the abort word, which the waits of the other
// blocks see, and `stop`, after which the computing warps finish what is published
// and the announcing warp ends with the last of it.
//
// Roles.  In each block NW warps compute; a feeding warp draws tickets, waits
// for their counters (acquire) and publishes ready items in a ring in shared
// memory; an announcing warp sees finished items and adds them to the counters
// behind one gpu-scope fence.  So no computing warp waits for a counter, a
// fence or another warp.  (Blocks of four computing warps that did all this
// themselves, with a barrier per item: 32 G node updates/s against 47 at
// 256x32x64; one warp for both roles: 43; groups of two tickets: 45.)
#pragma once

#include "lbm_internal.h"

namespace lbmgpu {

// n / d for n < 2^31 by a multiplication (Granlund and Montgomery 1994).
struct Div {
    unsigned d, m, s;
    __host__ void set(unsigned v) {
        d = v;
        s = 0;
        while ((1ull << s) < v) ++s;
        m = (unsigned)(((1ull << 32) * ((1ull << s) - v)) / v + 1);
    }
    __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(n, m) + n) >> s; }
};

struct ChainParams {
    unsigned* sync;     // [0] ticket, [1] abort, [32 ..] done[z * M + tile]
    unsigned total;     // tickets
    int nsteps, T;
    int odd0;           // parity of the first step
    unsigned groups;    // sweeps * nslab
    unsigned U;         // warp units per item
    unsigned lag;       // tiles
    unsigned R;         // rows per tile
    unsigned ns;        // warp segments per row
    unsigned skew;      // segments a slot stays behind the one before: 1, periodic
                        // ends 2; 0 with one slab, whose rows are whole
    Div M;              // tiles per plane (R rows of y each)
    Div bpt;            // items per tile
    Div per;            // T * bpt
    Div P;              // nz * M
    Div nslab;          // x slabs
    Div sw;             // warp segments per row and slab
    Div Ud;             // U
    unsigned long long limit_ns;   // longest wait for a counter
};

constexpr unsigned long long CHAIN_LIMIT_NS = 10000000000ull;   // only a defect waits that long
constexpr unsigned long long CHAIN_STALL_NS = 100000000ull;     // the limit under the test hook
constexpr unsigned CHAIN_COUNTERS = 32;   // first counter in ChainParams::sync (a line of its own)

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void red_add(unsigned* p, unsigned v) {
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long chain_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// An item: step n (< 0: none), its group nu in the tiles' counters, plane,
// tile, item of the tile and first segment.
struct ChainItem {
    int n, nu, z, tile, b, p0, turn;
};

__device__ __forceinline__ ChainItem chain_decode(const ChainParams& cp, unsigned t) {
    ChainItem i;
    i.n = -1; i.z = i.tile = i.b = i.nu = i.p0 = i.turn = 0;
    if (t >= cp.total) return i;
    const unsigned W = cp.per.div(t), r = t - W * cp.per.d;
    const unsigned s = cp.bpt.div(r);
    const int v = (int)W - (int)(s * cp.lag);
    if (v < 0) return i;
    const unsigned J = cp.P.div((unsigned)v);
    if (J >= cp.groups) return i;
    const unsigned q = (unsigned)v - J * cp.P.d;
    const unsigned z = cp.M.div(q);
    unsigned tile = q - z * cp.M.d + s;
    while (tile >= cp.M.d) tile -= cp.M.d;
    const unsigned sweep = cp.nslab.div(J), slab = J - sweep * cp.nslab.d;
    i.n = (int)(sweep * cp.T + s);
    i.nu = (int)(J * cp.T + s);
    i.z = (int)z;
    i.tile = (int)tile;
    i.b = (int)(r - s * cp.bpt.d);
    i.p0 = (int)(slab * cp.sw.d) - (int)(cp.skew * s);
    i.turn = cp.skew == 2 ? (int)s : 0;
    return i;
}

constexpr int CHAIN_GRP = 3;      // items the feeding warp polls at a time (nine lanes each)
constexpr int CHAIN_AHEAD = 3;    // items published ahead of those taken
constexpr int CHAIN_HELPERS = 2;  // the feeding and the announcing warp
constexpr int CHAIN_SLOTS = 32;   // ring of published items (one lane of the announcing warp each)

__device__ __forceinline__ unsigned lds_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
    return v;
}
__device__ __forceinline__ void sts_release(unsigned* p, unsigned v) {
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void reds_release(unsigned* p, unsigned v) {
    asm volatile("red.release.cta.shared::cta.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

struct ChainShared {
    ChainItem item[CHAIN_SLOTS];
    unsigned finished[CHAIN_SLOTS];   // warps done with the slot's item
    unsigned freed[CHAIN_SLOTS];      // times the slot was announced
    unsigned published;               // items published
    unsigned unit;                    // next warp unit to take
    unsigned stop;                    // the feeding warp has no more items (or gave up)
};

// NW compute warps, then the feeding warp, then the announcing warp.
template <int NW, typename Work>
__device__ __forceinline__ void chain_run(const KParams& kp, const ChainParams& cp, Work&& work) {
    __shared__ ChainShared sh;
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned* done = cp.sync + CHAIN_COUNTERS;
    if (threadIdx.x < CHAIN_SLOTS) { sh.finished[threadIdx.x] = 0; sh.freed[threadIdx.x] = 0; }
    if (threadIdx.x == 0) { sh.published = 0; sh.unit = 0; sh.stop = 0; }
    __syncthreads();
    const unsigned U = cp.U;
    if (wid < NW) {
        for (;;) {
            unsigned u = 0;
            if (lane == 0) u = atomicAdd(&sh.unit, 1u);
            u = __shfl_sync(0xffffffffu, u, 0);
            const unsigned q = cp.Ud.div(u), b = u - q * U;
            bool more = true;
            while ((int)(lds_acquire(&sh.published) - q) <= 0) {
                if (lds_acquire(&sh.stop) != 0u && (int)(lds_acquire(&sh.published) - q) <= 0) { more = false; break; }
                __nanosleep(32);
            }
            if (!__all_sync(0xffffffffu, more)) break;
            const unsigned slot = q % CHAIN_SLOTS;
            const ChainItem im = sh.item[slot];
            const unsigned g = (unsigned)im.b * U + b;
            const unsigned row = cp.sw.div(g);
            const int i = im.p0 + (int)(g - row * cp.sw.d);
            const unsigned y = (unsigned)im.tile * cp.R + row;
            if (row < cp.R && y < (unsigned)kp.ny && i >= 0 && i < (int)cp.ns && im.n < cp.nsteps) {
                int seg = i + im.turn;
                while (seg >= (int)cp.ns) seg -= (int)cp.ns;
                work(((cp.odd0 + im.n) & 1) != 0, seg, (int)y, im.z);
            }
            __syncwarp();
            if (lane == 0) reds_release(&sh.finished[slot], 1u);
        }
        return;
    }
    if (wid == NW) {
        // feeding warp: tickets, dependencies, publication
        const unsigned grp = lane / 9u, k = lane - grp * 9u;   // item of the group, neighbour
        const int dz = (int)(k / 3u) - 1, dy = (int)(k % 3u) - 1;
        const unsigned long long limit = cp.limit_ns;
        ChainItem im, nx;
        const unsigned *dep, *ndep;
        // the item of this lane's group in tickets t ..., and the counter of its
        // neighbour k
        auto look = [&](unsigned t, ChainItem& it, const unsigned*& d) {
            it = chain_decode(cp, grp < CHAIN_GRP ? t + grp : cp.total);
            d = nullptr;
            if (it.n < 0 || it.nu == 0) return;
            int zz = it.z + dz, yy = it.tile + dy;
            bool use = true;
            if (zz < 0 || zz >= kp.nz) {
                use = (kp.flags & LBM_FLAG_PERIODIC_Z) != 0;
                zz = zz < 0 ? zz + kp.nz : zz - kp.nz;
            }
            yy = yy < 0 ? yy + (int)cp.M.d : (yy >= (int)cp.M.d ? yy - (int)cp.M.d : yy);
            if (use) d = done + ((unsigned)zz * cp.M.d + (unsigned)yy);
        };
        auto draw = [&]() -> unsigned {
            return lane == 0 ? atomicAdd(cp.sync, (unsigned)CHAIN_GRP) : 0u;
        };
        unsigned t = __shfl_sync(0xffffffffu, draw(), 0);
        unsigned next = draw();
        look(t, nx, ndep);
        while (t < cp.total) {
            im = nx;
            dep = ndep;
            const unsigned need = (unsigned)im.nu * cp.bpt.d;
            // the next group's tickets are drawn before this group's counters are
            // read: an acquiring load holds back what follows it
            t = __shfl_sync(0xffffffffu, next, 0);
            next = draw();
            look(t, nx, ndep);
            unsigned have = need;
            if (dep) have = ld_acquire(dep);
            bool ok = (int)(have - need) >= 0;
            unsigned left = __ballot_sync(0xffffffffu, im.n >= 0 && grp < CHAIN_GRP);   // lanes of items to publish
            const unsigned long long t0 = chain_ns();
            bool fail = false;
            for (unsigned spin = 0; left; ++spin) {
                if (spin > 0) ok = ok || (int)(ld_acquire(dep) - need) >= 0;
                const unsigned okm = __ballot_sync(0xffffffffu, ok);
#pragma unroll
                for (int gi = 0; gi < CHAIN_GRP; ++gi) {
                    const unsigned m = 0x1ffu << (9 * gi);
                    if ((left & m) && (okm & m) == m) {
                        // a free slot: its last item was announced
                        const unsigned q = lds_acquire(&sh.published), slot = q % CHAIN_SLOTS;
                        while (lds_acquire(&sh.freed[slot]) < q / CHAIN_SLOTS ||
                               (int)(q * U - lds_acquire(&sh.unit)) > (int)(CHAIN_AHEAD * U)) {
                            if (chain_ns() - t0 > limit) { fail = true; break; }
                        }
                        __syncwarp();
                        if (!__any_sync(0xffffffffu, fail) && lane == 9u * gi) {
                            sh.item[slot] = im;
                            sts_release(&sh.published, q + 1u);
                        }
                        __syncwarp();
                        left &= ~m;
                    }
                }
                if ((spin & 63u) == 63u &&
                    (ld_acquire(cp.sync + 1) != 0u || chain_ns() - t0 > limit))
                    fail = true;
                if (__any_sync(0xffffffffu, fail)) { fail = true; break; }
            }
            if (__any_sync(0xffffffffu, fail)) {
                if (lane == 0) {
                    atomicOr(kp.devflags, LBM_DEVFLAG_TIMEOUT);
                    atomicExch(cp.sync + 1, 1u);
                }
                break;
            }
        }
        __syncwarp();
        if (lane == 0) sts_release(&sh.stop, 1u);
    } else {
        // announcing warp: lane l watches slot l
        unsigned seen = 0;   // announcements of the lane's slot
        for (;;) {
            const unsigned stop = lds_acquire(&sh.stop);
            const unsigned pub = lds_acquire(&sh.published);
            const unsigned mine = pub / CHAIN_SLOTS + (lane < pub % CHAIN_SLOTS ? 1u : 0u);
            const bool full = seen < mine && lds_acquire(&sh.finished[lane]) == U;
            if (__any_sync(0xffffffffu, full)) {
                const ChainItem im = sh.item[lane];
                fence_gpu();
                if (full) {
                    red_add(done + ((unsigned)im.z * cp.M.d + (unsigned)im.tile), 1u);
                    sh.finished[lane] = 0;
                    ++seen;
                    sts_release(&sh.freed[lane], seen);
                }
                __syncwarp();
            } else {
                if (__all_sync(0xffffffffu, stop != 0u && seen == mine)) break;
                __nanosleep(32);
            }
        }
    }
}

// Host side.  Warp units are segments of 64 nodes; 14 computing warps per block
// at 128 registers (lbm_bgk.cu).
constexpr int CHAIN_WARPS = 14;
constexpr int CHAIN_UNIT = 64;
constexpr int CHAIN_THREADS = 32 * (CHAIN_WARPS + CHAIN_HELPERS);

// Plans a chain of up to nsteps steps on a device of `sms` SMs (lbm_aux.cu); also
// read by lbm_step_plan.  Returns the steps planned (whole sweeps), 0 when they are
// better launched one by one or no chain kernel serves the kind of box.
struct ChainPlan {
    ChainParams p;      // p.sync is the launcher's to set
    unsigned grid;
};
int chain_plan(const KParams& kp, Kind k, unsigned sms, int nsteps, bool odd, ChainPlan& out);

// The plan on the current device, with its counters in the staging buffer of
// lbm_set_scalar (whose contents are not kept between calls), zeroed on the stream
// (LBM_FLAG_TEST_STALL: the first tile's starts one short, and is never full).
cudaError_t chain_prepare(const KParams& kp, Kind k, const Views& v, int nsteps, bool odd,
                          ChainPlan& out, int& done, cudaStream_t st);

}  // namespace lbmgpu
