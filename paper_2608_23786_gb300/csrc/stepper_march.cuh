// Several steps of an ensemble in one launch, ordered so that a step finds its input in L2.
//
// A launch per step streams the whole ensemble from HBM once per step (2 Q b bytes per node and
// step), however many steps a call asks for.  The samples are independent and a step reaches one
// plane into its neighbours, so a region can take several steps while it is in the 129 MB L2: this
// kernel walks the (step, region) pairs in a skewed order, `lanes` steps deep, in which step k
// follows step k - 1 at a distance of `lag` chunks of planes.  Per pass of `lanes` steps the state
// crosses HBM once; the other accesses are served by L2.
//
// Order.  A tile is BLOCK * VEC consecutive nodes (whole rows, or whole planes of a small
// lattice), a unit one plane (or one tile where a tile holds several planes), a chunk 2^logC units
// of one sample; the chunks of all samples form one sequence of `chunks`.  The work is a sequence of
// slots, slot s holding for every lane k the chunk s - k lag (mod chunks: the next pass follows
// without a gap) at step pass * lanes + k.  At step a the units of a sample are taken in order from
// unit a on (periodic), so that the units a chunk depends on at the step before (its own, the one
// before and the one after) are all in the same chunk or the next (two) of that sample's sequence,
// which earlier slots hold.  Tiles are dealt to the blocks of a persistent grid in this order.
//
// In place.  The steps alternate between the two parities of the AA pattern, so one lattice is all
// that the steps touch.  A pull lattice (f_i(x, t) in slot i of x - c_i) is the odd-time AA lattice with
// the slots of opposite velocities exchanged (SWAP): an odd-type step and an even-type step take it to
// the pull lattice two steps on, in place.  So pull contexts take an even number of steps here, in the
// lattice that holds their state, and half the L2 that two lattices would need.
//
// Trajectories.  The adjoint keeps every state of a segment: there each step reads the pull lattice of the
// state before and writes the next one's (kMarchTrajectory); what a step reads is still in L2, so
// the states cross HBM once, outwards.
//
// Dependences.  cnt[sample][unit] counts the tiles finished, over all steps.  A tile at step a may
// start when its unit and the two next to it have finished a * tiles_per_unit tiles: what it reads
// is then written, and the slots it overwrites are no longer read.  The tile with the lowest position
// in the order among the unfinished ones never waits, and a group of warps waits only when it has
// finished every tile of its own before, so the launch makes progress as long as its blocks are
// resident together (a cooperative launch, which starts when all of them fit: with 20 SMs held by another
// stream for 2.5 s it started then, and ended as usual).  Every wait is bounded, in time and in looks, and
// records MCLBM_ERR_TIMEOUT, which the calls that return results report.
//
// Roles.  Eight warps of a block collide, in two groups of four that each work on their own tiles.
// Of the four warps of the third warp group, two look at the counters of a group's next tile and hand
// the tile out through shared memory when it may start, and two report the tiles whose four warps
// have arrived: only they wait for the fence that makes a report a release (with the colliding warps
// reporting in turn, that wait took a quarter of the rate: 69 -> 52 GLUPS at 64^3 x 2, L2-resident).
// As in k_step_prefetch, a warp issues the loads of its next run before it collides the current one,
// when that tile has been handed out; otherwise it finishes its current tile first.  What other
// blocks stored is read with coherent loads (ld_cg).
#pragma once
#include "stepper_async.cuh"
#include "stepper_impl.cuh"
#include "stepper_staged.cuh"

namespace mclbm {

constexpr int kMarchGroup = 128;                 // threads of a group (one tile at a time)
constexpr int kMarchGroups = 2;                  // groups of a block
constexpr int kMarchThreads = (kMarchGroups + 1) * kMarchGroup;
// Registers a thread: at launch (384 threads of 168 fill the SM), and after the split, of the colliding
// warps and of the warp group that keeps the books (2 x 240 + 24 = 3 x 168; with 232 and 40 the FP32
// kernel spills 13 words in its main loop and runs at 58 instead of 61 GLUPS at 64^3 x 64).
constexpr int kMarchRegs = 168, kMarchRegsWork = 240, kMarchRegsBooks = 24;
static_assert(kMarchGroups * kMarchRegsWork + kMarchRegsBooks == (kMarchGroups + 1) * kMarchRegs,
              "a split takes no more registers than the launch has");
constexpr int kMarchAhead = 4;                   // tiles handed out beyond the last one reported
// Pause between two looks of the warps that keep the books: without it they take issue slots from the
// colliding warps of their partition (pull 64^3 x 64 61.5 -> 62.1 GLUPS, in another build 59.0 -> 62.1).
constexpr unsigned kMarchNapNs = 64;
// A wait gives up after 1 s of %globaltimer time and this many looks: a launch that was switched out for a
// second has looked a few times since, one that makes no progress a million times.
constexpr uint64_t kMarchLimitNs = 1000ull * 1000 * 1000;
constexpr unsigned kMarchLimitLooks = 1u << 16;

// What a step reads and writes: the AA pattern in place, the same with the slots of opposite velocities
// exchanged (a pull lattice), or pull from one lattice to the next.
enum MarchMode { kMarchAA = 0, kMarchSwap = 1, kMarchTrajectory = 2 };

template <class E>
struct MarchArgs {
    LevelArgs<E> lev;  // dst: the lattice; parity: of the first step (pull lattices: 1).  Trajectories: src
                       // the first state, dst the second
    int64_t hop;       // trajectories: elements from a state's lattice to the next one's, from the second on
    unsigned steps;
    unsigned lanes, lag;
    unsigned logT;  // tiles per unit
    unsigned logU;  // units per sample
    unsigned logC;  // units per chunk
    unsigned chunks;
    unsigned slots;
    int* cnt;  // [M][units], zero at launch
    int* err;
};

struct MarchTile {
    unsigned ctr;   // sample * units + unit
    unsigned tile;  // tile within the unit
    unsigned step;
    bool valid;
};

// Walks a group's tiles: positions first, first + stride, ... of the order.
struct MarchWalk {
    unsigned w, k, s, pass, slot;     // tile of the chunk, lane, slot (mod chunks), pass, slot
    unsigned dw, dk, ds;              // the stride in the same digits
};

template <class E>
__host__ __device__ __forceinline__ MarchWalk march_begin(const MarchArgs<E>& a, unsigned first, unsigned stride)
{
    const unsigned logct = a.logC + a.logT, ct = 1u << logct;
    MarchWalk p;
    p.dw = stride & (ct - 1);
    p.dk = (stride >> logct) % a.lanes;
    p.ds = (stride >> logct) / a.lanes;
    p.w = first & (ct - 1);
    p.k = (first >> logct) % a.lanes;
    p.slot = (first >> logct) / a.lanes;
    p.pass = p.slot / a.chunks;
    p.s = p.slot % a.chunks;
    return p;
}

template <class E>
__host__ __device__ __forceinline__ MarchTile march_next(const MarchArgs<E>& a, MarchWalk& p)
{
    const unsigned logct = a.logC + a.logT;
    const unsigned logP = a.logU - a.logC;  // chunks per sample
    MarchTile t;
    for (;;) {
        t.valid = p.slot < a.slots;
        const unsigned back = p.k * a.lag;
        const bool wrapped = p.s < back;
        const unsigned c = wrapped ? p.s + a.chunks - back : p.s - back;
        t.step = (p.pass - (wrapped ? 1u : 0u)) * a.lanes + p.k;  // before the first chunk: above any step
        const unsigned m = c >> logP;
        const unsigned pos = ((c & ((1u << logP) - 1)) << a.logC) + (p.w >> a.logT);
        t.ctr = (m << a.logU) + ((pos + t.step) & ((1u << a.logU) - 1));
        t.tile = p.w & ((1u << a.logT) - 1);
        p.w += p.dw;
        p.k += p.dk + (p.w >> logct);
        p.w &= (1u << logct) - 1;
        unsigned up = p.ds;
        if (p.k >= a.lanes) {
            p.k -= a.lanes;
            ++up;
        }
        p.slot += up;
        p.s += up;
        while (p.s >= a.chunks) {
            p.s -= a.chunks;
            ++p.pass;
        }
        if (!t.valid || t.step < a.steps) return t;
    }
}

// Whether phase `parity` of a barrier has completed (does not wait).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ int ld_acquire_gpu(const int* p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_add_relaxed_gpu(int* p, int v)
{
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire_cta(uint32_t p)
{
    int v;
    asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta(uint32_t p, int v)
{
    asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}

// The lattice that step k reads (trajectories; k == steps: the last one written).
template <class E>
__device__ __forceinline__ E* march_state(const MarchArgs<E>& a, unsigned k)
{
    return k == 0 ? const_cast<E*>(a.lev.src) : a.lev.dst + (int64_t)(k - 1) * a.hop;
}

template <class E, int VEC>
__device__ __forceinline__ RunLoc march_run(const MarchArgs<E>& a, const MarchTile& t)
{
    const Geom& g = a.lev.g;
    const unsigned um = (1u << a.logU) - 1;
    RunLoc p;
    p.l = 0;
    p.m = (int)(t.ctr >> a.logU);
    const unsigned node = (((t.ctr & um) << a.logT) + t.tile) * (unsigned)(kMarchGroup * VEC) + (threadIdx.x & (kMarchGroup - 1)) * VEC;
    p.node = node;
    p.x0 = (int)(node & (g.N - 1));
    p.y = (int)((node >> g.logN) & (g.N - 1));
    p.z = (int)(node >> (2 * g.logN));
    p.mode = (a.lev.parity + t.step) & 1 ? 2 : 1;
    return p;
}

struct MarchShared {
    uint64_t bar[kMarchGroups][kMarchAhead];  // arrivals of a tile's four warps
    MarchTile tile[kMarchGroups][2 * kMarchAhead];
    int out[kMarchGroups];       // tiles handed out (the last of them may be the end mark)
    int reported[kMarchGroups];  // tiles reported
    int last[kMarchGroups];      // the group's number of tiles, once known (else -1)
};

// Gives up a wait after `looks` looks since t0: true past both limits (recorded in the error word) or once
// the error word is set.
__device__ __forceinline__ bool march_give_up(uint64_t t0, unsigned looks, int* err)
{
    if (*(volatile const int*)err != 0) return true;
    if (looks < kMarchLimitLooks || global_ns() - t0 <= kMarchLimitNs) return false;
    atomicExch(err, kTimeoutCode);
    return true;
}

// Hands out the tiles of group g (one warp; lanes 0, 1 and 2 look at a tile's three counters).
template <class E>
__device__ __forceinline__ void march_hand_out(const MarchArgs<E>& a, MarchShared& sh, int g)
{
    const int lane = threadIdx.x & 31;
    const unsigned um = (1u << a.logU) - 1;
    const uint32_t out = smem_u32(&sh.out[g]), reported = smem_u32(&sh.reported[g]);
    MarchWalk walk = march_begin(a, blockIdx.x + g * gridDim.x, kMarchGroups * gridDim.x);
    for (int n = 0;; ++n) {
        const MarchTile t = march_next(a, walk);
        const int* c = a.cnt + ((t.ctr & ~um) | ((t.ctr + lane + um) & um));
        const int need = (int)(t.step << a.logT);
        const uint64_t t0 = global_ns();
        bool room = false;
        for (unsigned it = 1;; ++it) {
            if (!room) room = n < ld_acquire_cta(reported) + kMarchAhead;
            bool go = room;
            if (go && t.valid && lane < 3) go = ld_acquire_gpu(c) >= need;
            if (__all_sync(0xffffffffu, go)) break;
            __nanosleep(kMarchNapNs);
            if ((it & 63) == 0 && __any_sync(0xffffffffu, lane == 0 && march_give_up(t0, it, a.err))) return;
        }
        // Lanes 0, 1 and 2 each acquired one counter; a vote orders no memory, so without this lane 0's
        // release would not carry what lanes 1 and 2 acquired.
        __syncwarp();
        if (lane == 0) {
            sh.tile[g][n & (2 * kMarchAhead - 1)] = t;
            if (!t.valid) st_release_cta(smem_u32(&sh.last[g]), n);
            st_release_cta(out, n + 1);
        }
        __syncwarp();
        if (!t.valid) return;
    }
}

// Reports the finished tiles of group g (one thread).
template <class E>
__device__ __forceinline__ void march_report(const MarchArgs<E>& a, MarchShared& sh, int g)
{
    const uint32_t bar = smem_u32(&sh.bar[g][0]);
    for (int n = 0;; ++n) {
        const uint64_t t0 = global_ns();
        for (unsigned it = 1; !mbar_test(bar + 8 * (n & (kMarchAhead - 1)), (n / kMarchAhead) & 1); ++it) {
            __nanosleep(kMarchNapNs);
            if ((it & 15) == 0 && ld_acquire_cta(smem_u32(&sh.last[g])) == n) return;
            if ((it & 255) == 0 && march_give_up(t0, it, a.err)) return;
        }
        const unsigned ctr = sh.tile[g][n & (2 * kMarchAhead - 1)].ctr;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        red_add_relaxed_gpu(a.cnt + ctr, 1);
        st_release_cta(smem_u32(&sh.reported[g]), n + 1);
    }
}

// Whether the run ahead waits in shared memory (one cp.async slot a thread, as in k_step_slot) instead of
// registers: D3Q27 FP32, whose run of four nodes and the one ahead do not fit the registers together
// (16-byte copies, which go through L2 only, and no edge words): 64^3 x 16 109 -> 99 us per step against two
// nodes per thread in registers, AA 105 -> 99.
template <class E, int VEC, bool WRAP>
constexpr bool kMarchSlot = Q == 27 && WRAP && sizeof(E) == 4 && VEC == 4;

template <class E, int VEC, bool SLOT>
constexpr int march_smem()
{
    return SLOT ? AsyncRing<E, VEC, kMarchGroups * kMarchGroup, 1>::kVecBytes : 0;
}

// WRAP: rows within one warp.
template <class E, int VEC, int MODE, bool PACK, bool WRAP>
__global__ void __launch_bounds__(kMarchThreads, 1) k_march(const __grid_constant__ MarchArgs<E> a)
{
    using C = typename Storage<E>::compute;
    constexpr bool SWAP = MODE == kMarchSwap, SLOT = kMarchSlot<E, VEC, WRAP>;
    constexpr int kRing = kMarchGroups * kMarchGroup;
    extern __shared__ __align__(16) unsigned char march_dyn[];
    __shared__ MarchShared sh;
    const int lane = threadIdx.x & 31;
    const Geom g = a.lev.g;
    if (threadIdx.x < kMarchGroups * kMarchAhead) mbar_init(smem_u32(&sh.bar[0][0] + threadIdx.x), kMarchGroup / 32);
    if (threadIdx.x < kMarchGroups) {
        sh.out[threadIdx.x] = sh.reported[threadIdx.x] = 0;
        sh.last[threadIdx.x] = -1;
    }
    mbar_fence_init();
    __syncthreads();
    if (threadIdx.x >= kMarchGroups * kMarchGroup) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMarchRegsBooks));
        const int job = (threadIdx.x - kMarchGroups * kMarchGroup) >> 5;  // 0, 1: hand out; 2, 3: report
        if (job < kMarchGroups)
            march_hand_out(a, sh, job);
        else if (lane == 0)
            march_report(a, sh, job - kMarchGroups);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kMarchRegsWork));
    const int grp = threadIdx.x / kMarchGroup;
    const uint32_t bar0 = smem_u32(&sh.bar[grp][0]), out = smem_u32(&sh.out[grp]);
    MarchTile cur{}, nxt{};
    bool have = false;  // cur is loaded
    bool ended = false;
    int j = -1;  // number of cur among the group's tiles (of the last one when !have)
    RawRun<E, VEC> raw[SLOT ? 1 : Q];
    AsyncRing<E, VEC, kRing, 1> ring;
    ring.base = SLOT ? smem_u32(march_dyn) : 0u;
    ring.tid = threadIdx.x;
    for (;;) {
        C v[Q][VEC];
        RunLoc p;
        if (have) {
            p = march_run<E, VEC>(a, cur);
            if constexpr (SLOT) {
                cp_async_wait<0>();
                if constexpr (MODE == kMarchTrajectory)
                    async_finish_all<E, VEC, kRing, 1, 0, WRAP>(march_dyn, 0, threadIdx.x, g, p, lane, v);
                else if (p.mode == 1)
                    async_finish_all<E, VEC, kRing, 1, 1, WRAP>(march_dyn, 0, threadIdx.x, g, p, lane, v);
                else
                    async_finish_all<E, VEC, kRing, 1, 2, WRAP>(march_dyn, 0, threadIdx.x, g, p, lane, v);
                __syncwarp();  // the slot is read before it is refilled
            } else if constexpr (MODE == kMarchTrajectory)
                finish_all<E, VEC, 0, WRAP>(g, p, lane, raw, v);
            else if (p.mode == 1)
                finish_all<E, VEC, 1, WRAP>(g, p, lane, raw, v);
            else
                finish_all<E, VEC, 2, WRAP>(g, p, lane, raw, v);
        }
        bool ok = false;
        if (!ended) {
            ok = __all_sync(0xffffffffu, ld_acquire_cta(out) > j + 1);
            if (!ok && !have) {
                const uint64_t t0 = global_ns();
                for (unsigned it = 1; !ok; ++it) {
                    ok = __all_sync(0xffffffffu, ld_acquire_cta(out) > j + 1);
                    if (!ok && (it & 255) == 0 && __any_sync(0xffffffffu, lane == 0 && march_give_up(t0, it, a.err))) return;
                }
            }
            if (ok) {
                nxt = sh.tile[grp][(j + 1) & (2 * kMarchAhead - 1)];
                ended = !nxt.valid;
                ok = nxt.valid;
            }
        }
        if (ok) {
            const RunLoc q = march_run<E, VEC>(a, nxt);
            const E* src = (MODE == kMarchTrajectory ? march_state(a, nxt.step) : a.lev.dst) + (int64_t)q.m * Q * g.n;
            if constexpr (SLOT) {  // cp.async.cg: through L2, as ld_cg
                if constexpr (MODE == kMarchTrajectory)
                    async_issue_all<E, VEC, kRing, 1, 0, WRAP>(src, g, q, lane, ring, 0);
                else if (q.mode == 1)
                    async_issue_all<E, VEC, kRing, 1, 1, WRAP, SWAP>(src, g, q, lane, ring, 0);
                else
                    async_issue_all<E, VEC, kRing, 1, 2, WRAP, SWAP>(src, g, q, lane, ring, 0);
                cp_async_commit();
            } else if constexpr (MODE == kMarchTrajectory)
                issue_all<E, VEC, 0, WRAP, true>(src, g, q, lane, raw);
            else if (q.mode == 1)
                issue_all<E, VEC, 1, WRAP, true, SWAP>(src, g, q, lane, raw);
            else
                issue_all<E, VEC, 2, WRAP, true, SWAP>(src, g, q, lane, raw);
        }
        if (have) {
            collide_run<E, VEC, PACK>(v, a.lev);
            E* base = (MODE == kMarchTrajectory ? march_state(a, cur.step + 1) : a.lev.dst) + (int64_t)p.m * Q * g.n;
            if constexpr (MODE == kMarchTrajectory)
                scatter_all<E, VEC, 0>(base, g, p.x0, p.y, p.z, lane, v);
            else if (p.mode == 1)
                store_own_opp<E, VEC, SWAP>(base, g, p.node, v);
            else
                scatter_all<E, VEC, 1, WRAP, SWAP>(base, g, p.x0, p.y, p.z, lane, v);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 8 * (j & (kMarchAhead - 1)));
        }
        if (ok) {
            cur = nxt;
            have = true;
            ++j;
        } else {
            have = false;
            if (ended) break;
        }
    }
}

}  // namespace mclbm
