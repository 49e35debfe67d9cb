// Host side of the multi-step kernel (stepper_march.cuh): which calls take it, and the parameters of
// its order.
#include "internal.h"
#include "launch.h"
#include "level_args.cuh"
#include "stepper_march.cuh"

namespace mclbm {

cudaError_t launch_march_f32(MarchArgs<float>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s);
cudaError_t launch_march_f16(MarchArgs<__half>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s);
cudaError_t launch_march_f64(MarchArgs<double>& a, int vec, int mode, int num_sms, int64_t tiles, cudaStream_t s);

namespace {

// L2 that the tiles in work may take.  GB300's 129 MB also hold lines on their way out: 64^3 ensembles
// whose lattice fits whole run at full speed up to 100 MB (FP32 AA, copy within L2 13.4 TB/s at 100 MB,
// 11.6 at 160), so 90 MB is kept for the lattice or for the window.
constexpr int64_t kL2Bytes = int64_t(90) << 20;

// Tiles between a tile and the ones of the step before that it waits for, per group of warps: the
// tile in work, the one whose loads are in flight, and the report's way to the hand-out.  Measured at
// 64^3 x 64 and 128^3 x 32 FP32: 2.5 to 5 within 2% of each other, 2 with the window's edge in sight.
constexpr int64_t kDistance2 = 7;  // in halves

// Longest launch without a limit of the caller: about a second of steps, by the slowest step measured (a
// floor for the smallest ensembles, FP32 2.6 to 3 us, FP16 2.4 to 3, FP64 13.9; a rate beyond, D3Q27 FP32 42 and
// FP64 1.2 GLUPS).  The next launch adds 11 us.
int64_t longest_launch(const mclbm_ctx* c)
{
    if (c->step_limit > 0) return c->step_limit;
    const bool f64 = c->cfg.precision == MCLBM_FP64;
    const double floor_ns = f64 ? 14000.0 : 3000.0, nodes_ns = (f64 ? 1.0 : 0.03) * (double)c->M * (double)c->n;
    const double steps = 1e9 / (nodes_ns > floor_ns ? nodes_ns : floor_ns);
    return steps > 2.0 ? (int64_t)steps : 2;
}

int ilog2(int64_t v)
{
    int l = 0;
    while ((int64_t(1) << (l + 1)) <= v) ++l;
    return l;
}

// Fills in the order of `steps` steps; false where no window of two or more steps fits L2.
template <class E>
bool march_order(MarchArgs<E>& a, const mclbm_ctx* c, int vec, int64_t steps)
{
    const int64_t tile = (int64_t)kMarchGroup * vec;
    const int64_t plane = (int64_t)c->N * c->N;
    const int64_t unit = plane > tile ? plane : tile;
    const int64_t tiles = (int64_t)c->M * c->n / tile;
    const int64_t tile_bytes = tile * Q * (int64_t)sizeof(E);
    const int64_t distance = kDistance2 * c->num_sms * kMarchGroups / 2;
    a.logT = ilog2(unit / tile);
    a.logU = ilog2(c->n / unit);
    // chunks of up to 32 tiles: one plane, or several of a small lattice
    a.logC = 0;
    while (a.logC < a.logU && (1u << (a.logC + a.logT)) < 32) ++a.logC;
    const int64_t ct = int64_t(1) << (a.logC + a.logT);
    const int64_t chunks = tiles / ct;
    a.chunks = (unsigned)chunks;
    a.lanes = 1;
    a.lag = 0;
    if (tiles * tile_bytes > kL2Bytes) {
        // Depth: a pass of `lanes` steps crosses HBM once, so from four on HBM is no longer the bound;
        // of 4 to 12 take the one that leaves the fewest lanes idle in the last pass, the deepest of
        // equals; two or three where only they fit.  A chunk's dependences reach one chunk ahead at
        // the step before, two where a chunk is one unit (its last unit needs the next one).
        const int64_t reach = a.logC == 0 ? 2 : 1;
        int64_t best = 0, best_idle = 0;
        for (int64_t lanes = 12; lanes >= 2 && !(best && lanes < 4); --lanes) {
            const int64_t lag = (distance + lanes * ct - 1) / (lanes * ct) + reach;
            if (lanes * lag * ct * tile_bytes > kL2Bytes || chunks < (lanes - 1) * lag + 3) continue;
            const int64_t idle = (steps + lanes - 1) / lanes * lanes - steps;
            if (best == 0 || idle < best_idle) {
                best = lanes;
                best_idle = idle;
                a.lag = (unsigned)lag;
            }
        }
        if (best == 0) return false;
        a.lanes = (unsigned)best;
    }
    const int64_t passes = (steps + a.lanes - 1) / a.lanes;
    const int64_t slots = passes * chunks + (int64_t)(a.lanes - 1) * a.lag;
    if (tiles * (steps + 1) >= (int64_t)1 << 30 || slots * a.lanes * ct >= (int64_t)1 << 31) return false;
    a.steps = (unsigned)steps;
    a.slots = (unsigned)slots;
    return true;
}

// Whether `steps` steps of a context run faster in the multi-step kernel than with a launch per step.
// The kernel's start (counters, cooperative launch, fill and drain) costs about 11 us a call.  It fills the
// SMs it runs on, so contexts on several streams take turns: two FP32 contexts of 32^3 x 3 on two streams
// take 1.5 ms per 200 steps against 1.6 with a launch per step, four 3.1 against 2.5 from one host
// thread and 1.9 from four (one 0.78 against 1.24); from 64^3 on the kernel is faster at any number.  A
// launch of half the blocks leaves room for a second context but costs one alone 22% at 32^3, so
// this is left to mclbm_set_step_limit.
//
// FP32 storage, whose launch per step is at the HBM bound: per step the kernel saves 1 to 2 us below
// 2^16 nodes (4.2 against 2.6 to 3.8 us at 8^3 to 32^3), 3 us at 32^3 x 7 (8.3 against 5.0), 4 us at 64^3
// (10.4 against 5.9), and a third of the time from 64^3 x 2 on (64^3 x 64 381 against 271 us, AA 387 against
// 261; 128^3 x 8 385 against 270).  Three steps: 64^3 x 2 AA 47.9 against 38.9 us, 64^3 34.1 against 30.9
// us, 32^3 x 3 23.3 against 25.1 us.
//
// FP16 storage is bound by arithmetic, in a kernel with twice the nodes per thread (65 against 78 GLUPS
// at 64^3 x 64): here only what is bound by launches, latency and unfilled waves.  6.2 against 2.4 to 3.5 us
// per step up to 32^3, 64^3 8.3 against 5.2, 64^3 x 4 18.5 against 16.0, x 5 22.4 against 20.0, x 8 33.0
// against 31.9, AA 33.9 against 31.3; beyond, waves fill (x 10 39.6 against 40).  D3Q27, whose two nodes
// per thread reach 40 GLUPS: 64^3 x 2 14.4 against 13.2, AA 16.4 against 12.9, 64^3 x 3 20.6 against 19.7,
// AA 22.0 against 19.3, 32^3 x 25 20.6 in both, AA 22.6 against 19.9, 64^3 x 4 AA 25.7 in both.  Twelve
// steps: 64^3 x 8 33.4 against 32.8, D3Q27 64^3 x 3 20.84 against 20.82; six steps of those lose 1 to 5%.
//
// FP64 storage is bound by its pipe: a warp's collision holds a partition for 12 us, so a launch per
// step takes whole multiples of that (32^3: 1024 warps on 608 partitions) and the launch's 2 to 3 us.
// Without a barrier between the steps the partitions fill evenly: 32^3 26.7 -> 25.2 us per step, x 2
// 49.2 -> 39.2, x 3 71.8 -> 58.4, x 4 84.0 -> 77.8, x 8 164 -> 156, x 16 316 -> 312 (x 32 no gain: 627 and
// 625), 16^3 15.9 -> 14.2, 8^3 14.4 -> 13.9; D3Q27 32^3 x 2 69.6 -> 55.7.  Eight steps: 32^3 27.2 against
// 27.2, x 2 49.9 against 41.5, 8^3 15.0 against 15.2.  Rows within one warp only (N <= 32).
bool march_serves(const mclbm_ctx* c, int64_t steps)
{
    if ((c->cfg.options & MCLBM_OPT_EXACT_GAMMA) || c->launch_chosen || c->step_limit == 1) return false;
    const int64_t nodes = (int64_t)c->M * c->n;
    if (c->cfg.precision == MCLBM_FP64) return c->N <= 32 && nodes <= 1 << 19 && steps >= (nodes <= (1 << 15) ? 16 : 8);
    if (c->cfg.precision == MCLBM_FP16) {
        if constexpr (Q == 19) return nodes <= 1 << 20 ? steps >= 6 : steps >= 12 && nodes <= 1 << 21;
        if (nodes <= 1 << 18) return steps >= 6;
        return steps >= 12 && nodes <= (c->cfg.pattern == MCLBM_PULL ? 6 : 7) << 17;
    }
    return steps >= (nodes < (1 << 16) ? 12 : (nodes < (1 << 18) ? 6 : 3));
}

// Nodes per thread.  Four keep more independent work per warp, two halve a tile's latency and spread
// a small ensemble over more warps.  FP32: two up to 64^3 nodes (8^3 3.4 -> 2.6 us per step, 32^3 3.9 ->
// 3.1, 32^3 x 7 5.4 -> 5.0, 64^3 6.3 -> 5.9, but 64^3 x 2 8.9 -> 10.8; D3Q27 32^3 4.9 -> 3.4, 64^3 8.5 ->
// 7.2, 64^3 x 2 12.9 -> 13.9).  FP16: two up to 32^3 x 4 (32^3 3.4 -> 3.0, 32^3 x 7 4.5 -> 4.7), D3Q27, whose
// four and the four ahead spill, always (64^3 x 2 13.5 -> 13.2).  D3Q27 FP32 rows that span warps: two.
int march_vec(int precision, int N, int64_t nodes)
{
    if (precision == MCLBM_FP64) return 1;  // as the launch per step of small ensembles
    if (Q == 27) return precision == MCLBM_FP16 || nodes <= (1 << 18) || N > 128 ? 2 : 4;
    return nodes <= (precision == MCLBM_FP32 ? 1 << 18 : 1 << 17) ? 2 : 4;
}

// Takes `nsteps` steps in mode `mode`; *taken: how many were.  Trajectories: from src through dst,
// dst + hop, ... (elements).
template <class E>
cudaError_t march_t(mclbm_ctx* c, int mode, const void* src, void* dst, int64_t hop, int64_t nsteps, int64_t* taken)
{
    constexpr bool f32 = std::is_same<E, float>::value;
    const int vec = march_vec(c->cfg.precision, c->N, (int64_t)c->M * c->n);
    MarchArgs<E> a;
    memset(&a, 0, sizeof(a));
    const int64_t tiles = (int64_t)c->M * c->n / (kMarchGroup * vec);
    const int64_t most = longest_launch(c) & ~(int64_t)1;  // even: the next launch begins at the same parity
    while (*taken < nsteps) {
        int64_t k = nsteps - *taken < most ? nsteps - *taken : most;
        if (mode == kMarchSwap) k &= ~(int64_t)1;
        if (k < 2 || !march_order(a, c, vec, k)) break;
        const size_t cnt_bytes = sizeof(int) * ((size_t)c->M << a.logU);
        if (cnt_bytes > kPartialBytes) break;
        a.cnt = (int*)(c->work + c->wl.partial);
        a.err = (int*)(c->work + c->wl.flag) + 1;
        fill_level<E>(a.lev, c);
        if (mode == kMarchTrajectory) {
            a.lev.src = *taken == 0 ? (const E*)src : (const E*)dst + (*taken - 1) * hop;
            a.lev.dst = (E*)dst + *taken * hop;
            a.hop = hop;
        } else {
            a.lev.dst = (E*)lattice_ptr(c, mode == kMarchSwap ? c->cur : 0);
            if (mode == kMarchSwap) a.lev.parity = 1;
        }
        cudaError_t e = cudaMemsetAsync(a.cnt, 0, cnt_bytes, c->stream);
        if (e != cudaSuccess) return e;
        if constexpr (std::is_same<E, double>::value)
            e = launch_march_f64(a, vec, mode, c->num_sms, tiles, c->stream);
        else if constexpr (f32)
            e = launch_march_f32(a, vec, mode, c->num_sms, tiles, c->stream);
        else
            e = launch_march_f16(a, vec, mode, c->num_sms, tiles, c->stream);
        // part of the GPU only, or a build whose registers do not allow the kernel's split: launch by launch
        if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidConfiguration) {
            cudaGetLastError();
            break;
        }
        if (e != cudaSuccess) return e;
        *taken += k;
        c->multi_launches += 1;
        c->multi_steps += k;
    }
    return cudaSuccess;
}

cudaError_t march_any(mclbm_ctx* c, int mode, const void* src, void* dst, int64_t hop, int64_t nsteps, int64_t* taken)
{
    switch (c->cfg.precision) {
        case MCLBM_FP64: return march_t<double>(c, mode, src, dst, hop, nsteps, taken);
        case MCLBM_FP32: return march_t<float>(c, mode, src, dst, hop, nsteps, taken);
        default: return march_t<__half>(c, mode, src, dst, hop, nsteps, taken);
    }
}

}  // namespace

bool march_serves_call(const mclbm_ctx* c, int64_t nsteps)
{
    return march_serves(c, c->cfg.pattern == MCLBM_PULL ? nsteps & ~(int64_t)1 : nsteps);
}

// Takes steps of a call for `nsteps` steps in the multi-step kernel, where it serves the context;
// *taken is the number taken (the caller takes the others launch by launch).
cudaError_t launch_march(mclbm_ctx* c, int64_t nsteps, int64_t* taken)
{
    *taken = 0;
    const int mode = c->cfg.pattern == MCLBM_PULL ? kMarchSwap : kMarchAA;
    if (!march_serves_call(c, nsteps)) return cudaSuccess;
    const cudaError_t e = march_any(c, mode, nullptr, nullptr, 0, nsteps, taken);
    c->steps += *taken;
    return e;
}

// The same for pull steps from the lattice src through the lattices at dst, dst + hop_bytes, ..., each
// of which keeps its state; the context's own state is not touched.
cudaError_t launch_march_trajectory(mclbm_ctx* c, const void* src, void* dst, size_t hop_bytes, int64_t nsteps,
                                    int64_t* taken)
{
    *taken = 0;
    if (!march_serves(c, nsteps)) return cudaSuccess;
    const int64_t hop = (int64_t)(hop_bytes / c->elem_bytes);
    return march_any(c, kMarchTrajectory, src, dst, hop, nsteps, taken);
}

}  // namespace mclbm
