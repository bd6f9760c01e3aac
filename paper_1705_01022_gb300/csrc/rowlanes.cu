// Launches of the row-lane device step (rowlanes.cuh).
//
// Two forms.  A lattice of at most kBlockWarps warps runs all its MCS in one
// launch of one block, with the lattice in shared memory.  Larger ones take one
// launch per device step, each started while the one before writes back
// (programmatic dependent launch): the draws, which do not depend on the lattice,
// run before the wait for it.  A cluster of eight blocks for lattices in between
// was slower than the launches (L=1024, p=0.95, q=0.05, 8 MCS and a W^2: 309 and
// 253 us): its few SMs share more warps each.
#include "oct_internal.h"

#include "rowlanes.cuh"
#include "tiles.cuh"

namespace oct {
namespace {

// Warps per block of a device-step launch: one while they still find free
// places, so that the blocks spread evenly over the schedulers, else four.  8 MCS
// and a W^2, us with one and with four, p=0.95, q=0.05: L=1536 280, 284; L=4096
// 347, 378; L=6144 (2304 warps) 511, 540; L=7168 (3136) 667, 680; L=8192 (4096)
// 828, 730; KPZ: 147, 166; 215, 246; 338, 354; 437, 474; 451, 468.
constexpr uint32_t kRowWarps = 4;
constexpr uint32_t kRowSingleMax = 152u * 20u;   // warps of a step in one-warp blocks
// One block up to a warp per scheduler: 8 MCS and a W^2 at L=256 KPZ 135 us,
// 149 with launches.
constexpr uint32_t kBlockWarps = 4;
// Its lattice in bytes at most: a lane holds 128 sites, a step a quarter of the
// sites, four sites a byte (L <= 256).  With the warps' own areas it stays below
// the 48 KB that a launch may take without raising its limit.
constexpr uint32_t kBlockLattice = kBlockWarps * 32u * 128u;
static_assert(kBlockLattice + kBlockWarps * row_smem_words<true>() * 4u <= 48u * 1024u, "within the default limit");

template <bool RANDOM, int SPEC, bool ONE, bool SHARED = false, class Ready, class Done>
__device__ __forceinline__ void row_step(const StepArgs &a, uint32_t *lat, uint32_t warp, uint32_t t, uint32_t k, uint32_t *sm,
                                         int &net, int &draws, int &tails, Ready ready, Done done) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t S = ONE ? 32u : row_segment(a.GX, a.By), per_warp = 32u / S;
    const uint32_t seg = lane / S, sub = lane % S, w = warp * per_warp + seg, n_tiles = work_tiles(a);
    const TilePlace pl = place_tile(a, w < n_tiles ? w : 0u, t, k);
    RowLane rl;
    rl.GX = static_cast<int>(a.GX);
    rl.TR = static_cast<int>(a.By / 4u);
    rl.gx = static_cast<int>(sub % a.GX);
    rl.tr = static_cast<int>(sub / a.GX);
    rl.m = static_cast<uint32_t>(rl.tr) & 3u;
    rl.active = rl.tr < rl.TR && w < n_tiles;
    LaneCtx<KeysConst> c;
    c.t = t;
    c.k = k;
    c.T = pl.T;
    c.g = (static_cast<uint32_t>(rl.tr) >> 2) * a.GX + static_cast<uint32_t>(rl.gx);
    rl.gw = seg * (S / 4u) + c.g;
    c.key.a = &a;
    c.first_round();
    c.thr_p = a.thr_p;
    c.thr_q = a.thr_q;
    c.p_always = a.p_always;
    c.q_always = a.q_always;
    c.p_random = a.p_random;
    c.q_random = a.q_random;
    int n = 0, d = 0, b = 0;
    run_rows<RANDOM, SPEC, ONE, SHARED>(lat, a.L, a.plane_rows, a.wpr, pl.x0, pl.y0, c, rl, sm, n, d, b, ready, done);
    if (rl.active) {
        net += n;
        draws += d;
        tails += b;
    }
}

template <bool RANDOM>
__device__ __forceinline__ void row_counters(const StepArgs &a, uint32_t warp, int net, int draws, int tails) {
    const uint32_t lane = threadIdx.x & 31u;
    const int total = __reduce_add_sync(kFull, net);
    if (lane == 0 && total != 0)
        atomicAdd(&a.net[warp % kNetSlots], static_cast<unsigned long long>(static_cast<long long>(total)));
    if (RANDOM) {
        const unsigned nd = __reduce_add_sync(kFull, static_cast<unsigned>(draws));
        if (lane == 0 && nd != 0u) atomicAdd(&a.draws[warp % kNetSlots], static_cast<unsigned long long>(nd));
        const unsigned nb = __reduce_add_sync(kFull, static_cast<unsigned>(tails));
        if (lane == 0 && nb != 0u) atomicAdd(&a.tails[warp % kNetSlots], static_cast<unsigned long long>(nb));
    }
}

template <bool RANDOM, int SPEC, bool ONE, uint32_t WARPS>
__global__ void __launch_bounds__(WARPS * 32) row_step_kernel(const __grid_constant__ StepArgs a) {
    __shared__ __align__(16) uint32_t sm[WARPS * row_smem_words<RANDOM>()];
    const uint32_t S = ONE ? 32u : row_segment(a.GX, a.By);
    const uint32_t warp = blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (warp * (32u / S) >= work_tiles(a)) return;  // the whole warp leaves together
    int net = 0, draws = 0, tails = 0;
    row_step<RANDOM, SPEC, ONE>(a, a.lat, warp, *a.t_ptr + a.dt, a.k, sm + (threadIdx.x >> 5) * row_smem_words<RANDOM>(), net,
                                draws, tails, [] { wait_for_previous_grid(); }, [] { launch_dependents(); });
    row_counters<RANDOM>(a, warp, net, draws, tails);
}

// n MCS of a lattice that one block holds in shared memory.
template <bool RANDOM, int SPEC, bool ONE>
__global__ void __launch_bounds__(kBlockWarps * 32)
    row_block_kernel(const __grid_constant__ StepArgs a, uint32_t *t_out, uint32_t n) {
    extern __shared__ __align__(16) uint32_t row_block_smem[];
    const uint32_t words = a.L * a.wpr * 2u, warp = threadIdx.x >> 5;
    uint32_t *const lat = row_block_smem + (blockDim.x >> 5) * row_smem_words<RANDOM>();
    uint32_t *const sm = row_block_smem + warp * row_smem_words<RANDOM>();
    for (uint32_t i = 4u * threadIdx.x; i < words; i += 4u * blockDim.x)
        *reinterpret_cast<uint4 *>(lat + i) = *reinterpret_cast<const uint4 *>(a.lat + i);
    const uint32_t t0 = *a.t_ptr;
    int net = 0, draws = 0, tails = 0;
    for (uint32_t i = 0; i < n; ++i)
        for (uint32_t k = 0; k < 4u; ++k)
            row_step<RANDOM, SPEC, ONE, true>(a, lat, warp, t0 + i, k, sm, net, draws, tails, [] { __syncthreads(); },
                                              [] {});
    __syncthreads();
    for (uint32_t i = 4u * threadIdx.x; i < words; i += 4u * blockDim.x)
        *reinterpret_cast<uint4 *>(a.lat + i) = *reinterpret_cast<const uint4 *>(lat + i);
    if (threadIdx.x == 0u) *t_out = t0 + n;
    row_counters<RANDOM>(a, warp, net, draws, tails);
}

uint32_t row_warps(const StepArgs &a) {
    const uint32_t per = 32u / row_segment(a.GX, a.By);
    return (work_tiles(a) + per - 1u) / per;
}

template <bool RANDOM, int SPEC, bool ONE>
cudaError_t launch_row_step_as(const StepArgs &a, bool overlap, cudaStream_t st) {
    const uint32_t warps = row_warps(a);
    if (warps <= kRowSingleMax)
        return launch_overlapped(row_step_kernel<RANDOM, SPEC, ONE, 1u>, dim3(warps), dim3(32u), overlap, st, a);
    return launch_overlapped(row_step_kernel<RANDOM, SPEC, ONE, kRowWarps>, dim3((warps + kRowWarps - 1u) / kRowWarps),
                             dim3(kRowWarps * 32u), overlap, st, a);
}

template <bool RANDOM, int SPEC, bool ONE>
cudaError_t launch_row_run_as(const StepArgs &a, uint32_t *t_out, uint32_t n, cudaStream_t st) {
    const uint32_t warps = row_warps(a), smem = a.L * a.wpr * 8u + warps * row_smem_words<RANDOM>() * 4u;
    row_block_kernel<RANDOM, SPEC, ONE><<<1, warps * 32u, smem, st>>>(a, t_out, n);
    return cudaGetLastError();
}

}  // namespace

bool rows_take(const StepArgs &a) {
    return a.scheme == 0u && a.cx == 4u && a.cy == 4u && (a.GX & (a.GX - 1u)) == 0u && a.GX * (a.By / 4u) <= 32u &&
           row_warps(a) <= kRowWarpsMax;
}

bool rows_fit_block(const StepArgs &a) { return row_warps(a) <= kBlockWarps; }

#define OCT_ROWS(FN, ...)                                                                                \
    do {                                                                                                 \
        const bool one = row_segment(a.GX, a.By) == 32u;                                                 \
        if (!any_random && a.p_always == 0xFFFFFFFFu && a.q_always == 0u)                                \
            return one ? FN<false, 1, true>(__VA_ARGS__) : FN<false, 1, false>(__VA_ARGS__);             \
        if (any_random && a.p_random && a.q_random && !ties_matter(a.thr_p, a.thr_q))                    \
            return one ? FN<true, 3, true>(__VA_ARGS__) : FN<true, 3, false>(__VA_ARGS__);               \
        if (any_random && a.p_random && a.q_random)                                                      \
            return one ? FN<true, 2, true>(__VA_ARGS__) : FN<true, 2, false>(__VA_ARGS__);               \
        if (any_random) return one ? FN<true, 0, true>(__VA_ARGS__) : FN<true, 0, false>(__VA_ARGS__);   \
        return one ? FN<false, 0, true>(__VA_ARGS__) : FN<false, 0, false>(__VA_ARGS__);                 \
    } while (0)

cudaError_t launch_row_step(const StepArgs &a, bool any_random, bool overlap, cudaStream_t st) {
    OCT_ROWS(launch_row_step_as, a, overlap, st);
}

cudaError_t launch_row_run(const StepArgs &a, bool any_random, uint32_t *t_out, uint32_t n, cudaStream_t st) {
    OCT_ROWS(launch_row_run_as, a, t_out, n, st);
}
#undef OCT_ROWS

}  // namespace oct
