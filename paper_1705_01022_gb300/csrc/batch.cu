// Batched DTrDT: many independent realizations (replicas) of different L, p, q
// advanced together, one device step of every replica per launch.
//
// Each replica is its own DTrDT simulation (its own key, origin, set order
// and lattice; Sec. 3 / 3.1); batching changes only how the work reaches the
// GPU.  The device-step work of all replicas is a list of (replica, device
// tile) items.  A replica whose sub-tile holds G lane groups of 32 x 16
// sites (G = 8 for 64 x 64 sub-tiles, 2 for 32 x 32) takes G consecutive
// lanes, so one warp carries 32/G sub-tiles, possibly of different replicas.
// Items are bucketed by G and by acceptance mode and packed into warp
// descriptors; persistent warps claim descriptors from an atomic queue.
// Because the sub-tiles of one warp draw their own block-level sets, the
// collective step takes the set per lane (step_candidates_rt / step_apply_rt);
// sub-tiles of 32 groups fill a warp alone and take the uniform path.  All
// replicas advance in lock step: one MCS is four device steps, each one launch
// per acceptance mode and warp kind, captured once in a CUDA graph and
// replayed.  A batch too small to fill the chip takes one launch per device step
// for all modes, with a TC row per lane (batch_row_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/oct.h"
#include "grow.h"
#include "oct_internal.h"
#include "overlap.cuh"
#include "rowlanes.cuh"
#include "subtile.cuh"

namespace oct {
namespace {

struct ReplicaDev {
    uint32_t *lat;
    unsigned long long *counters;  // [net flips, acceptance draws]
    uint32_t L, wpr, Bx, By, GX, GY, tiles_x, tiles_y;
    uint32_t k0, k1, thr_p, thr_q;
    uint32_t p_always, q_always, p_random, q_random;
};

struct BatchItem {
    uint32_t rep;
    uint32_t T;
};

struct WarpDesc {
    uint32_t first;  // first item
    uint32_t n;      // items in this warp (32 / G at most)
    uint32_t G;      // lanes per item
    uint32_t GX;     // lane columns per item
    uint32_t kpz;    // row lanes: every item's replica is deposition only (p = 1, q = 0)
};

constexpr int kBatchWarps = 4;
constexpr int kBatchBlocksPerSM = 4;

// LANE_SETS: the warp holds several sub-tiles (fewer than 32 groups each), each
// with its own set draws; otherwise one sub-tile fills the warp and the step
// takes the uniform row-offset path of the plain kernel.
// SCHEME: 0 DTrDT, 4 with deposition only (p = 1, q = 0), 10 with both rates
// strictly inside (0, 1) (the step variants of the plain kernel).
template <bool RANDOM, bool LANE_SETS, int SCHEME>
__global__ void __launch_bounds__(kBatchWarps * 32, kBatchBlocksPerSM)
    batch_step_kernel(const ReplicaDev *reps, const BatchItem *items, const WarpDesc *descs,
                      uint32_t n_descs, const uint32_t *t_of, uint32_t k, uint32_t *queue) {
    __shared__ __align__(16) uint32_t ring[kBatchWarps * 32 * kRingWordsPerLane];
    const int lane = threadIdx.x & 31;
    for (;;) {
        uint32_t di = 0;
        if (lane == 0) di = atomicAdd(queue, 1u);
        di = __shfl_sync(kFull, di, 0);
        if (di >= n_descs) break;  // the whole warp leaves together
        const WarpDesc wd = descs[di];
        const int G = static_cast<int>(wd.G);
        const int slot = lane / G, sub = lane % G;
        const bool active = slot < static_cast<int>(wd.n);
        const BatchItem it = items[wd.first + (active ? slot : 0)];
        const ReplicaDev R = reps[it.rep];
        const uint32_t t = t_of[it.rep];  // this replica's MCS index
        const uint32_t L = R.L;
        const uint4 M = philox4x32_10(t, 0u, 0u, kTagMcs << 28, R.k0, R.k1);
        const uint32_t sigma = static_cast<uint32_t>(perm_element(__umulhi(M.z, 24u), k));
        const uint32_t ty = it.T / R.tiles_x, tx = it.T - ty * R.tiles_x;
        // (an offset plus a place lies below 2L)
        uint32_t x0 = __umulhi(M.x, L) + R.Bx * (2u * tx + (sigma & 1u));
        if (x0 >= L) x0 -= L;
        uint32_t y0 = __umulhi(M.y, L) + R.By * (2u * ty + (sigma >> 1));
        if (y0 >= L) y0 -= L;
        using Keys = std::conditional_t<SCHEME == 4, KeysWeyl, KeysFma>;
        LaneCtx<Keys> c;
        c.GX = static_cast<int>(wd.GX);
        c.GY = G / c.GX;
        c.gx = sub % c.GX;
        c.gy = sub / c.GX;
        c.active = active;
        c.base = lane & ~(G - 1);
        c.t = t;
        c.k = k;
        c.T = it.T;
        c.g = static_cast<uint32_t>(sub);
        c.key = Keys(R.k0, R.k1);
        c.first_round();
        c.thr_p = R.thr_p;
        c.thr_q = R.thr_q;
        c.p_always = R.p_always;
        c.q_always = R.q_always;
        c.p_random = R.p_random;
        c.q_random = R.q_random;
        int net = 0, draws = 0, tails = 0;
        run_subtile<RANDOM, LANE_SETS, SCHEME>(R.lat, L, L, R.wpr, x0, y0, active, c,
                                  ring + ((threadIdx.x >> 5) * 32 + (lane & ~(G - 1))) * kRingWordsPerLane,
                                  net, draws, tails);
        // sum over the G lanes of the item (items start at multiples of G)
        for (int o = G >> 1; o > 0; o >>= 1) {
            net += __shfl_xor_sync(kFull, net, o);
            draws += __shfl_xor_sync(kFull, draws, o);
        }
        if (active && sub == 0) {
            if (net != 0)
                atomicAdd(&R.counters[0], static_cast<unsigned long long>(static_cast<long long>(net)));
            if (RANDOM && draws != 0) atomicAdd(&R.counters[1], static_cast<unsigned long long>(draws));
        }
    }
}

// A batch too small to fill the chip: one device step of every replica in one
// launch, a TC row per lane (rowlanes.cuh), a descriptor per warp.  All modes
// share the launch (two forms of the step: deposition only, and the general
// one), so that no replica waits for another's kernel, and a membership that
// soon changes has no graph to capture (kRowLaunchMcs).  Latency bound like
// rowlanes.cuh: 16 MCS and the W^2 of 64 replicas of L = 64..512 take 0.72 ms.
template <bool RANDOM, int SPEC, bool ONE>
__device__ __forceinline__ void batch_row_item(const ReplicaDev &R, const WarpDesc &wd, uint32_t T, bool held, uint32_t t,
                                               uint32_t k, uint32_t *sm) {
    const uint32_t lane = threadIdx.x & 31u, S = ONE ? 32u : wd.G, seg = lane / S, sub = lane % S;
    const uint32_t L = R.L;
    const uint4 M = philox4x32_10(t, 0u, 0u, kTagMcs << 28, R.k0, R.k1);
    const uint32_t sigma = static_cast<uint32_t>(perm_element(__umulhi(M.z, 24u), k));
    const uint32_t ty = T / R.tiles_x, tx = T - ty * R.tiles_x;
    uint32_t x0 = __umulhi(M.x, L) + R.Bx * (2u * tx + (sigma & 1u));
    if (x0 >= L) x0 -= L;
    uint32_t y0 = __umulhi(M.y, L) + R.By * (2u * ty + (sigma >> 1));
    if (y0 >= L) y0 -= L;
    RowLane rl;
    rl.GX = static_cast<int>(wd.GX);
    rl.TR = static_cast<int>(R.By / 4u);
    rl.gx = static_cast<int>(sub % wd.GX);
    rl.tr = static_cast<int>(sub / wd.GX);
    rl.m = static_cast<uint32_t>(rl.tr) & 3u;
    rl.active = held;
    LaneCtx<KeysWeyl> c;
    c.t = t;
    c.k = k;
    c.T = T;
    c.g = (static_cast<uint32_t>(rl.tr) >> 2) * wd.GX + static_cast<uint32_t>(rl.gx);
    rl.gw = seg * (S / 4u) + c.g;
    c.key = KeysWeyl(R.k0, R.k1);
    c.first_round();
    c.thr_p = R.thr_p;
    c.thr_q = R.thr_q;
    c.p_always = R.p_always;
    c.q_always = R.q_always;
    c.p_random = R.p_random;
    c.q_random = R.q_random;
    int net = 0, draws = 0, tails = 0;
    run_rows<RANDOM, SPEC, ONE, false>(R.lat, L, L, R.wpr, x0, y0, c, rl, sm, net, draws, tails,
                                       [] { wait_for_previous_grid(); }, [] { launch_dependents(); });
    for (uint32_t o = S >> 1; o > 0; o >>= 1) {
        net += __shfl_xor_sync(kFull, net, o);
        if (RANDOM) draws += __shfl_xor_sync(kFull, draws, o);
    }
    if (held && sub == 0) {
        if (net != 0) atomicAdd(&R.counters[0], static_cast<unsigned long long>(static_cast<long long>(net)));
        if (RANDOM && draws != 0) atomicAdd(&R.counters[1], static_cast<unsigned long long>(draws));
    }
}

// Larger batches take the graph's branches, whose lanes of four TC rows need
// fewer instructions per attempt (16 MCS and the W^2 of n replicas of L=2048, 256
// warps each, ms in row lanes and with the graph: n=16 1.36, 1.96; 24 1.98, 2.29;
// 32 2.49, 2.64; 40 3.02, 2.87; 64 4.66, 3.25).
constexpr uint32_t kBatchRowWarpsMax = 152u * 54u;

// One warp per block, so that the blocks spread evenly over the schedulers (16
// replicas of L=2048, 16 MCS and their W^2: 1.57 ms, 1.78 with four).
__global__ void __launch_bounds__(32)
    batch_row_kernel(const ReplicaDev *reps, const BatchItem *items, const WarpDesc *descs, const uint32_t *t_of,
                     uint32_t dt, uint32_t k) {
    __shared__ __align__(16) uint32_t sm[row_smem_words<true>()];
    const WarpDesc wd = descs[blockIdx.x];
    const uint32_t slot = (threadIdx.x & 31u) / wd.G;
    const bool held = slot < wd.n;
    const BatchItem it = items[wd.first + (held ? slot : 0u)];
    const ReplicaDev R = reps[it.rep];
    const uint32_t t = t_of[it.rep] + dt;
    if (wd.G == 32u) {
        if (wd.kpz)
            batch_row_item<false, 1, true>(R, wd, it.T, held, t, k, sm);
        else
            batch_row_item<true, -1, true>(R, wd, it.T, held, t, k, sm);
    } else {
        if (wd.kpz)
            batch_row_item<false, 1, false>(R, wd, it.T, held, t, k, sm);
        else
            batch_row_item<true, -1, false>(R, wd, it.T, held, t, k, sm);
    }
}

// Adds n to the MCS counter of every active replica.
__global__ void batch_advance_kernel(uint32_t *t_of, const uint32_t *active, uint32_t n_active, uint32_t n) {
    launch_dependents();
    wait_for_previous_grid();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_active; i += gridDim.x * blockDim.x)
        t_of[active[i]] += n;
}

}  // namespace
}  // namespace oct

namespace {

constexpr int kModes = 4;
constexpr int kKinds = 2 * kModes;  // acceptance mode x (several sub-tiles per warp, or one)
// Each kind's replicas are split into up to kParts parts of about equal
// sites, each of at least kMinPartSites sites; a branch (kind, part) is the
// unit of the captured graph (see enqueue_mcs).
constexpr int kParts = 3;
constexpr uint64_t kMinPartSites = uint64_t{1} << 26;
constexpr int kBranches = kKinds * kParts;

int bfail(int code, const std::string &msg) {
    oct::set_last_error(msg);
    return code;
}

#define BATCH_CUDA(call)                                                                  \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) return bfail(OCT_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

uint32_t thr32(double p) { return static_cast<uint32_t>(std::floor(std::ldexp(p, 32))); }

}  // namespace

namespace oct {
namespace {

// One of the two alternating copies of the work list (replica table, items,
// warp descriptors, active slots).  A rebuild fills the copy the running work
// does not read, from pinned staging memory, in stream order: no host wait.
struct WorkBuf {
    ReplicaDev *reps = nullptr;
    size_t reps_cap = 0;
    BatchItem *items = nullptr;
    size_t items_cap = 0;
    WarpDesc *descs = nullptr;
    size_t descs_cap = 0;
    uint32_t *active = nullptr;
    size_t active_cap = 0;
    char *host = nullptr;     // pinned staging of the last copy into this set
    size_t host_cap = 0;
    cudaEvent_t copied = nullptr;  // recorded after that copy
};

// A W^2 measurement: the exact sums, the replica's counters and its time,
// written to pinned host memory by the reduction itself.
struct MeasureRecord {
    W2Result res;
    long long cnt[2];
    uint32_t t;
    uint32_t pad[3];
};
// Rows reduced by one launch of a measurement of all replicas (32 MiB of row
// records); larger batches take several launches.
constexpr uint64_t kMeasureRows = uint64_t{1} << 20;
constexpr int kMeasureRing = 1024;
// Rows one launch of an asynchronous measurement takes beyond its first
// replica: the batch's scratch grows to at most 3 MB for it.
constexpr int64_t kPackRows = 65536;
constexpr int kMarkRing = 64;
constexpr int kGraphMcs = 4;  // MCS in the batch's longer captured graph
// A batch in row lanes takes four launches per MCS.  The driver queues about a
// thousand launches; past that a call waits for the device, so a long run would
// no longer return at once (3000 MCS of four small replicas: the call took 90 of
// 99 ms, 1.2 of 97 with replays).  After kRowLaunchMcs MCS of one membership the
// rest is replayed from graphs of kRowGraphMcs and kRowGraphShort MCS (a batch
// whose replicas change sooner, as in serving, never pays for their capture).
// Replays break the overlap of launches at their ends: us per MCS of that batch
// launched, and in graphs of 4, 8, 16 and 32 MCS, 31.6, 32.2, 31.9, 31.7 and 31.6.
constexpr int64_t kRowLaunchMcs = 128;
constexpr int kRowGraphMcs = 32;
constexpr int kRowGraphShort = 8;

}  // namespace
}  // namespace oct

struct oct_batch {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaMemPool_t pool = nullptr;     // replica lattices, stream-ordered
    // slots (a replica keeps its slot until removed)
    std::vector<oct_replica> reps;
    std::vector<uint32_t *> lat;      // per slot, nullptr if free
    std::vector<char> used;
    std::vector<int64_t> free_slots;
    size_t capacity = 0;
    uint32_t *d_t = nullptr;            // capacity MCS counters
    unsigned long long *counters = nullptr;  // 2 * capacity: net flips, draws
    // work list of the current membership
    bool dirty = true;
    oct::WorkBuf wb[2];
    int cur = 0;  // the copy the enqueued work reads
    uint32_t n_active = 0;
    // work lists by kind = 2 * mode + (one sub-tile per warp); modes: 0 no
    // acceptance draws, 1 draws, 2 draws for both rates, 3 deposition only
    // work lists by branch = kParts * kind + part
    uint32_t n_desc[kBranches] = {};
    uint32_t desc_first[kBranches] = {};
    // the active replicas ordered by branch: act_n[br] of them from act_first[br]
    uint32_t act_first[kBranches] = {};
    uint32_t act_n[kBranches] = {};
    int64_t row_mcs = 0;          // MCS launched one by one in row lanes since the last rebuild
    uint32_t row_descs = 0;       // warps of a device step in row lanes; 0: the branches below carry the batch
    uint32_t *d_queue = nullptr;  // 4 * kBranches counters: (device step, branch)
    oct::W2RowSums *d_rows = nullptr;
    size_t rows_cap = 0;
    void *h_small = nullptr;
    // measurement of all replicas: job list (device, and its pinned staging),
    // records by slot, and the launches' ranges; rebuilt after a membership change
    bool jobs_dirty = true;
    oct::W2Job *d_jobs = nullptr;
    oct::W2Job *h_jobs = nullptr;
    oct::MeasureRecord *h_all = nullptr;
    size_t all_cap = 0;
    std::vector<std::pair<uint32_t, uint32_t>> job_ranges;  // (first job, warp tasks) of each launch
    uint32_t n_jobs = 0;
    // two-time autocorrelations: per slot, the lattice at its waiting time
    std::vector<uint32_t *> snap;
    std::vector<int64_t> snap_t;
    oct::AcRowSums *d_ac_rows = nullptr;
    int64_t ac_rows_cap = 0;
    oct::AcResult *d_ac = nullptr;
    uint64_t ticks = 0;  // MCS run by oct_batch_run
    int grid = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;        // one MCS (kRowGraphShort in row lanes)
    cudaGraph_t graph_n = nullptr;
    cudaGraphExec_t exec_n = nullptr;      // kGraphMcs MCS (kRowGraphMcs)
    // side streams and events of the captured MCS: one branch per kind
    cudaStream_t side[kBranches] = {};
    cudaEvent_t fork_ev = nullptr;
    cudaEvent_t join_ev[kBranches] = {};
    // asynchronous measurements: a ring of pinned records
    oct::MeasureRecord *h_req = nullptr;
    std::vector<cudaEvent_t> req_ev;
    std::vector<int64_t> req_L;
    std::vector<int> req_at;  // ring index of the event recorded behind the ticket's launches
    int64_t req_next = 0;  // tickets handed out so far
    // stream marks (oct_batch_mark): a ring of events
    std::vector<cudaEvent_t> mark_ev;
    int64_t mark_next = 0;  // marks handed out so far
    bool timing = false;
    std::vector<cudaEvent_t> ev;
    int ev_used = 0;
    double step_ms = 0.0;
    int64_t step_launches = 0;
};

namespace {

void drop_graph(oct_batch *b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->exec_n) cudaGraphExecDestroy(b->exec_n);
    if (b->graph_n) cudaGraphDestroy(b->graph_n);
    b->exec = nullptr;
    b->graph = nullptr;
    b->exec_n = nullptr;
    b->graph_n = nullptr;
}

void batch_free(oct_batch *b) {
    drop_graph(b);
    for (uint32_t *p : b->lat)
        if (p) cudaFreeAsync(p, b->stream);
    for (uint32_t *p : b->snap)
        if (p) cudaFreeAsync(p, b->stream);
    if (b->stream) cudaStreamSynchronize(b->stream);
    cudaFree(b->d_ac_rows);
    cudaFree(b->d_ac);
    cudaFree(b->d_t);
    cudaFree(b->counters);
    for (oct::WorkBuf &w : b->wb) {
        cudaFree(w.reps);
        cudaFree(w.items);
        cudaFree(w.descs);
        cudaFree(w.active);
        if (w.host) cudaFreeHost(w.host);
        if (w.copied) cudaEventDestroy(w.copied);
    }
    cudaFree(b->d_jobs);
    if (b->h_jobs) cudaFreeHost(b->h_jobs);
    if (b->h_all) cudaFreeHost(b->h_all);
    if (b->h_req) cudaFreeHost(b->h_req);
    for (cudaEvent_t e : b->req_ev)
        if (e) cudaEventDestroy(e);  // ring events are created on first use
    for (cudaEvent_t e : b->mark_ev)
        if (e) cudaEventDestroy(e);
    cudaFree(b->d_queue);
    for (int br = 0; br < kBranches; ++br) {
        if (b->side[br]) cudaStreamDestroy(b->side[br]);
        if (b->join_ev[br]) cudaEventDestroy(b->join_ev[br]);
    }
    if (b->fork_ev) cudaEventDestroy(b->fork_ev);
    cudaFree(b->d_rows);
    if (b->h_small) cudaFreeHost(b->h_small);
    for (cudaEvent_t e : b->ev)
        if (e) cudaEventDestroy(e);
    if (b->pool) cudaMemPoolDestroy(b->pool);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
}

int check_replica(oct_replica &R) {
    if (R.L < 64 || R.L > 16384 || R.L % 64) return bfail(OCT_EINVAL, "replica L must be a multiple of 64 in [64, 16384]");
    if (!(R.p >= 0.0 && R.p <= 1.0 && R.q >= 0.0 && R.q <= 1.0))
        return bfail(OCT_EINVAL, "replica p and q must lie in [0, 1]");
    if (R.Bx == 0 && R.By == 0) {
        R.Bx = (R.L % 128 == 0) ? 64 : 32;
        R.By = R.Bx;
    }
    const int GX = R.Bx / 32, GY = R.By / 16, G = GX * GY;
    if (R.Bx < 32 || R.By < 16 || R.Bx % 32 || R.By % 16 || R.L % (2 * R.Bx) || R.L % (2 * R.By) ||
        (GX & (GX - 1)) || (GY & (GY - 1)) || G > 32)
        return bfail(OCT_EINVAL, "replica sub-tile must be a power-of-two number (at most 32) of "
                                 "32x16-site groups in each direction and divide L/2");
    return OCT_OK;
}

oct::ReplicaDev replica_dev(const oct_batch *b, int64_t slot) {
    const oct_replica &R = b->reps[slot];
    oct::ReplicaDev D;
    D.lat = b->lat[slot];
    D.counters = b->counters + 2 * slot;
    D.L = static_cast<uint32_t>(R.L);
    D.wpr = static_cast<uint32_t>(R.L / 32);
    D.Bx = static_cast<uint32_t>(R.Bx);
    D.By = static_cast<uint32_t>(R.By);
    D.GX = static_cast<uint32_t>(R.Bx / 32);
    D.GY = static_cast<uint32_t>(R.By / 16);
    D.tiles_x = static_cast<uint32_t>(R.L / (2 * R.Bx));
    D.tiles_y = static_cast<uint32_t>(R.L / (2 * R.By));
    D.k0 = static_cast<uint32_t>(R.seed & 0xFFFFFFFFu);
    D.k1 = static_cast<uint32_t>(R.seed >> 32);
    const bool pr = R.p > 0.0 && R.p < 1.0, qr = R.q > 0.0 && R.q < 1.0;
    D.thr_p = pr ? thr32(R.p) : 0u;
    D.thr_q = qr ? thr32(R.q) : 0u;
    D.p_always = (R.p == 1.0) ? 0xFFFFFFFFu : 0u;
    D.q_always = (R.q == 1.0) ? 0xFFFFFFFFu : 0u;
    D.p_random = pr ? 0xFFFFFFFFu : 0u;
    D.q_random = qr ? 0xFFFFFFFFu : 0u;
    return D;
}

// Stream-ordered: work already enqueued may still read the old buffer.
template <typename T>
cudaError_t grow_async(T **p, size_t *cap, size_t n, cudaStream_t st) {
    return oct::grow_buffer(
        p, cap, n, [st](T **q, size_t k) { return cudaMallocAsync(reinterpret_cast<void **>(q), sizeof(T) * k, st); },
        [st](T *old) { return cudaFreeAsync(old, st); });
}

template <typename T>
cudaError_t ensure(T **p, size_t *cap, size_t need, cudaStream_t st) {
    if (need <= *cap) return cudaSuccess;
    return grow_async(p, cap, std::max<size_t>(need, 2 * *cap), st);
}

// Grows the per-slot tables, keeping the device-resident counters.
cudaError_t grow_slots(oct_batch *b, size_t need) {
    if (need <= b->capacity) return cudaSuccess;
    const size_t n = std::max<size_t>(need, std::max<size_t>(64, 2 * b->capacity));
    uint32_t *t = nullptr;
    unsigned long long *c = nullptr;
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e == cudaSuccess) e = cudaMalloc(&t, sizeof(uint32_t) * n);
    if (e == cudaSuccess) e = cudaMalloc(&c, sizeof(unsigned long long) * 2 * n);
    if (e == cudaSuccess && b->capacity) {
        e = cudaMemcpy(t, b->d_t, sizeof(uint32_t) * b->capacity, cudaMemcpyDeviceToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(c, b->counters, sizeof(unsigned long long) * 2 * b->capacity, cudaMemcpyDeviceToDevice);
    }
    if (e != cudaSuccess) {
        cudaFree(t);
        cudaFree(c);
        return e;
    }
    cudaFree(b->d_t);
    cudaFree(b->counters);
    b->d_t = t;
    b->counters = c;
    b->capacity = n;
    b->dirty = true;
    b->jobs_dirty = true;
    return cudaSuccess;
}

// The batch in row lanes, if every sub-tile fits a warp that way and a device
// step has at most kBatchRowWarpsMax warps: items of one form and lane layout
// packed into descriptors.  Leaves the lists empty otherwise.
void row_lists(const std::vector<oct::ReplicaDev> &rd, const std::vector<uint32_t> &active,
               std::vector<oct::BatchItem> &items, std::vector<oct::WarpDesc> &descs) {
    uint64_t lanes = 0;
    for (uint32_t slot : active) {
        const oct::ReplicaDev &D = rd[slot];
        if (D.GX * (D.By / 4u) > 32u) return;
        lanes += static_cast<uint64_t>(D.tiles_x) * D.tiles_y * oct::row_segment(D.GX, D.By);
    }
    if (lanes > 32ull * oct::kBatchRowWarpsMax) return;
    std::vector<oct::BatchItem> bucket[2][6][6];  // form, log2 of GX, of the lanes per sub-tile
    for (uint32_t slot : active) {
        const oct::ReplicaDev &D = rd[slot];
        int gi = 0, si = 0;
        while ((1u << gi) < D.GX) ++gi;
        while ((1u << si) < oct::row_segment(D.GX, D.By)) ++si;
        const bool kpz = D.p_always && !D.q_always && !D.q_random;
        auto &bk = bucket[kpz ? 1 : 0][gi][si];
        for (uint32_t T = 0; T < D.tiles_x * D.tiles_y; ++T) bk.push_back({slot, T});
    }
    for (uint32_t kpz = 0; kpz < 2u; ++kpz)
        for (uint32_t gi = 0; gi < 6u; ++gi)
            for (uint32_t si = 0; si < 6u; ++si) {
                const auto &bk = bucket[kpz][gi][si];
                const size_t per = 32u >> si;
                for (size_t i = 0; i < bk.size(); i += per) {
                    const uint32_t n = static_cast<uint32_t>(std::min<size_t>(per, bk.size() - i));
                    descs.push_back({static_cast<uint32_t>(items.size()), n, 1u << si, 1u << gi, kpz});
                    items.insert(items.end(), bk.begin() + i, bk.begin() + i + n);
                }
            }
}

// Rebuilds the replica table and the warp work list of the active replicas
// into the work-list copy the enqueued work does not read, by asynchronous
// copies on the batch's stream (the host waits only for the staging memory of
// the copy before last, long finished).
cudaError_t rebuild(oct_batch *b) {
    cudaError_t e = cudaSuccess;
    drop_graph(b);  // an executable graph still running is freed when it completes
    std::vector<oct::ReplicaDev> rd(b->capacity);
    // replicas by kind, then each kind split into up to kParts parts of about
    // equal sites (largest first, each to the lightest part)
    std::vector<uint32_t> by_kind[kKinds];
    for (size_t slot = 0; slot < b->reps.size(); ++slot) {
        if (!b->used[slot]) continue;
        rd[slot] = replica_dev(b, static_cast<int64_t>(slot));
        const oct::ReplicaDev &D = rd[slot];
        const int mode = (D.p_random && D.q_random) ? 2
                         : (D.p_random || D.q_random) ? 1
                         : (D.p_always && !D.q_always) ? 3 : 0;
        by_kind[2 * mode + (D.GX * D.GY == 32u ? 1 : 0)].push_back(static_cast<uint32_t>(slot));
    }
    std::vector<uint32_t> by_branch[kBranches];
    for (int kind = 0; kind < kKinds; ++kind) {
        std::vector<uint32_t> &v = by_kind[kind];
        std::stable_sort(v.begin(), v.end(), [&](uint32_t a, uint32_t c) { return rd[a].L > rd[c].L; });
        uint64_t sites = 0;
        for (uint32_t slot : v) sites += static_cast<uint64_t>(rd[slot].L) * rd[slot].L;
        const int parts = static_cast<int>(std::max<uint64_t>(1, std::min<uint64_t>(kParts, sites / kMinPartSites)));
        uint64_t load[kParts] = {};
        for (uint32_t slot : v) {
            int part = 0;
            for (int q = 1; q < parts; ++q)
                if (load[q] < load[part]) part = q;
            load[part] += static_cast<uint64_t>(rd[slot].L) * rd[slot].L;
            by_branch[kind * kParts + part].push_back(slot);
        }
    }
    std::vector<uint32_t> active;
    std::vector<oct::BatchItem> items;
    std::vector<oct::WarpDesc> descs;
    for (int br = 0; br < kBranches; ++br) active.insert(active.end(), by_branch[br].begin(), by_branch[br].end());
    row_lists(rd, active, items, descs);
    b->row_descs = static_cast<uint32_t>(descs.size());
    b->row_mcs = 0;
    active.clear();
    for (int br = 0; br < kBranches; ++br) {
        b->act_first[br] = static_cast<uint32_t>(active.size());
        b->act_n[br] = static_cast<uint32_t>(by_branch[br].size());
        active.insert(active.end(), by_branch[br].begin(), by_branch[br].end());
        b->n_desc[br] = 0;
        if (b->row_descs) continue;
        // the branch's items bucketed by lane layout, then packed into warps
        std::vector<oct::BatchItem> bucket[6][6];
        for (uint32_t slot : by_branch[br]) {
            const oct::ReplicaDev &D = rd[slot];
            int gxi = 0, gyi = 0;
            while ((1u << gxi) < D.GX) ++gxi;
            while ((1u << gyi) < D.GY) ++gyi;
            for (uint32_t T = 0; T < D.tiles_x * D.tiles_y; ++T) bucket[gxi][gyi].push_back({slot, T});
        }
        b->desc_first[br] = static_cast<uint32_t>(descs.size());
        for (int gxi = 5; gxi >= 0; --gxi)
            for (int gyi = 5; gyi >= 0; --gyi) {
                const uint32_t GX = 1u << gxi, G = GX << gyi;
                if (G > 32u) continue;
                const uint32_t per = 32u / G;
                auto &bk = bucket[gxi][gyi];
                for (size_t i = 0; i < bk.size(); i += per) {
                    oct::WarpDesc d;
                    d.first = static_cast<uint32_t>(items.size());
                    d.n = static_cast<uint32_t>(std::min<size_t>(per, bk.size() - i));
                    d.G = G;
                    d.GX = GX;
                    d.kpz = 0;
                    for (uint32_t j = 0; j < d.n; ++j) items.push_back(bk[i + j]);
                    descs.push_back(d);
                }
            }
        b->n_desc[br] = static_cast<uint32_t>(descs.size()) - b->desc_first[br];
    }
    const int nxt = 1 - b->cur;
    oct::WorkBuf &w = b->wb[nxt];
    const size_t n_reps = std::max<size_t>(1, b->capacity);
    e = ensure(&w.reps, &w.reps_cap, n_reps, b->stream);
    if (e == cudaSuccess) e = ensure(&w.items, &w.items_cap, std::max<size_t>(1, items.size()), b->stream);
    if (e == cudaSuccess) e = ensure(&w.descs, &w.descs_cap, std::max<size_t>(1, descs.size()), b->stream);
    if (e == cudaSuccess) e = ensure(&w.active, &w.active_cap, std::max<size_t>(1, active.size()), b->stream);
    // pinned staging: reps, items, descs, active back to back (16-byte aligned parts)
    auto up16 = [](size_t v) { return (v + 15) & ~static_cast<size_t>(15); };
    const size_t o_items = up16(sizeof(oct::ReplicaDev) * b->capacity);
    const size_t o_descs = o_items + up16(sizeof(oct::BatchItem) * items.size());
    const size_t o_active = o_descs + up16(sizeof(oct::WarpDesc) * descs.size());
    const size_t bytes = std::max<size_t>(16, o_active + sizeof(uint32_t) * active.size());
    if (e == cudaSuccess && w.copied) e = cudaEventSynchronize(w.copied);  // its last copy has left the staging
    if (e == cudaSuccess && bytes > w.host_cap) {
        if (w.host) cudaFreeHost(w.host);
        w.host = nullptr;
        w.host_cap = 0;
        e = cudaMallocHost(reinterpret_cast<void **>(&w.host), 2 * bytes);
        if (e == cudaSuccess) w.host_cap = 2 * bytes;
    }
    if (e == cudaSuccess && !w.copied) e = cudaEventCreateWithFlags(&w.copied, cudaEventDisableTiming);
    if (e != cudaSuccess) return e;
    if (b->capacity) std::memcpy(w.host, rd.data(), sizeof(oct::ReplicaDev) * b->capacity);
    if (!items.empty()) std::memcpy(w.host + o_items, items.data(), sizeof(oct::BatchItem) * items.size());
    if (!descs.empty()) std::memcpy(w.host + o_descs, descs.data(), sizeof(oct::WarpDesc) * descs.size());
    if (!active.empty()) std::memcpy(w.host + o_active, active.data(), sizeof(uint32_t) * active.size());
    if (b->capacity)
        e = cudaMemcpyAsync(w.reps, w.host, sizeof(oct::ReplicaDev) * b->capacity, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess && !items.empty())
        e = cudaMemcpyAsync(w.items, w.host + o_items, sizeof(oct::BatchItem) * items.size(), cudaMemcpyHostToDevice,
                            b->stream);
    if (e == cudaSuccess && !descs.empty())
        e = cudaMemcpyAsync(w.descs, w.host + o_descs, sizeof(oct::WarpDesc) * descs.size(), cudaMemcpyHostToDevice,
                            b->stream);
    if (e == cudaSuccess && !active.empty())
        e = cudaMemcpyAsync(w.active, w.host + o_active, sizeof(uint32_t) * active.size(), cudaMemcpyHostToDevice,
                            b->stream);
    if (e == cudaSuccess) e = cudaEventRecord(w.copied, b->stream);
    if (e != cudaSuccess) return e;
    b->cur = nxt;
    b->n_active = static_cast<uint32_t>(active.size());
    b->dirty = false;
    return cudaSuccess;
}

// Enqueues device step k of the current MCS of the replicas of one branch.
cudaError_t enqueue_branch_step(oct_batch *b, uint32_t k, int br, cudaStream_t st) {
    uint32_t *q = b->d_queue + kBranches * k + br;
    cudaError_t e = cudaMemsetAsync(q, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    const oct::WorkBuf &w = b->wb[b->cur];
    const oct::WarpDesc *descs = w.descs + b->desc_first[br];
    const uint32_t nd = b->n_desc[br];
    const int kind = br / kParts;
    const int blocks = std::min<int>(b->grid, static_cast<int>((nd + oct::kBatchWarps - 1) / oct::kBatchWarps));
    const dim3 grid(blocks), block(oct::kBatchWarps * 32);
#define OCT_BATCH(R, LS, SC) \
    oct::batch_step_kernel<R, LS, SC><<<grid, block, 0, st>>>(w.reps, w.items, descs, nd, b->d_t, k, q)
    switch (kind) {
        case 0: OCT_BATCH(false, true, 0); break;
        case 1: OCT_BATCH(false, false, 0); break;
        case 2: OCT_BATCH(true, true, 0); break;
        case 3: OCT_BATCH(true, false, 0); break;
        case 4: OCT_BATCH(true, true, 10); break;
        case 5: OCT_BATCH(true, false, 10); break;
        case 6: OCT_BATCH(false, true, 4); break;
        default: OCT_BATCH(false, false, 4); break;
    }
#undef OCT_BATCH
    return cudaGetLastError();
}

// Enqueues device step k, dt MCS past the counters, of a batch in row lanes.
// overlap: its head may run during the tail of the step enqueued before it.
cudaError_t enqueue_row_step(oct_batch *b, uint32_t dt, uint32_t k, bool overlap, cudaStream_t st) {
    const oct::WorkBuf &w = b->wb[b->cur];
    return oct::launch_overlapped(oct::batch_row_kernel, dim3(b->row_descs), dim3(32), overlap, st, w.reps, w.items,
                                  w.descs, b->d_t, dt, k);
}

// Enqueues device step k of the current MCS of every active replica, branch by branch.
cudaError_t enqueue_step(oct_batch *b, uint32_t k, cudaStream_t st) {
    if (b->row_descs) return enqueue_row_step(b, 0, k, false, st);
    for (int br = 0; br < kBranches; ++br) {
        if (b->n_desc[br] == 0) continue;
        cudaError_t e = enqueue_branch_step(b, k, br, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t enqueue_advance(oct_batch *b, uint32_t n, cudaStream_t st) {
    if (b->n_active == 0) return cudaSuccess;
    const int blocks = static_cast<int>(std::min<uint32_t>(1024u, (b->n_active + 255u) / 256u));
    const uint32_t *active = b->wb[b->cur].active;
    return oct::launch_overlapped(oct::batch_advance_kernel, dim3(blocks), dim3(256), true, st, b->d_t, active,
                                  b->n_active, n);
}

// Advances the MCS counters of the replicas of one branch.
cudaError_t enqueue_advance_branch(oct_batch *b, int br, cudaStream_t st) {
    const uint32_t n = b->act_n[br];
    if (n == 0) return cudaSuccess;
    const int blocks = static_cast<int>(std::min<uint32_t>(1024u, (n + 255u) / 256u));
    oct::batch_advance_kernel<<<blocks, 256, 0, st>>>(b->d_t, b->wb[b->cur].active + b->act_first[br], n, 1u);
    return cudaGetLastError();
}

// nmcs MCS of a batch in row lanes: launch by launch, each overlapping the one
// before; the counters advance at the end.
cudaError_t enqueue_row_mcs(oct_batch *b, cudaStream_t st, uint32_t nmcs) {
    cudaError_t e = cudaSuccess;
    for (uint32_t i = 0; i < nmcs; ++i)
        for (uint32_t k = 0; k < 4 && e == cudaSuccess; ++k) e = enqueue_row_step(b, i, k, i > 0 || k > 0, st);
    if (e == cudaSuccess && nmcs > 0) e = enqueue_advance(b, nmcs, st);
    return e;
}

// nmcs MCS for capture on st.  The replicas of different branches (kinds,
// and parts of a kind) share no memory and no counter, so each branch's
// device steps and its own MCS-counter advances form a branch of the graph
// (forked from st on a side stream and joined back at the end); the branches
// run concurrently, so one branch's launches fill the device while another's
// drain, and over several MCS no branch waits for the others at MCS
// boundaries.
cudaError_t enqueue_mcs(oct_batch *b, cudaStream_t st, int nmcs) {
    cudaError_t e = cudaSuccess;
    if (!b->fork_ev) e = cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(b->fork_ev, st);
    for (int br = 0; br < kBranches && e == cudaSuccess; ++br) {
        if (b->n_desc[br] == 0) continue;
        if (!b->side[br]) e = cudaStreamCreateWithFlags(&b->side[br], cudaStreamNonBlocking);
        if (e == cudaSuccess && !b->join_ev[br]) e = cudaEventCreateWithFlags(&b->join_ev[br], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->side[br], b->fork_ev, 0);
        for (int i = 0; i < nmcs && e == cudaSuccess; ++i) {
            for (uint32_t k = 0; k < 4 && e == cudaSuccess; ++k) e = enqueue_branch_step(b, k, br, b->side[br]);
            if (e == cudaSuccess) e = enqueue_advance_branch(b, br, b->side[br]);
        }
        if (e == cudaSuccess) e = cudaEventRecord(b->join_ev[br], b->side[br]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, b->join_ev[br], 0);
    }
    return e;
}

// Captures nmcs MCS of the current membership into *graph / *exec.
cudaError_t capture_mcs(oct_batch *b, int nmcs, cudaGraph_t *graph, cudaGraphExec_t *exec) {
    cudaStream_t cap = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const cudaError_t e2 = b->row_descs ? enqueue_row_mcs(b, cap, static_cast<uint32_t>(nmcs)) : enqueue_mcs(b, cap, nmcs);
        e = cudaStreamEndCapture(cap, graph);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, *graph, 0);
    cudaStreamDestroy(cap);
    return e;
}

int flush_batch_timing(oct_batch *b) {
    if (b->ev_used == 0) return OCT_OK;
    BATCH_CUDA(cudaEventSynchronize(b->ev[2 * (b->ev_used - 1) + 1]));
    for (int i = 0; i < b->ev_used; ++i) {
        float ms = 0.f;
        BATCH_CUDA(cudaEventElapsedTime(&ms, b->ev[2 * i], b->ev[2 * i + 1]));
        b->step_ms += ms;
    }
    b->ev_used = 0;
    return OCT_OK;
}

bool valid_slot(const oct_batch *b, int64_t slot) {
    return slot >= 0 && slot < static_cast<int64_t>(b->reps.size()) && b->used[slot];
}

int add_replica(oct_batch *b, const oct_replica *in, int64_t *slot_out) {
    oct_replica R = *in;
    int rc = check_replica(R);
    if (rc) return rc;
    int64_t slot;
    if (!b->free_slots.empty()) {
        slot = b->free_slots.back();
        b->free_slots.pop_back();
    } else {
        slot = static_cast<int64_t>(b->reps.size());
        BATCH_CUDA(grow_slots(b, static_cast<size_t>(slot) + 1));
        b->reps.emplace_back();
        b->lat.push_back(nullptr);
        b->used.push_back(0);
        b->snap.push_back(nullptr);
        b->snap_t.push_back(-1);
    }
    const size_t bytes = static_cast<size_t>(R.L) * R.L / 4;
    uint32_t *p = nullptr;
    cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&p), bytes, b->pool, b->stream);
    if (e != cudaSuccess) {
        b->free_slots.push_back(slot);
        return e == cudaErrorMemoryAllocation ? bfail(OCT_ENOMEM, "no device memory for the replica lattice")
                                              : bfail(OCT_ECUDA, std::string("cudaMallocFromPoolAsync: ") + cudaGetErrorString(e));
    }
    b->reps[slot] = R;
    b->lat[slot] = p;
    b->used[slot] = 1;
    BATCH_CUDA(oct::launch_init_flat(p, static_cast<uint32_t>(R.L), b->stream));
    BATCH_CUDA(cudaMemsetAsync(b->d_t + slot, 0, sizeof(uint32_t), b->stream));
    BATCH_CUDA(cudaMemsetAsync(b->counters + 2 * slot, 0, 2 * sizeof(unsigned long long), b->stream));
    b->dirty = true;
    b->jobs_dirty = true;
    if (slot_out) *slot_out = slot;
    return OCT_OK;
}

// W^2 from an asynchronous measurement record (numerator in 128-bit integers).
void record_to_w2(const oct::MeasureRecord &r, int64_t L, oct_w2 *out) {
    const __int128 N = static_cast<__int128>(L) * L;
    const __int128 S2 = static_cast<__int128>((static_cast<unsigned __int128>(r.res.s2_hi) << 64) | r.res.s2_lo);
    const __int128 num = N * S2 - static_cast<__int128>(r.res.s1) * r.res.s1;
    out->t = static_cast<int64_t>(r.t);
    out->n_sites = static_cast<int64_t>(N);
    out->s1 = r.res.s1;
    out->s2_lo = r.res.s2_lo;
    out->s2_hi = r.res.s2_hi;
    out->net_flips = static_cast<int64_t>(r.cnt[0]);
    out->hmax = r.res.hmax;
    out->w2 = static_cast<double>(num) / (static_cast<double>(N) * static_cast<double>(N));
}

// The reduction of the replica in one slot into the pinned record m.
oct::W2Job replica_job(const oct_batch *b, int64_t slot, oct::MeasureRecord *m) {
    oct::W2Job j{};
    j.lat = b->lat[slot];
    j.L = j.nrows = j.plane_rows = static_cast<uint32_t>(b->reps[slot].L);
    j.res = &m->res;
    j.cnt = b->counters + 2 * slot;
    j.cnt_n = 1;
    j.cnt_off = 1;
    j.cnt_out = m->cnt;
    j.t = b->d_t + slot;
    j.t_out = &m->t;
    return j;
}

// Row records for `rows` rows.  They never shrink, also when growing fails: the
// built job list (build_jobs) relies on those that it asked for.
int ensure_rows(oct_batch *b, int64_t rows) {
    if (static_cast<size_t>(rows) > b->rows_cap)
        BATCH_CUDA(grow_async(&b->d_rows, &b->rows_cap, static_cast<size_t>(rows), b->stream));
    return OCT_OK;
}

int measure_slot(oct_batch *b, int64_t slot, oct_w2 *out) {
    int rc = ensure_rows(b, b->reps[slot].L);
    if (rc) return rc;
    auto *m = static_cast<oct::MeasureRecord *>(b->h_small);
    oct::W2Job j = replica_job(b, slot, m);
    BATCH_CUDA(oct::launch_w2_small_pack(&j, 1, b->d_rows, b->stream));
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    record_to_w2(*m, b->reps[slot].L, out);
    return OCT_OK;
}

// The job list of all replicas, in launches of at most kMeasureRows rows.
// Called with no measurement of all replicas in flight (each one waits for
// its records), so the staging memory is free.
int build_jobs(oct_batch *b) {
    const size_t n = b->reps.size();
    if (n > b->all_cap) {
        const size_t cap = std::max<size_t>(b->capacity, n);
        cudaFree(b->d_jobs);
        if (b->h_jobs) cudaFreeHost(b->h_jobs);
        if (b->h_all) cudaFreeHost(b->h_all);
        b->d_jobs = nullptr;
        b->h_jobs = nullptr;
        b->h_all = nullptr;
        b->all_cap = 0;
        BATCH_CUDA(cudaMalloc(&b->d_jobs, sizeof(oct::W2Job) * cap));
        BATCH_CUDA(cudaMallocHost(&b->h_jobs, sizeof(oct::W2Job) * cap));
        BATCH_CUDA(cudaMallocHost(&b->h_all, sizeof(oct::MeasureRecord) * cap));
        b->all_cap = cap;
    }
    b->job_ranges.clear();
    uint32_t nj = 0;
    int64_t most = 0;
    size_t slot = 0;
    while (slot < n) {
        const uint32_t first = nj;
        uint64_t rows = 0;
        for (; slot < n; ++slot) {
            if (!b->used[slot]) continue;
            if (nj > first && rows + b->reps[slot].L > oct::kMeasureRows) break;
            rows += b->reps[slot].L;
            b->h_jobs[nj++] = replica_job(b, static_cast<int64_t>(slot), b->h_all + slot);
        }
        if (nj == first) break;
        b->job_ranges.emplace_back(first, oct::w2_small_split(b->h_jobs + first, nj - first));
        most = std::max<int64_t>(most, static_cast<int64_t>(rows));
    }
    b->n_jobs = nj;
    if (nj)
        BATCH_CUDA(cudaMemcpyAsync(b->d_jobs, b->h_jobs, sizeof(oct::W2Job) * nj, cudaMemcpyHostToDevice, b->stream));
    int rc = ensure_rows(b, most);
    if (rc) return rc;
    b->jobs_dirty = false;
    return OCT_OK;
}

int ticket_index(oct_batch *b, int64_t ticket, int *idx) {
    if (ticket < 0 || ticket >= b->req_next || ticket < b->req_next - oct::kMeasureRing)
        return bfail(OCT_EINVAL, "unknown or expired measurement ticket");
    *idx = static_cast<int>(ticket % oct::kMeasureRing);
    return OCT_OK;
}

}  // namespace

extern "C" {

int oct_batch_measure_async(oct_batch *b, int64_t slot, int64_t *ticket) {
    return oct_batch_measure_slots_async(b, &slot, 1, ticket);
}

int oct_batch_measure_slots_async(oct_batch *b, const int64_t *slots, int64_t n, int64_t *tickets) {
    if (!b || n < 0 || n > oct::kMeasureRing || (n > 0 && (!slots || !tickets)))
        return bfail(OCT_EINVAL, "bad slot list");
    for (int64_t i = 0; i < n; ++i)
        if (!valid_slot(b, slots[i])) return bfail(OCT_EINVAL, "no replica in that slot");
    if (n == 0) return OCT_OK;
    BATCH_CUDA(cudaSetDevice(b->device));
    if (!b->h_req) {
        b->req_ev.assign(oct::kMeasureRing, nullptr);
        b->req_L.assign(oct::kMeasureRing, 0);
        b->req_at.assign(oct::kMeasureRing, 0);
        BATCH_CUDA(cudaMallocHost(&b->h_req, sizeof(oct::MeasureRecord) * oct::kMeasureRing));
    }
    for (int64_t first = 0; first < n;) {
        oct::W2Job jobs[oct::kW2PackJobs];
        uint32_t m = 0;
        int64_t rows = 0;
        while (first + m < n && m < oct::kW2PackJobs) {
            const int64_t slot = slots[first + m], L = b->reps[slot].L, ticket = b->req_next + m;
            if (m > 0 && rows + L > oct::kPackRows) break;
            const int i = static_cast<int>(ticket % oct::kMeasureRing);
            if (ticket >= oct::kMeasureRing)  // the ring wrapped: the oldest record is done
                BATCH_CUDA(cudaEventSynchronize(b->req_ev[b->req_at[i]]));
            jobs[m++] = replica_job(b, slot, b->h_req + i);
            rows += L;
        }
        const int at = static_cast<int>((b->req_next + m - 1) % oct::kMeasureRing);
        if (!b->req_ev[at]) BATCH_CUDA(cudaEventCreateWithFlags(&b->req_ev[at], cudaEventDisableTiming));
        int rc = ensure_rows(b, rows);
        if (rc) return rc;
        BATCH_CUDA(oct::launch_w2_small_pack(jobs, m, b->d_rows, b->stream));
        BATCH_CUDA(cudaEventRecord(b->req_ev[at], b->stream));
        for (uint32_t i = 0; i < m; ++i) {
            const int r = static_cast<int>(b->req_next % oct::kMeasureRing);
            b->req_L[r] = b->reps[slots[first]].L;
            b->req_at[r] = at;
            tickets[first++] = b->req_next++;
        }
    }
    return OCT_OK;
}

int oct_batch_poll(oct_batch *b, int64_t ticket, oct_w2 *out, int *ready) {
    if (!b || !out || !ready) return bfail(OCT_EINVAL, "NULL argument");
    int i = 0;
    int rc = ticket_index(b, ticket, &i);
    if (rc) return rc;
    BATCH_CUDA(cudaSetDevice(b->device));
    const cudaError_t e = cudaEventQuery(b->req_ev[b->req_at[i]]);
    if (e == cudaErrorNotReady) {
        (void)cudaGetLastError();  // "not ready" is an answer, not an error: do not leave it behind
        *ready = 0;
        return OCT_OK;
    }
    if (e != cudaSuccess) return bfail(OCT_ECUDA, std::string("oct_batch_poll: ") + cudaGetErrorString(e));
    record_to_w2(b->h_req[i], b->req_L[i], out);
    *ready = 1;
    return OCT_OK;
}

int oct_batch_wait(oct_batch *b, int64_t ticket, oct_w2 *out) {
    if (!b || !out) return bfail(OCT_EINVAL, "NULL argument");
    int i = 0;
    int rc = ticket_index(b, ticket, &i);
    if (rc) return rc;
    BATCH_CUDA(cudaSetDevice(b->device));
    BATCH_CUDA(cudaEventSynchronize(b->req_ev[b->req_at[i]]));
    record_to_w2(b->h_req[i], b->req_L[i], out);
    return OCT_OK;
}

int oct_replica_seed(uint64_t master_seed, uint32_t r, uint64_t *seed) {
    if (!seed) return bfail(OCT_EINVAL, "seed must not be NULL");
    const uint4 w = oct::philox4x32_10(r, 0u, 0u, oct::kTagReplica << 28,
                                       static_cast<uint32_t>(master_seed & 0xFFFFFFFFu),
                                       static_cast<uint32_t>(master_seed >> 32));
    *seed = static_cast<uint64_t>(w.x) | (static_cast<uint64_t>(w.y) << 32);
    return OCT_OK;
}

int oct_batch_create(int64_t n, const oct_replica *reps, void *stream, oct_batch **out) {
    if (n < 0 || (n > 0 && !reps) || !out) return bfail(OCT_EINVAL, "need n >= 0 replicas and non-NULL arrays");
    for (int64_t r = 0; r < n; ++r) {
        oct_replica R = reps[r];
        int rc = check_replica(R);
        if (rc) return rc;
    }
    oct_batch *b = new (std::nothrow) oct_batch();
    if (!b) return bfail(OCT_ENOMEM, "host allocation failed");
    cudaError_t e = cudaGetDevice(&b->device);
    if (e == cudaSuccess) {
        if (stream) {
            b->stream = static_cast<cudaStream_t>(stream);
        } else {
            e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
            b->own_stream = (e == cudaSuccess);
        }
    }
    if (e == cudaSuccess) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = b->device;
        e = cudaMemPoolCreate(&b->pool, &props);
        if (e == cudaSuccess) {
            uint64_t keep = ~uint64_t{0};  // keep freed lattices in the pool for reuse
            e = cudaMemPoolSetAttribute(b->pool, cudaMemPoolAttrReleaseThreshold, &keep);
        }
    }
    if (e == cudaSuccess) e = cudaMalloc(&b->d_queue, sizeof(uint32_t) * 4 * kBranches);
    if (e == cudaSuccess) e = cudaMallocHost(&b->h_small, 256);
    if (e == cudaSuccess) {
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
        b->grid = sms * oct::kBatchBlocksPerSM;
    }
    if (e == cudaSuccess) e = grow_slots(b, static_cast<size_t>(std::max<int64_t>(n, 1)));
    if (e != cudaSuccess) {
        const bool oom = (e == cudaErrorMemoryAllocation);
        batch_free(b);
        delete b;
        return oom ? bfail(OCT_ENOMEM, "device allocation failed")
                   : bfail(OCT_ECUDA, std::string("oct_batch_create: ") + cudaGetErrorString(e));
    }
    for (int64_t r = 0; r < n; ++r) {
        int rc = add_replica(b, &reps[r], nullptr);
        if (rc) {
            batch_free(b);
            delete b;
            return rc;
        }
    }
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) {
        batch_free(b);
        delete b;
        return bfail(OCT_ECUDA, "oct_batch_create: initialisation failed");
    }
    *out = b;
    return OCT_OK;
}

int oct_batch_add(oct_batch *b, const oct_replica *r, int64_t *slot) {
    if (!b || !r) return bfail(OCT_EINVAL, "NULL argument");
    BATCH_CUDA(cudaSetDevice(b->device));
    return add_replica(b, r, slot);
}

int oct_batch_remove(oct_batch *b, int64_t slot) {
    if (!b || !valid_slot(b, slot)) return bfail(OCT_EINVAL, "no replica in that slot");
    BATCH_CUDA(cudaSetDevice(b->device));
    BATCH_CUDA(cudaFreeAsync(b->lat[slot], b->stream));
    b->lat[slot] = nullptr;
    if (b->snap[slot]) {
        BATCH_CUDA(cudaFreeAsync(b->snap[slot], b->stream));
        b->snap[slot] = nullptr;
    }
    b->snap_t[slot] = -1;
    b->used[slot] = 0;
    b->free_slots.push_back(slot);
    b->dirty = true;
    b->jobs_dirty = true;
    return OCT_OK;
}

int oct_batch_run(oct_batch *b, int64_t n) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    if (n < 0) return bfail(OCT_EINVAL, "bad MCS count");
    BATCH_CUDA(cudaSetDevice(b->device));
    if (b->dirty) BATCH_CUDA(rebuild(b));
    if (b->n_active == 0 || n == 0) {
        b->ticks += static_cast<uint64_t>(n);
        return OCT_OK;
    }
    if (b->timing) {
        // launch by launch, each device step bracketed by events
        for (int64_t i = 0; i < n; ++i) {
            for (uint32_t k = 0; k < 4; ++k) {
                if (b->ev_used == 256) {
                    int rc = flush_batch_timing(b);
                    if (rc) return rc;
                }
                BATCH_CUDA(cudaEventRecord(b->ev[2 * b->ev_used], b->stream));
                BATCH_CUDA(enqueue_step(b, k, b->stream));
                BATCH_CUDA(cudaEventRecord(b->ev[2 * b->ev_used + 1], b->stream));
                ++b->ev_used;
                ++b->step_launches;
            }
            BATCH_CUDA(enqueue_advance(b, 1u, b->stream));
        }
    } else if (b->row_descs) {
        // launch by launch at first, replays of graphs once the membership has
        // lasted (see kRowLaunchMcs); they are captured behind the first launches,
        // while the device works on them.  A caller's capture takes the launches.
        cudaStreamCaptureStatus outer = cudaStreamCaptureStatusNone;
        if (n >= oct::kRowGraphShort) BATCH_CUDA(cudaStreamIsCapturing(b->stream, &outer));
        int64_t left = n;
        while (left > 0) {
            if (left >= oct::kRowGraphShort && b->row_mcs >= oct::kRowLaunchMcs && outer == cudaStreamCaptureStatusNone) {
                const bool longer = left >= oct::kRowGraphMcs;
                const int mcs = longer ? oct::kRowGraphMcs : oct::kRowGraphShort;
                cudaGraphExec_t &exec = longer ? b->exec_n : b->exec;
                if (!exec) {
                    const cudaError_t e = capture_mcs(b, mcs, longer ? &b->graph_n : &b->graph, &exec);
                    if (e != cudaSuccess) return bfail(OCT_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
                }
                BATCH_CUDA(cudaGraphLaunch(exec, b->stream));
                left -= mcs;
                continue;
            }
            const int64_t part = std::min<int64_t>(left, oct::kRowLaunchMcs);
            BATCH_CUDA(enqueue_row_mcs(b, b->stream, static_cast<uint32_t>(part)));
            b->row_mcs += part;
            left -= part;
        }
    } else {
        // kGraphMcs MCS per graph launch while that many are left, then one
        // at a time; each graph is captured on a private stream on first use
        // after a membership change and replayed on the batch's stream
        int64_t left = n;
        if (left >= oct::kGraphMcs) {
            if (!b->exec_n) {
                const cudaError_t e = capture_mcs(b, oct::kGraphMcs, &b->graph_n, &b->exec_n);
                if (e != cudaSuccess) return bfail(OCT_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
            }
            for (; left >= oct::kGraphMcs; left -= oct::kGraphMcs) BATCH_CUDA(cudaGraphLaunch(b->exec_n, b->stream));
        }
        if (left > 0) {
            if (!b->exec) {
                const cudaError_t e = capture_mcs(b, 1, &b->graph, &b->exec);
                if (e != cudaSuccess) return bfail(OCT_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
            }
            for (; left > 0; --left) BATCH_CUDA(cudaGraphLaunch(b->exec, b->stream));
        }
    }
    b->ticks += static_cast<uint64_t>(n);
    return OCT_OK;
}

int oct_batch_measure_w2(oct_batch *b, oct_w2 *out, int64_t n) {
    if (!b || !out || n != static_cast<int64_t>(b->reps.size()))
        return bfail(OCT_EINVAL, "out must hold one entry per slot");
    BATCH_CUDA(cudaSetDevice(b->device));
    if (b->jobs_dirty) {
        int rc = build_jobs(b);
        if (rc) return rc;
    }
    for (size_t i = 0; i < b->job_ranges.size(); ++i) {
        const uint32_t first = b->job_ranges[i].first;
        const uint32_t end = i + 1 < b->job_ranges.size() ? b->job_ranges[i + 1].first : b->n_jobs;
        if (end - first == 1u) {
            oct::W2Job j = b->h_jobs[first];
            BATCH_CUDA(oct::launch_w2_small_pack(&j, 1, b->d_rows, b->stream));
        } else {
            BATCH_CUDA(
                oct::launch_w2_small(b->d_jobs + first, end - first, b->job_ranges[i].second, b->d_rows, b->stream));
        }
    }
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    for (int64_t slot = 0; slot < n; ++slot) {
        if (b->used[slot])
            record_to_w2(b->h_all[slot], b->reps[slot].L, &out[slot]);
        else
            std::memset(&out[slot], 0, sizeof(oct_w2));
    }
    return OCT_OK;
}

int oct_batch_measure_slot(oct_batch *b, int64_t slot, oct_w2 *out) {
    if (!b || !out || !valid_slot(b, slot)) return bfail(OCT_EINVAL, "no replica in that slot");
    BATCH_CUDA(cudaSetDevice(b->device));
    return measure_slot(b, slot, out);
}

int oct_batch_snapshot(oct_batch *b, int64_t slot) {
    if (!b || !valid_slot(b, slot)) return bfail(OCT_EINVAL, "no replica in that slot");
    BATCH_CUDA(cudaSetDevice(b->device));
    const int64_t L = b->reps[slot].L;
    const size_t bytes = static_cast<size_t>(L) * L / 4;
    if (!b->snap[slot]) {
        uint32_t *p = nullptr;
        cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&p), bytes, b->pool, b->stream);
        if (e != cudaSuccess)
            return e == cudaErrorMemoryAllocation ? bfail(OCT_ENOMEM, "no device memory for the snapshot")
                                                  : bfail(OCT_ECUDA, std::string("cudaMallocFromPoolAsync: ") + cudaGetErrorString(e));
        b->snap[slot] = p;
    }
    BATCH_CUDA(cudaMemcpyAsync(b->snap[slot], b->lat[slot], bytes, cudaMemcpyDeviceToDevice, b->stream));
    auto *tt = reinterpret_cast<uint32_t *>(static_cast<char *>(b->h_small) + 96);
    BATCH_CUDA(cudaMemcpyAsync(tt, b->d_t + slot, sizeof(uint32_t), cudaMemcpyDeviceToHost, b->stream));
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    b->snap_t[slot] = static_cast<int64_t>(*tt);
    return OCT_OK;
}

int oct_batch_measure_ac(oct_batch *b, int64_t slot, oct_ac *out) {
    if (!b || !out || !valid_slot(b, slot)) return bfail(OCT_EINVAL, "no replica in that slot");
    if (!b->snap[slot]) return bfail(OCT_EINVAL, "no snapshot in that slot: call oct_batch_snapshot first");
    BATCH_CUDA(cudaSetDevice(b->device));
    const int64_t L = b->reps[slot].L;
    if (L > b->ac_rows_cap) {
        cudaFree(b->d_ac_rows);
        b->d_ac_rows = nullptr;
        b->ac_rows_cap = 0;
        BATCH_CUDA(cudaMalloc(&b->d_ac_rows, sizeof(oct::AcRowSums) * L));
        b->ac_rows_cap = L;
    }
    if (!b->d_ac) BATCH_CUDA(cudaMalloc(&b->d_ac, sizeof(oct::AcResult)));
    BATCH_CUDA(oct::launch_two_time(b->lat[slot], b->snap[slot], static_cast<uint32_t>(L), b->d_ac_rows, b->d_ac,
                                    b->stream));
    oct::AcResult r{};
    BATCH_CUDA(cudaMemcpyAsync(&r, b->d_ac, sizeof(r), cudaMemcpyDeviceToHost, b->stream));
    auto *tt = reinterpret_cast<uint32_t *>(static_cast<char *>(b->h_small) + 96);
    BATCH_CUDA(cudaMemcpyAsync(tt, b->d_t + slot, sizeof(uint32_t), cudaMemcpyDeviceToHost, b->stream));
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    oct::fill_ac(L, r, out);
    out->t = static_cast<int64_t>(*tt);
    out->s = b->snap_t[slot];
    return OCT_OK;
}

int oct_batch_get_planes(oct_batch *b, int64_t slot, uint32_t *host, size_t words) {
    if (!b || !host || !valid_slot(b, slot)) return bfail(OCT_EINVAL, "no replica in that slot");
    const int64_t L = b->reps[slot].L;
    if (words != static_cast<size_t>(L) * L / 16) return bfail(OCT_EINVAL, "words must equal L*L/16");
    BATCH_CUDA(cudaSetDevice(b->device));
    BATCH_CUDA(cudaMemcpyAsync(host, b->lat[slot], words * 4, cudaMemcpyDeviceToHost, b->stream));
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    return OCT_OK;
}

int oct_batch_get_stats(oct_batch *b, int64_t *ticks, int64_t *n_active, int64_t *active_sites, int64_t *draws) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    BATCH_CUDA(cudaSetDevice(b->device));
    int64_t sites = 0, na = 0;
    for (size_t s = 0; s < b->reps.size(); ++s)
        if (b->used[s]) {
            sites += b->reps[s].L * b->reps[s].L;
            ++na;
        }
    if (ticks) *ticks = static_cast<int64_t>(b->ticks);
    if (n_active) *n_active = na;
    if (active_sites) *active_sites = sites;
    if (draws) {
        std::vector<unsigned long long> cnt(2 * b->reps.size());
        if (!cnt.empty()) {
            BATCH_CUDA(cudaMemcpyAsync(cnt.data(), b->counters, sizeof(unsigned long long) * cnt.size(),
                                       cudaMemcpyDeviceToHost, b->stream));
            BATCH_CUDA(cudaStreamSynchronize(b->stream));
        }
        int64_t d = 0;
        for (size_t s = 0; s < b->reps.size(); ++s)
            if (b->used[s]) d += static_cast<int64_t>(cnt[2 * s + 1]);
        *draws = d;
    }
    return OCT_OK;
}

int oct_batch_sync(oct_batch *b) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    BATCH_CUDA(cudaSetDevice(b->device));
    BATCH_CUDA(cudaStreamSynchronize(b->stream));
    return OCT_OK;
}

int oct_batch_mark(oct_batch *b, int64_t *mark) {
    if (!b || !mark) return bfail(OCT_EINVAL, "NULL argument");
    BATCH_CUDA(cudaSetDevice(b->device));
    if (b->mark_ev.empty()) b->mark_ev.assign(oct::kMarkRing, nullptr);
    const int i = static_cast<int>(b->mark_next % oct::kMarkRing);
    if (b->mark_ev[i]) {
        // the ring wrapped: the mark recorded here kMarkRing marks ago is passed first
        BATCH_CUDA(cudaEventSynchronize(b->mark_ev[i]));
    } else {
        BATCH_CUDA(cudaEventCreateWithFlags(&b->mark_ev[i], cudaEventDisableTiming));
    }
    BATCH_CUDA(cudaEventRecord(b->mark_ev[i], b->stream));
    *mark = b->mark_next++;
    return OCT_OK;
}

int oct_batch_mark_done(oct_batch *b, int64_t mark, int *done) {
    if (!b || !done) return bfail(OCT_EINVAL, "NULL argument");
    if (mark < 0 || mark >= b->mark_next) return bfail(OCT_EINVAL, "unknown stream mark");
    if (mark < b->mark_next - oct::kMarkRing) {  // its event was reused after the device passed it
        *done = 1;
        return OCT_OK;
    }
    BATCH_CUDA(cudaSetDevice(b->device));
    const cudaError_t e = cudaEventQuery(b->mark_ev[mark % oct::kMarkRing]);
    if (e == cudaErrorNotReady) {
        (void)cudaGetLastError();
        *done = 0;
        return OCT_OK;
    }
    if (e != cudaSuccess) return bfail(OCT_ECUDA, std::string("oct_batch_mark_done: ") + cudaGetErrorString(e));
    *done = 1;
    return OCT_OK;
}

int oct_batch_mark_wait(oct_batch *b, int64_t mark) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    if (mark < 0 || mark >= b->mark_next) return bfail(OCT_EINVAL, "unknown stream mark");
    if (mark < b->mark_next - oct::kMarkRing) return OCT_OK;
    BATCH_CUDA(cudaSetDevice(b->device));
    BATCH_CUDA(cudaEventSynchronize(b->mark_ev[mark % oct::kMarkRing]));
    return OCT_OK;
}

int oct_batch_set_timing(oct_batch *b, int enable) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    BATCH_CUDA(cudaSetDevice(b->device));
    if (b->ev.empty()) {
        b->ev.resize(512);
        for (auto &e : b->ev) BATCH_CUDA(cudaEventCreate(&e));
    }
    int rc = flush_batch_timing(b);
    if (rc) return rc;
    b->timing = enable != 0;
    b->step_ms = 0.0;
    b->step_launches = 0;
    return OCT_OK;
}

int oct_batch_get_timing(oct_batch *b, double *step_ms, int64_t *step_launches) {
    if (!b) return bfail(OCT_EINVAL, "NULL batch");
    int rc = flush_batch_timing(b);
    if (rc) return rc;
    if (step_ms) *step_ms = b->step_ms;
    if (step_launches) *step_launches = b->step_launches;
    return OCT_OK;
}

int oct_batch_destroy(oct_batch *b) {
    if (!b) return OCT_OK;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    batch_free(b);
    delete b;
    return OCT_OK;
}

}  // extern "C"
