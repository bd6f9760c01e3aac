// Device code shared by the plain and the batched device-step kernels: one
// device step on a sub-tile held by warp lanes, with the block layer of
// DTrDT, DTrDB or DTrDTr (see dtrdt.cu for the method and the lane layout).
// Streams beyond those listed in dtrdt.cu: DTrDB draws a site of the whole
// cell from (t, k|s<<2, T, SITE_DB<<28|g), DTrDTr its block-layer origin from
// (t, k, T, BORG<<28), byte s of the device step.
#pragma once
#include <cstdint>

#include "oct_internal.h"
#include "overlap.cuh"
#include "philox.cuh"

namespace oct {

constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kNib = 0x11111111u;  // bit 0 of every 4-bit TC column

// Element k of the idx-th permutation of (0,1,2,3) in lexicographic order: the
// first one is idx / 6, the others are the (idx % 6)-th permutation of the
// three that are left, in order.
__device__ __forceinline__ int perm_element(uint32_t idx, uint32_t k) {
    // two bits per element: 012 021 102 120 201 210
    constexpr uint64_t kPerm3 = (0x24ull << 0) | (0x18ull << 6) | (0x21ull << 12) | (0x09ull << 18) | (0x12ull << 24) |
                                (0x06ull << 30);
    const uint32_t first = idx / 6u, r = idx - 6u * first;
    if (k == 0u) return static_cast<int>(first);
    const uint32_t e = static_cast<uint32_t>(kPerm3 >> (6u * r + 2u * (k - 1u))) & 3u;
    return static_cast<int>(e + (e >= first ? 1u : 0u));
}

// Sets the bits of *w selected by mask to those of v, leaving the others, as
// two reductions (no value returned, so the warp does not wait for them).
__device__ __forceinline__ void reduce_bits(uint32_t *w, uint32_t v, uint32_t mask) {
    atomicAnd(w, v | ~mask);
    atomicOr(w, v & mask);
}

// A 1 that the compiler does not know: one * c + x is then a multiply-add on the
// FMA pipe, where x + c would run on the integer pipe that binds the step.
__device__ __forceinline__ uint32_t opaque_one() {
    uint32_t v;
    asm volatile("mov.u32 %0, 1;" : "=r"(v));
    return v;
}

// Round keys of Philox: from the launch's arguments (constant memory, neither
// registers nor additions), by multiply-adds, or by plain additions.  One MCS at
// L=2^17 (1024x16, p=0.95, q=0.05) 9.57, 9.45 and 9.8 ms, at L=32768 KPZ (which
// draws one block in two steps) additions 355 us, multiply-adds 357 us; DTrDB at
// L=12288 constants 437 us, multiply-adds 446 us; DTrDTr at L=8192 270, 275 us.
struct KeysConst {
    const StepArgs *a;
    __device__ __forceinline__ uint32_t lo(int r) const { return a->rk0[r]; }
    __device__ __forceinline__ uint32_t hi(int r) const { return a->rk1[r]; }
};
struct KeysFma {
    uint32_t k0, k1, one;
    __device__ __forceinline__ KeysFma() {}
    __device__ __forceinline__ KeysFma(uint32_t lo_word, uint32_t hi_word)
        : k0(lo_word), k1(hi_word), one(opaque_one()) {}
    __device__ __forceinline__ uint32_t lo(int r) const { return one * (static_cast<uint32_t>(r) * 0x9E3779B9u) + k0; }
    __device__ __forceinline__ uint32_t hi(int r) const { return one * (static_cast<uint32_t>(r) * 0xBB67AE85u) + k1; }
};
struct KeysWeyl {
    uint32_t k0, k1;
    __device__ __forceinline__ KeysWeyl() {}
    __device__ __forceinline__ KeysWeyl(uint32_t lo_word, uint32_t hi_word) : k0(lo_word), k1(hi_word) {}
    __device__ __forceinline__ uint32_t lo(int r) const { return k0 + static_cast<uint32_t>(r) * 0x9E3779B9u; }
    __device__ __forceinline__ uint32_t hi(int r) const { return k1 + static_cast<uint32_t>(r) * 0xBB67AE85u; }
};

template <class Keys>
struct LaneCtx {
    uint32_t t, k, T, g;
    Keys key;
    // the first round's products of (t, ., T, .), the high halves with its keys
    uint32_t h0, l0, h1, l1;
    __device__ __forceinline__ void first_round() {
        h0 = __umulhi(0xD2511F53u, t) ^ key.hi(0);
        l0 = 0xD2511F53u * t;
        h1 = __umulhi(0xCD9E8D57u, T) ^ key.lo(0);
        l1 = 0xCD9E8D57u * T;
    }
    // Philox-4x32-10 at counter (t, c1, T, c3)
    __device__ __forceinline__ uint4 draw(uint32_t c1, uint32_t c3) const {
        uint32_t x0 = h1 ^ c1, x1 = l1, x2 = h0 ^ c3, x3 = l0;
#pragma unroll
        for (int r = 1; r < 10; ++r) {
            const uint32_t a0 = __umulhi(0xD2511F53u, x0), b0 = 0xD2511F53u * x0;
            const uint32_t a1 = __umulhi(0xCD9E8D57u, x2), b1 = 0xCD9E8D57u * x2;
            x0 = a1 ^ x1 ^ key.lo(r);
            x2 = a0 ^ x3 ^ key.hi(r);
            x1 = b1;
            x3 = b0;
        }
        return make_uint4(x0, x1, x2, x3);
    }
    uint32_t thr_p, thr_q;
    uint32_t p_always, q_always, p_random, q_random;
    int gx, gy, GX, GY;
    int base;      // lane of the sub-tile's first group
    bool active;   // this lane holds a group of a sub-tile
};

// Net flips (depositions minus removals) among the flips f of one row (x: the
// row's X bits before the flips) that were accepted without a draw (p = 1 or
// q = 1).  Flips decided by a draw are counted once per step from the packed
// acceptance bits instead (random_net).
template <bool RANDOM, class Ctx>
__device__ __forceinline__ int always_net(uint32_t f, uint32_t x, const Ctx &c) {
    if (RANDOM) {
        if ((c.p_always | c.q_always) == 0u) return 0;
        return __popc(f & ~x & c.p_always) - __popc(f & x & c.q_always);
    }
    if (c.q_always == 0u) return __popc(f);   // only depositions are possible
    if (c.p_always == 0u) return -__popc(f);  // only removals
    return __popc(f & ~x) - __popc(f & x);
}

// Net flips among the packed candidates accepted by their draw.
__device__ __forceinline__ int random_net(uint32_t acc, uint32_t pmin, uint32_t pmax) {
    return __popc(acc & pmin) - __popc(acc & pmax);
}

// Tail words read at once for the first ties (accept_candidates), per block
// layer, as measured at L=2^17: DTrDT on full warps gains 2.6 % from three;
// on packed warps, in DTrDB (three acceptance passes per step, often with
// few ties) and in DTrDTr the loop alone is as fast or faster.
constexpr int kPreDt = 3, kPrePacked = 0, kPreDb = 0, kPreDtr = 0;

// Each lane keeps its group's tail stream (see accept_candidates) in its own
// slot of kRingWordsPerLane words of shared memory, a ring above the live
// window: fewer than (ties of one step, at most 32) + 4 words.
constexpr int kRingWordsPerLane = 64;

struct TailPool {
    uint32_t *ring;  // the lane's own slot of kRingWordsPerLane words
    uint32_t head;   // words of the group's tail stream used so far in this device step
    uint32_t end;    // words generated into the slot so far in this device step
    uint32_t rounds; // Philox blocks the lane generated into its slot
};

// Tops up the lane's slot until it holds the `need` words after head; every
// lane of the warp takes part in each round (one Philox block per lane, block
// end/4 of its group's stream, kept only if the slot has room).
template <class Ctx>
__device__ __forceinline__ void tail_refill(uint32_t need, uint32_t g, const Ctx &c, TailPool &tp) {
    while (__any_sync(kFull, tp.end < tp.head + need)) {
        const uint4 B = c.draw(c.k | ((tp.end >> 2) << 2), (kTagTail << 28) | g);
        if (tp.end - tp.head <= static_cast<uint32_t>(kRingWordsPerLane - 4)) {
            *reinterpret_cast<uint4 *>(tp.ring + (tp.end & static_cast<uint32_t>(kRingWordsPerLane - 1))) = B;
            tp.end += 4u;
            ++tp.rounds;
        }
    }
}

// Whether a tied candidate can be accepted: with rates that are multiples of 1/16
// (among them 1/2) the bits after the first four are below no threshold, so every
// tie is refused and the tail stream need not be read.  p=q=1/2: 8 MCS and the W^2 of
// L=4096 349 to 256 us; two MCS at L=32768 (1024x16) 1.25 to 1.03 ms, at L=8192 with 8 x 8
// cells 868 to 656 us, in DTrDTr 268 to 230 us.
__host__ __device__ __forceinline__ bool ties_matter(uint32_t thr_p, uint32_t thr_q) {
    return ((thr_p | thr_q) << 4) != 0u;
}
// What a step knows of it when it is compiled (the question costs the others 0.3 to 3 %).
constexpr int kTiesAsk = 0, kTiesCount = 1, kTiesRefused = 2;

// Acceptance of the packed candidates (bit 4j+m = thread cell column j, TC
// row m).  The uniform u of a candidate, most significant bit first:
//  * bits 31..28 come from the four level words of the lane's group (bit
//    4j+m of word l is bit 31-l), one Philox block per step; all 32 thread
//    cells of the lane are compared with P32 together, one level at a time;
//    the comparison is decided unless the four bits equal P32's;
//  * a candidate still tied takes its bits 27..0 from the top of the next word
//    of its group's tail stream (word i = word i%4 of Philox(t, k|(i/4)<<2, T,
//    TAIL<<28|g), counted from 0 each device step), the group's ties of a step
//    in order of position.  A lane holds one group, so it takes its own words.
template <class Ctx>
__device__ __forceinline__ uint4 level_words(uint32_t s, const Ctx &c) {
    return c.draw(c.k | ((s * 8u) << 2), (kTagAcc << 28) | c.g);
}

// PRE: tail words the lane reads at once for its first ties (0: one word per
// tie in the loop); the fastest choice differs between the block layers.
// und: the tied candidates (of them, pmin: minima); returns acc with those that
// their tail words accept.
template <int PRE, int TIES, class Ctx>
__device__ __forceinline__ uint32_t resolve_ties(uint32_t acc, uint32_t und, uint32_t pmin, const Ctx &c, TailPool &tp) {
    // Skip the tail stage only when no lane of the warp needs it: every lane
    // takes part in the refill rounds.
    if (TIES == kTiesRefused) return acc;
    if (__all_sync(kFull, und == 0u || (TIES == kTiesAsk && !ties_matter(c.thr_p, c.thr_q)))) return acc;
    const uint32_t nt = static_cast<uint32_t>(__popc(und));
    tail_refill(nt, c.g, c, tp);
    // (w >> 4) < (P32 mod 2^28)  <=>  w < 16 (P32 mod 2^28)
    const uint32_t low_p = c.thr_p << 4, low_q = c.thr_q << 4;
    // The lane's next PRE tail words are read at once and its first PRE ties
    // decided without a branch (a lane has fewer than one tie per step on
    // average); further ties take the loop, one word each.
    constexpr uint32_t kMask = static_cast<uint32_t>(kRingWordsPerLane - 1);
    const uint32_t h = tp.head;
    if (PRE > 0) {
        uint32_t wp[PRE > 0 ? PRE : 1];
#pragma unroll
        for (int j = 0; j < PRE; ++j) wp[j] = tp.ring[(h + static_cast<uint32_t>(j)) & kMask];
#pragma unroll
        for (int j = 0; j < PRE; ++j) {
            const uint32_t bit = und & (0u - und);  // lowest tied position (0 once none is left)
            und ^= bit;
            acc |= (wp[j] < ((pmin & bit) ? low_p : low_q)) ? bit : 0u;
        }
    }
    uint32_t hn = h + static_cast<uint32_t>(PRE);
    while (und) {
        const uint32_t bit = und & (0u - und);
        und ^= bit;
        const uint32_t w = tp.ring[hn & kMask];
        ++hn;
        acc |= (w < ((pmin & bit) ? low_p : low_q)) ? bit : 0u;
    }
    tp.head = h + nt;
    return acc;
}

// The packed candidates against P32 on the four levels, then the ties.
template <int PRE, int TIES = kTiesAsk, class Ctx>
__device__ __forceinline__ uint32_t accept_candidates(uint32_t pmin, uint32_t pmax, const uint4 &W,
                                                      const Ctx &c, TailPool &tp) {
    const uint32_t lw[4] = {W.x, W.y, W.z, W.w};
    uint32_t acc = 0, und = pmin | pmax;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t bit = 31u - static_cast<uint32_t>(i);
        const uint32_t tb = (((c.thr_p >> bit) & 1u) ? pmin : 0u) | (((c.thr_q >> bit) & 1u) ? pmax : 0u);
        acc |= und & tb & ~lw[i];
        und &= ~(tb ^ lw[i]);
    }
    return resolve_ties<PRE, TIES>(acc, und, pmin, c, tp);
}

// A lane's flips at column 31, or 0, gathered by row with one funnel shift per row
// (a shift and an and-or otherwise): one MCS at L=2^17 (1024x16, p=0.95, q=0.05)
// 9.68 to 9.57 ms, DTrDB KPZ at L=12288 218 to 202 us for two.
// Bits 31 of rows f0[m], f1[m] at bits 4m+2, 4m+3 (the shift by three also brings
// in bits 29 and 30 of f0, which the mask drops).
__device__ __forceinline__ uint32_t gather_msb_pairs(const uint32_t (&f0)[4], const uint32_t (&f1)[4]) {
    uint32_t v = 0u;
#pragma unroll
    for (int m = 3; m >= 0; --m) {
        v = __funnelshift_l(f1[m], v, 1);
        v = __funnelshift_l(f0[m], v, 3);
    }
    return v & 0xCCCCu;
}
// Bits 0 of rows f0[m], f1[m] at bits 4m, 4m+1.
__device__ __forceinline__ uint32_t gather_lsb_pairs(const uint32_t (&f0)[4], const uint32_t (&f1)[4]) {
    uint32_t v = 0u;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        v = __funnelshift_r(v, f0[m], 1);
        v = __funnelshift_r(v, f1[m], 3);
    }
    return (v >> 16) & 0x3333u;
}
// Bits 31, and bits 0, of rows f[0..15] at bits 0..15.
__device__ __forceinline__ uint32_t gather_msb(const uint32_t (&f)[16]) {
    uint32_t v = 0u;
#pragma unroll
    for (int r = 15; r >= 0; --r) v = __funnelshift_l(f[r], v, 1);
    return v;
}
__device__ __forceinline__ uint32_t gather_lsb(const uint32_t (&f)[16]) {
    uint32_t v = 0u;
#pragma unroll
    for (int r = 0; r < 16; ++r) v = __funnelshift_r(v, f[r], 1);
    return v >> 16;
}

// Constants that the compiler does not know (see opaque_one), for the additive
// flips of a step.
struct FlipConsts {
    uint32_t one, neg, c16;
    __device__ __forceinline__ FlipConsts() : one(opaque_one()) {
        neg = 0u - one;
        asm volatile("mov.u32 %0, 16;" : "=r"(c16));
    }
};
// floor(a b / 2^32) + c
__device__ __forceinline__ uint32_t mad_hi_signed(uint32_t a, uint32_t b, uint32_t c) {
    int r;
    asm("mad.hi.s32 %0, %1, %2, %3;"
        : "=r"(r)
        : "r"(static_cast<int>(a)), "r"(static_cast<int>(b)), "r"(static_cast<int>(c)));
    return static_cast<uint32_t>(r);
}
// Signed flips of a row: a candidate f has X(s) != X(s+x), Y(s) != Y(s+y) and
// X(s) == Y(s), so a minimum (X(s) = 0) takes 2^s from the row's X, adds it to Y(s)
// and takes it from Y(s+y), and a maximum does the opposite: with h = +-f a flip is
// a few multiply-adds, where exclusive ors would run on the integer pipe that binds
// the step (77 % of its rate on packed warps, the FMA pipe 20 %), and a row offset per lane
// is a factor 0 or 1 in place of masks.  Column 31 works modulo 2^32.  One MCS at L=19456 in
// 64 x 64 sub-tiles, p=0.95, q=0.05: 326 to 308 us, KPZ 201 to 178 us (with the
// candidates' columns and packed bits by multiply-adds too, 2.8 and 1.7 % of it); on full
// warps KPZ at L=32768 350 to 343 us, L=2^17 with draws 9.45 to 9.36 ms.
template <int SPEC>
__device__ __forceinline__ uint32_t signed_flips(uint32_t f, uint32_t x) {
    return SPEC == 1 ? f : f - 2u * (f & x);
}
// The changes that flips at column 31 of the left lane make to column 0: v has
// their bits at 4m + I (m: TC row), e0 the column's own bits there.  Field m
// of the word, 4 bits from bit 4m + I on, is -1 or +1 (0 without a flip);
// column_fields moves field m to the top (m = 3 first), and mad_hi_signed of it
// with 16 adds it.
template <int SPEC, int I, bool NEGATE>
__device__ __forceinline__ uint32_t column_fields(uint32_t v, uint32_t e0) {
    const uint32_t b = v & (0x1111u << I);
    const uint32_t w = SPEC == 1 ? (NEGATE ? b : b * 15u) : b + 14u * (NEGATE ? b & ~e0 : b & e0);
    return w << (16 - I);
}

// A collective step runs in three phases: the candidates of every thread
// cell of the lane (specialised on the set's row offset dy), the acceptance
// draws (one copy of the code, shared by both offsets), and the flips with
// the neighbour exchange (specialised again).
//
// Phase 1 with sub-cell set (dx, DY).  X/Y hold the lane's 16 rows, E bit r
// the X bit just right of row r, D the Y row just below row 15.  An attempt at
// s is eligible iff X(s) != X(s+x), Y(s) != Y(s+y) and X(s) == Y(s): then
// X(s) = 0 is the minimum of Eq. (1), X(s) = 1 the maximum.  Candidates that
// need an acceptance draw are packed to bit 4j+m (TC column j, TC row m).
// SPEC 1 (deposition only: p = 1, q = 0, the KPZ case): every eligible
// minimum flips and no maximum does, so the candidates are the minima
// themselves.  SPEC 2 (both 0 < p < 1 and 0 < q < 1): every candidate needs a
// draw, so no always/never masks are applied.
template <int DY, bool RANDOM, int SPEC = 0, class Ctx>
__device__ __forceinline__ void step_candidates(const uint32_t (&X)[16], const uint32_t (&Y)[16],
                                                uint32_t E, uint32_t D, const uint4 &site, uint32_t dx,
                                                const Ctx &c, uint32_t (&cnd0)[4],
                                                uint32_t (&cnd1)[4], uint32_t &pmin, uint32_t &pmax) {
    const uint32_t sw[4] = {site.x, site.y, site.z, site.w};
    const uint32_t sh2 = 2u * dx;
    pmin = 0u;
    pmax = 0u;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        // Site draw: bit 4j = x offset, bit 4j+1 = y offset of TC column j (for odd
        // steps run_subtile has shifted the words down to the step's field).
        const uint32_t u = sw[m];
        const uint32_t col = ((u & kNib) + kNib) << sh2;  // 1 + xoff: one-hot, no carries
        // the y offset, spread over the two columns col can take (bits 2dx, 2dx+1)
        const uint32_t yoff = dx ? (u & (kNib << 1)) * 6u : ((u >> 1) & kNib) * 3u;
        const int r0 = 4 * m + 2 * DY, r1 = r0 + 1;
        const uint32_t xa = X[r0], xb = X[r1];
        // (column 31 is a candidate's only for dx = 1)
        const uint32_t xra = dx ? __funnelshift_r(xa, E >> r0, 1) : xa >> 1;
        const uint32_t xrb = dx ? __funnelshift_r(xb, E >> r1, 1) : xb >> 1;
        const uint32_t ya = Y[r0], yb = Y[r1];
        const uint32_t yc = (r1 + 1 < 16) ? Y[(r1 + 1) & 15] : D;
        if (SPEC == 1) {
            // minimum: X(s) = 0, X(s+x) = 1, Y(s) = 0, Y(s+y) = 1
            cnd0[m] = col & ~yoff & ~xa & xra & ~ya & yb;
            cnd1[m] = col & yoff & ~xb & xrb & ~yb & yc;
            continue;
        }
        cnd0[m] = col & ~yoff & (xa ^ xra) & (ya ^ yb) & ~(xa ^ ya);
        cnd1[m] = col & yoff & (xb ^ xrb) & (yb ^ yc) & ~(xb ^ yb);
        if (RANDOM && SPEC == 2) {
            const uint32_t cc = cnd0[m] | cnd1[m];
            const uint32_t mx = (cnd0[m] & xa) | (cnd1[m] & xb);
            pmin |= (((cc * 3u) >> (sh2 + 1u)) & kNib) << m;
            pmax |= (((mx * 3u) >> (sh2 + 1u)) & kNib) << m;
        } else if (RANDOM) {
            const uint32_t mn = (cnd0[m] & ~xa) | (cnd1[m] & ~xb);
            const uint32_t mx = (cnd0[m] & xa) | (cnd1[m] & xb);
            const uint32_t cmn = mn & c.p_random, cmx = mx & c.q_random;
            // a cell has at most one candidate, at bit 4j + sh2 + xoff: 3 cmn sets bit
            // 4j + sh2 + 1 for either xoff (no carries: candidates are >= 3 bits apart)
            pmin |= (((cmn * 3u) >> (sh2 + 1u)) & kNib) << m;
            pmax |= (((cmx * 3u) >> (sh2 + 1u)) & kNib) << m;
        }
    }
    if (RANDOM && SPEC == 2) pmin &= ~pmax;  // pmin held every candidate: keep the minima
}

// Phase 3 with sub-cell set (dx, DY): flips of the accepted candidates (acc:
// packed acceptance bits) and the exchange with the neighbouring lanes.
template <int DY, bool RANDOM, int SPEC = 0, class Ctx>
__device__ __forceinline__ void step_apply(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                           uint32_t dx, uint32_t acc, const uint32_t (&cnd0)[4],
                                           const uint32_t (&cnd1)[4], const Ctx &c, const FlipConsts &k, int &net) {
    uint32_t f0s[4], f1s[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int r0 = 4 * m + 2 * DY, r1 = r0 + 1;
        uint32_t amin = c.p_always, amax = c.q_always, spread = 0u;
        if (RANDOM) {
            spread = ((acc >> m) & kNib) * 0xFu;
            amin |= spread & c.p_random;
            amax |= spread & c.q_random;
        }
        const uint32_t xa = X[r0], xb = X[r1];
        // accepted minima are where the candidate has X(s) = 0
        uint32_t f0, f1;
        if (SPEC == 1) {
            f0 = cnd0[m];
            f1 = cnd1[m];
            net += __popc(f0 | f1);  // a thread cell flips in one of the two rows
        } else if (SPEC == 2) {
            f0 = cnd0[m] & spread;  // the draw decides every candidate
            f1 = cnd1[m] & spread;
        } else {
            f0 = cnd0[m] & ((~xa & amin) | (xa & amax));
            f1 = cnd1[m] & ((~xb & amin) | (xb & amax));
            net += always_net<RANDOM>(f0, xa, c) + always_net<RANDOM>(f1, xb, c);
        }
        const uint32_t h0 = signed_flips<SPEC>(f0, xa), h1 = signed_flips<SPEC>(f1, xb);
        X[r0] = h0 * k.neg + xa;
        X[r1] = h1 * k.neg + xb;
        Y[r0] = h0 * k.one + Y[r0];
        Y[r1] = h1 * k.one + (h0 * k.neg + Y[r1]);
        if (r1 + 1 < 16)
            Y[(r1 + 1) & 15] = h1 * k.neg + Y[(r1 + 1) & 15];
        else
            D = h1 * k.neg + D;
        f0s[m] = f0;
        f1s[m] = f1;
    }

    // Keep the neighbour copies consistent (dx is uniform over the warp here).
    if (dx) {
        // Flips at bit 31 changed column 0 of the right neighbour (this lane's E).
        const uint32_t dE = gather_msb_pairs(f0s, f1s) >> (DY ? 0 : 2);
        E ^= dE;
        uint32_t v = __shfl_up_sync(kFull, dE, 1);
        if (SPEC == 1) {
            v = c.gx > 0 ? v >> (2 * DY) : 0u;
            uint32_t w0 = column_fields<1, 0, false>(v, 0u), w1 = column_fields<1, 1, false>(v, 0u);
#pragma unroll
            for (int m = 3; m >= 0; --m) {
                const int r0 = 4 * m + 2 * DY, r1 = r0 + 1;
                X[r0] = mad_hi_signed(w0, k.c16, X[r0]);
                X[r1] = mad_hi_signed(w1, k.c16, X[r1]);
                w0 *= k.c16;
                w1 *= k.c16;
            }
        } else if (c.gx > 0) {  // the signs cost more here than the multiply-adds save
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int r0 = 4 * m + 2 * DY, r1 = r0 + 1;
                X[r0] ^= (v >> r0) & 1u;
                X[r1] ^= (v >> r1) & 1u;
            }
        }
    } else {
        // Flips at bit 0 changed this lane's column 0, mirrored by the left neighbour's E.
        const uint32_t dB0 = gather_lsb_pairs(f0s, f1s) << (DY ? 2 : 0);
        const uint32_t v = __shfl_down_sync(kFull, dB0, 1);
        if (c.gx < c.GX - 1) E ^= v;
    }
    if (DY) {
        // Row 16 (D) belongs to the lane below.
        const uint32_t v = __shfl_up_sync(kFull, f1s[3], c.GX);
        if (c.gy > 0) Y[0] ^= v;
    } else {
        // Row 0 is mirrored by the lane above in its D.
        const uint32_t v = __shfl_down_sync(kFull, f0s[0], c.GX);
        if (c.gy < c.GY - 1) D ^= v;
    }
}

// The same two phases when the lanes of one warp belong to different
// sub-tiles, each with its own set draw: the row offset dy is a run-time value
// per lane (rows picked with selects instead of branches), and every shuffle
// runs unconditionally so that all 32 lanes take part.
template <bool RANDOM, int SPEC = 0, class Ctx>
__device__ __forceinline__ void step_candidates_rt(const uint32_t (&X)[16], const uint32_t (&Y)[16],
                                                   uint32_t E, uint32_t D, const uint4 &site, uint32_t dx,
                                                   uint32_t dy, const Ctx &c,
                                                   uint32_t (&cnd0)[4], uint32_t (&cnd1)[4],
                                                   uint32_t &pmin, uint32_t &pmax) {
    const uint32_t sw[4] = {site.x, site.y, site.z, site.w};  // shifted to the step's field by run_subtile
    // column factor of the set, and the one that brings a candidate's cell to bit 4j+3
    // (the cell's one candidate lies at bit 4j + 2dx + xoff; no carries)
    const uint32_t cs = dx ? 4u : 1u, ps = dx ? 3u : 12u, kc = dx ? kNib * 4u : kNib;
    const uint32_t Es = E >> (2u * dy);
    pmin = 0u;
    pmax = 0u;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t u = sw[m];
        const uint32_t col = (u & kNib) * cs + kc;  // 1 + xoff: one-hot, no carries
        const uint32_t yoff = ((u >> 1) & kNib) * 0xFu;
        const uint32_t xa = dy ? X[4 * m + 2] : X[4 * m];
        const uint32_t xb = dy ? X[4 * m + 3] : X[4 * m + 1];
        const uint32_t ya = dy ? Y[4 * m + 2] : Y[4 * m];
        const uint32_t yb = dy ? Y[4 * m + 3] : Y[4 * m + 1];
        const uint32_t yc = dy ? (m < 3 ? Y[(4 * m + 4) & 15] : D) : Y[4 * m + 2];
        const uint32_t xra = __funnelshift_r(xa, Es >> (4 * m), 1);
        const uint32_t xrb = __funnelshift_r(xb, Es >> (4 * m + 1), 1);
        if (SPEC == 1) {
            cnd0[m] = col & ~yoff & ~xa & xra & ~ya & yb;  // the minima
            cnd1[m] = col & yoff & ~xb & xrb & ~yb & yc;
            continue;
        }
        cnd0[m] = col & ~yoff & (xa ^ xra) & (ya ^ yb) & ~(xa ^ ya);
        cnd1[m] = col & yoff & (xb ^ xrb) & (yb ^ yc) & ~(xb ^ yb);
        if (RANDOM) {
            const uint32_t mx = (cnd0[m] & xa) | (cnd1[m] & xb);
            const uint32_t mn = SPEC == 2 ? cnd0[m] | cnd1[m] : (cnd0[m] & ~xa) | (cnd1[m] & ~xb);
            const uint32_t cmn = SPEC == 2 ? mn : mn & c.p_random, cmx = SPEC == 2 ? mx : mx & c.q_random;
            pmin = ((cmn * ps) & (kNib << 3)) | (pmin >> 1);
            pmax = ((cmx * ps) & (kNib << 3)) | (pmax >> 1);
        }
    }
    if (RANDOM && SPEC == 2) pmin &= ~pmax;  // pmin held every candidate: keep the minima
}

template <bool RANDOM, int SPEC = 0, class Ctx>
__device__ __forceinline__ void step_apply_rt(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                              uint32_t dy, uint32_t acc, const uint32_t (&cnd0)[4],
                                              const uint32_t (&cnd1)[4], const Ctx &c, const FlipConsts &k, uint32_t &E0,
                                              int &net) {
    const uint32_t ro = 2u * dy;
    // the factors with which a flip counts in the rows of one offset and the other
    const uint32_t B = dy, A = 1u - dy, nB = 0u - B, nA = 0u - A;
    uint32_t g0[4], g1[4], f0s[4], f1s[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        uint32_t amin = c.p_always, amax = c.q_always, spread = 0u;
        if (RANDOM) {
            spread = ((acc >> m) & kNib) * 0xFu;
            amin |= spread & c.p_random;
            amax |= spread & c.q_random;
        }
        uint32_t f0, f1, xa = 0u, xb = 0u;
        if (SPEC != 1) {
            xa = dy ? X[4 * m + 2] : X[4 * m];
            xb = dy ? X[4 * m + 3] : X[4 * m + 1];
        }
        if (SPEC == 1) {
            f0 = cnd0[m];
            f1 = cnd1[m];
            net += __popc(f0 | f1);
        } else if (SPEC == 2) {
            f0 = cnd0[m] & spread;
            f1 = cnd1[m] & spread;
        } else {
            f0 = cnd0[m] & ((~xa & amin) | (xa & amax));
            f1 = cnd1[m] & ((~xb & amin) | (xb & amax));
            net += always_net<RANDOM>(f0, xa, c) + always_net<RANDOM>(f1, xb, c);
        }
        const uint32_t h0 = signed_flips<SPEC>(f0, xa), h1 = signed_flips<SPEC>(f1, xb);
        const uint32_t h = h0 * k.neg + h1;
        Y[4 * m] = h0 * A + Y[4 * m];
        Y[4 * m + 1] = h * A + Y[4 * m + 1];
        Y[4 * m + 2] = h0 * B + (h1 * nA + Y[4 * m + 2]);
        Y[4 * m + 3] = h * B + Y[4 * m + 3];
        if (m < 3)
            Y[(4 * m + 4) & 15] = h1 * nB + Y[(4 * m + 4) & 15];
        else
            D = h1 * nB + D;
        g0[m] = h0;  // the changes of X are applied after the exchange
        g1[m] = h1;
        f0s[m] = f0;
        f1s[m] = f1;
    }
    const uint32_t dD = f1s[3] * B, dY0 = f0s[0] * A;
    uint32_t dE = gather_msb_pairs(f0s, f1s) >> 2;
    if (c.GX > 1) {  // warp-uniform: every sub-tile of a warp has the same shape
        dE <<= ro;
        const uint32_t dB0 = gather_lsb_pairs(f0s, f1s) << ro;
        E ^= dE;
        uint32_t vr = __shfl_up_sync(kFull, dE, 1);
        const uint32_t vl = __shfl_down_sync(kFull, dB0, 1);
        vr = c.gx > 0 ? vr : 0u;  // the left lane is in the same sub-tile: same row offset
        const uint32_t vs = vr >> ro, es = E0 >> ro;
        uint32_t w0 = column_fields<SPEC, 0, true>(vs, es), w1 = column_fields<SPEC, 1, true>(vs, es);
        if (SPEC != 1) E0 ^= vr ^ dB0;
#pragma unroll
        for (int m = 3; m >= 0; --m) {
            g0[m] = mad_hi_signed(w0, k.c16, g0[m]);
            g1[m] = mad_hi_signed(w1, k.c16, g1[m]);
            w0 *= k.c16;
            w1 *= k.c16;
        }
        if (c.gx < c.GX - 1) E ^= vl;
    } else {
        E ^= dE << ro;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        X[4 * m] = g0[m] * nA + X[4 * m];
        X[4 * m + 1] = g1[m] * nA + X[4 * m + 1];
        X[4 * m + 2] = g0[m] * nB + X[4 * m + 2];
        X[4 * m + 3] = g1[m] * nB + X[4 * m + 3];
    }
    const uint32_t vd = __shfl_up_sync(kFull, dD, c.GX);
    const uint32_t vu = __shfl_down_sync(kFull, dY0, c.GX);
    if (c.gy > 0) Y[0] ^= vd;
    if (c.gy < c.GY - 1) D ^= vu;
}

// The column 1 << x of every cell's DB site (bits 4j, 4j+1 of the site word u).
__device__ __forceinline__ uint32_t db_column(uint32_t u) {
    const uint32_t base = (u & kNib) + kNib;                // 1 << (x & 1)
    const uint32_t high = base & (((u >> 1) & kNib) * 3u);  // the cells with x >= 2
    return high * 3u + base;
}

// One-hot row masks of a DB step: sel[4m + r] holds, for every cell of TC row m
// whose site lies in its row r, the site's column (site word m: bits 4j, 4j+1
// = x offset, 4j+2, 4j+3 = y offset of cell j).
__device__ __forceinline__ void db_select(const uint4 &site, uint32_t (&sel)[16]) {
    const uint32_t sw[4] = {site.x, site.y, site.z, site.w};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t u = sw[m];
        const uint32_t col = db_column(u);
        const uint32_t C = ((u >> 2) & kNib) * 0xFu, Dd = ((u >> 3) & kNib) * 0xFu;
        sel[4 * m + 0] = col & ~C & ~Dd;
        sel[4 * m + 1] = col & C & ~Dd;
        sel[4 * m + 2] = col & ~C & Dd;
        sel[4 * m + 3] = col & C & Dd;
    }
}

// Flips f[R] of the lane's 16 rows and the exchange with the neighbouring
// lanes (all lanes take part).  Flips of one row may be adjacent here (a last
// column next to a first one), so the second X bit is a shift, not 3f.
template <class Ctx>
__device__ __forceinline__ void db_apply(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                         const uint32_t (&f)[16], const Ctx &c) {
    const uint32_t dE = gather_msb(f), dB0 = gather_lsb(f);
#pragma unroll
    for (int R = 0; R < 16; ++R) {
        X[R] ^= f[R] ^ (f[R] << 1);
        Y[R] ^= R ? f[R] ^ f[R - 1] : f[R];
    }
    D ^= f[15];
    E ^= dE;
    const uint32_t vr = __shfl_up_sync(kFull, dE, 1);
    const uint32_t vl = __shfl_down_sync(kFull, dB0, 1);
    if (c.gx > 0) {
#pragma unroll
        for (int r = 0; r < 16; ++r) X[r] ^= (vr >> r) & 1u;
    }
    if (c.gx < c.GX - 1) E ^= vl;
    const uint32_t vd = __shfl_up_sync(kFull, f[15], c.GX);
    const uint32_t vu = __shfl_down_sync(kFull, f[0], c.GX);
    if (c.gy > 0) Y[0] ^= vd;
    if (c.gy < c.GY - 1) D ^= vu;
}

// One collective step of single-hit DB (dead border) with 4 x 4-site thread
// cells, all attempts of the step decided on the state before it: with one
// rate zero no two accepted flips meet.  Every cell attempts a uniform site of
// the whole cell.  SPEC as for step_candidates: 1 deposition only.
template <bool RANDOM, int SPEC = 0, class Ctx>
__device__ __forceinline__ void db_step(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                        const uint4 &site, uint32_t s, const Ctx &c, TailPool &tp,
                                        int &net, int &draws) {
    uint32_t f[16];  // the attempted sites, then the candidates, then the flips
    db_select(site, f);
#pragma unroll
    for (int R = 0; R < 16; ++R) {
        const uint32_t x = X[R];
        const uint32_t xr = __funnelshift_r(x, E >> R, 1);
        const uint32_t y = Y[R], yd = (R < 15) ? Y[(R + 1) & 15] : D;
        if (SPEC == 1)
            f[R] &= ~x & xr & ~y & yd;  // the minima
        else
            f[R] &= (x ^ xr) & (y ^ yd) & ~(x ^ y);
    }
    uint32_t acc = 0u;
    if (RANDOM) {
        uint32_t pmin = 0u, pmax = 0u;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            uint32_t mn = 0u, mx = 0u;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                mn |= f[4 * m + r] & ~X[4 * m + r];
                mx |= f[4 * m + r] & X[4 * m + r];
            }
            mn &= c.p_random;
            mx &= c.q_random;
            pmin |= ((mn | (mn >> 1) | (mn >> 2) | (mn >> 3)) & kNib) << m;
            pmax |= ((mx | (mx >> 1) | (mx >> 2) | (mx >> 3)) & kNib) << m;
        }
        draws += __popc(pmin | pmax);
        acc = accept_candidates<kPreDb>(pmin, pmax, level_words(s, c), c, tp);
        net += random_net(acc, pmin, pmax);
    }
#pragma unroll
    for (int R = 0; R < 16; ++R) {
        if (SPEC == 1) {
            net += __popc(f[R]);
            continue;
        }
        const uint32_t x = X[R];
        uint32_t amin = c.p_always, amax = c.q_always;
        if (RANDOM) {
            const uint32_t spread = ((acc >> (R >> 2)) & kNib) * 0xFu;
            amin |= spread & c.p_random;
            amax |= spread & c.q_random;
        }
        f[R] &= (~x & amin) | (x & amax);
        net += always_net<RANDOM>(f[R], x, c);
    }
    db_apply(X, Y, E, D, f, c);
}

// The four leading bits of every cell's uniform against P32's, for p and for q:
// below (lt) and equal (eq), from the last level up.
struct LevelCmp {
    uint32_t ltp, eqp, ltq, eqq;
};
template <class Ctx>
__device__ __forceinline__ LevelCmp level_compare(const uint4 &W, const Ctx &c) {
    const uint32_t lw[4] = {W.x, W.y, W.z, W.w};
    LevelCmp v{0u, kFull, 0u, kFull};
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        const uint32_t tp = (c.thr_p >> (31 - i)) & 1u ? kFull : 0u, tq = (c.thr_q >> (31 - i)) & 1u ? kFull : 0u;
        v.ltp = (tp & ~lw[i]) | (~(tp ^ lw[i]) & v.ltp);
        v.eqp &= ~(tp ^ lw[i]);
        v.ltq = (tq & ~lw[i]) | (~(tq ^ lw[i]) & v.ltq);
        v.eqq &= ~(tq ^ lw[i]);
    }
    return v;
}

// Bitwise v[2 d + c].
__device__ __forceinline__ uint32_t mux4(uint32_t c, uint32_t d, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
    const uint32_t lo = (c & v1) | (~c & v0), hi = (c & v3) | (~c & v2);
    return (d & hi) | (~d & lo);
}

// Four words holding one value bit per cell of TC row m in nibble j (at most
// one bit set, at any of its four places; a zero nibble is 0): packed to bit
// 4j+m.  The words are folded in pairs, so that a fold serves two of them.
__device__ __forceinline__ uint32_t pack_cells(uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
    constexpr uint32_t k3 = 0x33333333u, k5 = 0x55555555u;
    v0 |= v0 >> 2;
    v1 |= v1 >> 2;
    v2 |= v2 >> 2;
    v3 |= v3 >> 2;
    uint32_t a = (v0 & k3) | ((v2 << 2) & ~k3);  // bits 0, 1: TC row 0; bits 2, 3: TC row 2
    uint32_t b = (v1 & k3) | ((v3 << 2) & ~k3);
    a |= a >> 1;
    b |= b >> 1;
    return (a & k5) | ((b << 1) & ~k5);
}

// The cells' bit b of their site word nibbles for all TC rows: q[b] bit 4j+m =
// bit 4j+b of word m (a 4 x 4 transposition in every nibble).
__device__ __forceinline__ void transpose_nibbles(const uint4 &site, uint32_t (&q)[4]) {
    constexpr uint32_t k3 = 0x33333333u, k5 = 0x55555555u;
    const uint32_t a0 = (site.x & k5) | ((site.y << 1) & ~k5), a1 = ((site.x >> 1) & k5) | (site.y & ~k5);
    const uint32_t b0 = (site.z & k5) | ((site.w << 1) & ~k5), b1 = ((site.z >> 1) & k5) | (site.w & ~k5);
    q[0] = (a0 & k3) | ((b0 << 2) & ~k3);
    q[1] = (a1 & k3) | ((b1 << 2) & ~k3);
    q[2] = ((a0 >> 2) & k3) | (b0 & ~k3);
    q[3] = ((a1 >> 2) & k3) | (b1 & ~k3);
}

// The DB step with delayed borders (both rates non-zero): bulk attempts, then
// border attempts (last column x = 3 or last row y = 3 of a cell, where an
// update reaches the next cell), then corner attempts (both), each decided on
// the state the earlier ones left.
//
// The rows are visited twice only, once to read the four slope bits of every
// attempt and once to flip, instead of in each of the three phases: a cell
// makes one attempt a step, so the only flips that a later attempt can see
// are those of the cell to its right at the same height (it changes X(s+x) of
// a border attempt in the last column by a bulk flip at x = 0, and of a corner
// by a border flip at (0, 3)) and of the cell below it at the same column
// (Y(s+y), by a bulk flip at y = 0, and for a corner by a border flip at
// (3, 0)).  So the phases run on words of one bit per cell (bit 4j+m, where
// the acceptance draws are anyway): a = X(s) != X(s+x) and b = Y(s) != Y(s+y)
// before the step, toggled where such a flip was accepted.  A third fewer
// shuffles too (8 instead of 12).  Bound by the integer pipe on large
// lattices and by latency where a step has few warps per scheduler: 2 MCS of
// L=12288 (256x64, p=0.95, q=0.05; 3.8 warps per scheduler) went from 628 to
// 511 us, and from 465 to 437 us when the attempt's row is picked by bit masks
// (three selects per quantity instead of an and-or per row) and one comparison
// of the level words serves the three phases.
template <bool RANDOM, int SPEC = 0, int TIES = kTiesAsk, class Ctx>
__device__ __forceinline__ void db_step_delayed(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                                const uint4 &site, uint32_t s, const Ctx &c, TailPool &tp,
                                                int &net, int &draws) {
    const uint32_t sw[4] = {site.x, site.y, site.z, site.w};
    uint32_t col[4], C[4], Dd[4];  // the site's column, one-hot; its row's bits, over the cell
    uint32_t a[4], b[4], lo[4], hi[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t u = sw[m];
        col[m] = db_column(u);
        C[m] = ((u >> 2) & kNib) * 0xFu;
        Dd[m] = ((u >> 3) & kNib) * 0xFu;
        uint32_t x[4], xr[4], y[5];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int R = 4 * m + r;
            x[r] = X[R];
            xr[r] = __funnelshift_r(x[r], E >> R, 1);
            y[r] = Y[R];
        }
        y[4] = m < 3 ? Y[(4 * m + 4) & 15] : D;
        const uint32_t xs = mux4(C[m], Dd[m], x[0], x[1], x[2], x[3]), xn = mux4(C[m], Dd[m], xr[0], xr[1], xr[2], xr[3]);
        const uint32_t ys = mux4(C[m], Dd[m], y[0], y[1], y[2], y[3]), yn = mux4(C[m], Dd[m], y[1], y[2], y[3], y[4]);
        a[m] = col[m] & (xs ^ xn);
        b[m] = col[m] & (ys ^ yn);
        lo[m] = col[m] & ~xs & ~ys;
        hi[m] = col[m] & xs & ys;
    }
    uint32_t A = pack_cells(a[0], a[1], a[2], a[3]), B = pack_cells(b[0], b[1], b[2], b[3]);
    const uint32_t LO = pack_cells(lo[0], lo[1], lo[2], lo[3]);  // X(s) = Y(s) = 0: a minimum where a and b
    const uint32_t HI = pack_cells(hi[0], hi[1], hi[2], hi[3]);  // X(s) = Y(s) = 1: a maximum
    uint32_t q[4];
    transpose_nibbles(site, q);
    const uint32_t x0 = q[0], x1 = q[1], y0 = q[2], y1 = q[3];  // site coordinates in the cell
    const uint32_t xlast = x0 & x1, ylast = y0 & y1;
    LevelCmp lv{0u, 0u, 0u, 0u};
    if (RANDOM) lv = level_compare(level_words(s, c), c);
    uint32_t dmin = 0u, dmax = 0u, dacc = 0u;  // candidates decided by draws, and those accepted

    // accepted flips of one phase (cls: its cells)
    auto phase = [&](uint32_t cls) {
        const uint32_t can = A & B & cls, mn = can & LO, mx = can & HI;
        uint32_t f = 0u;
        if (RANDOM) {
            const uint32_t pmin = SPEC == 2 ? mn : mn & c.p_random, pmax = SPEC == 2 ? mx : mx & c.q_random;
            f = resolve_ties<kPreDb, TIES>((pmin & lv.ltp) | (pmax & lv.ltq), (pmin & lv.eqp) | (pmax & lv.eqq), pmin, c, tp);
            dmin |= pmin;
            dmax |= pmax;
            dacc |= f;
        }
        if (SPEC != 2) {
            const uint32_t fn = mn & c.p_always, fx = mx & c.q_always;
            net += __popc(fn) - __popc(fx);
            f |= fn | fx;
        }
        return f;
    };
    // v of the cell to the right (from the next lane's low nibble vr) and below (vb: the next lane row's TC row 0)
    auto right = [](uint32_t v, uint32_t vr) { return __funnelshift_r(v, vr, 4); };
    auto below = [](uint32_t v, uint32_t vb) { return ((v >> 1) & 0x77777777u) | ((vb & kNib) << 3); };
    const bool has_r = c.gx < c.GX - 1, has_b = c.gy < c.GY - 1;

    uint32_t F = phase(~(xlast | ylast));  // bulk
    {
        const uint32_t gl = F & ~(x0 | x1), gt = F & ~(y0 | y1);  // flips in a cell's first column, first row
        uint32_t pr = (gl & 15u) | ((y0 & 15u) << 4) | ((y1 & 15u) << 8);
        uint32_t pb = (gt & kNib) | ((x0 & kNib) << 1) | ((x1 & kNib) << 2);
        pr = __shfl_down_sync(kFull, pr, 1);
        pb = __shfl_down_sync(kFull, pb, c.GX);
        if (!has_r) pr = 0u;
        if (!has_b) pb = 0u;
        A ^= xlast & right(gl, pr) & ~(y0 ^ right(y0, pr >> 4)) & ~(y1 ^ right(y1, pr >> 8));
        B ^= ylast & below(gt, pb) & ~(x0 ^ below(x0, pb >> 1)) & ~(x1 ^ below(x1, pb >> 2));
    }
    const uint32_t F2 = phase(xlast ^ ylast);  // borders
    {
        const uint32_t gl = F2 & ~(x0 | x1) & ylast, gt = F2 & ~(y0 | y1) & xlast;
        uint32_t pr = __shfl_down_sync(kFull, gl, 1), pb = __shfl_down_sync(kFull, gt, c.GX);
        if (!has_r) pr = 0u;
        if (!has_b) pb = 0u;
        A ^= right(gl, pr);
        B ^= below(gt, pb);
    }
    F |= F2 | phase(xlast & ylast);  // corners
    if (RANDOM) {
        draws += __popc(dmin | dmax);
        net += random_net(dacc, dmin, dmax);
    }
    uint32_t f[16];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t fc = col[m] & (((F >> m) & kNib) * 0xFu);
        f[4 * m + 0] = fc & ~C[m] & ~Dd[m];
        f[4 * m + 1] = fc & C[m] & ~Dd[m];
        f[4 * m + 2] = fc & ~C[m] & Dd[m];
        f[4 * m + 3] = fc & C[m] & Dd[m];
    }
    db_apply(X, Y, E, D, f, c);
}

// A collective step of DTrDTr (Sec. 4.1.2): DT whose
// block-layer origin moves after every step, the cell grid wrapping around
// the sub-tile.  With the active sub-cell of every cell starting at column c0
// and row R0 (uniform in [0, 4): the set's offset plus the moved origin), the
// attempt of TC (j, m) of a lane is at (4j + c0 + rx, 4m + R0 + ry).  For
// c0 = 3 the pair of TC 7 reaches column 32, i.e. column 0 of the lane to the
// right (of the sub-tile's first lane, for the last lane: the wrap); for
// R0 = 3 the pair of TC row 3 reaches row 16, row 0 of the lane below (or of
// the first lane row), and TC (7, 3) can reach the lane diagonally below.
// The lane holding such a site tests it; the candidate goes back to the
// owning lane, which draws its acceptance with its own level words (so the
// uniforms, and the order of ties, stay those of the owning thread cell), and
// the decision returns to the holder, which flips.  The neighbour copies E, D
// are kept as in DT: the lattice itself does not wrap inside the sub-tile.
// As for DT the step runs in three phases, with one copy of the acceptance code
// between the candidates and the flips.
// PACKED: the warp holds several sub-tiles, each with its own phase (c0, R0),
// so every shuffle runs on all lanes and its value is taken where the lane's
// phase asks for it (a lane only reads lanes of its own sub-tile).
struct DtrLanes {
    int lL, lR, lA, lB, lAL, lBR;  // lanes of the sub-tile left, right, above, below, above-left, below-right (wrapping)
};

template <class Ctx>
__device__ __forceinline__ DtrLanes dtr_lanes(const Ctx &c) {
    const int gxl = c.gx == 0 ? c.GX - 1 : c.gx - 1, gxr = c.gx == c.GX - 1 ? 0 : c.gx + 1;
    const int gya = c.gy == 0 ? c.GY - 1 : c.gy - 1, gyb = c.gy == c.GY - 1 ? 0 : c.gy + 1;
    DtrLanes n;
    n.lL = c.base + gxl + c.gy * c.GX;
    n.lR = c.base + gxr + c.gy * c.GX;
    n.lA = c.base + c.gx + gya * c.GX;
    n.lB = c.base + c.gx + gyb * c.GX;
    n.lAL = c.base + gxl + gya * c.GX;
    n.lBR = c.base + gxr + gyb * c.GX;
    return n;
}

// v[k] for a run-time k in 0..3 (selects, no branch).
__device__ __forceinline__ uint32_t pick4(uint32_t k, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
    const uint32_t lo = (k & 1u) ? v1 : v0, hi = (k & 1u) ? v3 : v2;
    return (k & 2u) ? hi : lo;
}

// Phase 1.  The row phase R0 is a run-time value (one copy of the code for all
// four phases; four specialised copies overflowed the instruction caches).
// ca[m], cb[m]: candidates in rows a = 4m+R0 and b = a+1 held by this lane;
// row 16 (m = 3, R0 = 3) is the lane below's row 0, and cb[3] then holds this
// lane's row 0 (the wrapped row of the lane above) instead.
// pmin / pmax: packed candidates of this lane's own thread cells.
template <bool RANDOM, bool PACKED, class Ctx>
__device__ __forceinline__ void dtr_candidates(const uint32_t (&X)[16], const uint32_t (&Y)[16], uint32_t E,
                                               uint32_t D, const uint4 &site, uint32_t s, uint32_t c0,
                                               uint32_t R0, const Ctx &c, const DtrLanes &n,
                                               uint32_t (&ca)[4], uint32_t (&cb)[4], uint32_t &pmin,
                                               uint32_t &pmax) {
    const bool SX = c0 == 3u;  // pairs reach column 32
    const bool SY = R0 == 3u;  // pairs reach row 16
    const uint32_t sw[4] = {site.x, site.y, site.z, site.w};
    const uint32_t par = 2u * (s & 1u);
    // Selected sites: own thread cells in place, those past column 31 in xw
    // (bit = row; bit 16 = row 16), those in row 16 in yw (bit = column).
    uint32_t xw = 0u, yw = 0u;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint32_t u = sw[m] >> par;
        const uint32_t col = ((u & kNib) << 1) | (~u & kNib);  // bit 4j + rx
        const uint32_t yoff = ((u >> 1) & kNib) * 0xFu;         // thread cells with ry = 1
        const uint64_t a64 = static_cast<uint64_t>(col & ~yoff) << c0;
        const uint64_t b64 = static_cast<uint64_t>(col & yoff) << c0;
        const uint32_t ya = 4u * m + R0;
        ca[m] = static_cast<uint32_t>(a64);
        xw |= static_cast<uint32_t>(a64 >> 32) << ya;
        if (m == 3 && SY) {
            cb[m] = 0u;
            yw = static_cast<uint32_t>(b64);
            xw |= static_cast<uint32_t>(b64 >> 32) << 16;
        } else {
            cb[m] = static_cast<uint32_t>(b64);
            xw |= static_cast<uint32_t>(b64 >> 32) << (ya + 1u);
        }
    }
    // sites of neighbouring lanes' thread cells held by this lane
    if (PACKED || SX) {
        uint32_t v = __shfl_sync(kFull, xw, n.lL);
        if (PACKED) v = SX ? v : 0u;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t ya = 4u * m + R0;
            ca[m] |= (v >> ya) & 1u;
            if (!(m == 3 && SY)) cb[m] |= (v >> (ya + 1u)) & 1u;
        }
    }
    if (PACKED || SY) {
        const uint32_t v = __shfl_sync(kFull, yw, n.lA);
        uint32_t corner = 0u;
        if (PACKED || SX) corner = (__shfl_sync(kFull, xw, n.lAL) >> 16) & (SX ? 1u : 0u);
        if (SY) cb[3] = v | corner;  // row 0
    }
    // eligibility; rows a and b of TC row m picked by the row phase (for
    // m = 3 the row after 15 is D for Y, and row b = "16" is row 0)
    uint32_t cw = 0u;  // column-0 candidates: minima in bits 0..15, maxima in 16..31 (row = bit)
    uint32_t xa_[4], xb_[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int r = 4 * m;
        const uint32_t X4 = m < 3 ? X[(r + 4) & 15] : X[0];
        const uint32_t Y4 = m < 3 ? Y[(r + 4) & 15] : D;
        const uint32_t Yb4 = m < 3 ? Y[(r + 4) & 15] : Y[0];  // row b's own Y when b = "16"
        const uint32_t Y5 = m < 3 ? Y[(r + 5) & 15] : Y[1];
        const uint32_t ya = static_cast<uint32_t>(r) + R0, yb = (ya + 1u) & 15u;
        const uint32_t xa = pick4(R0, X[r], X[r + 1], X[r + 2], X[r + 3]);
        const uint32_t yA = pick4(R0, Y[r], Y[r + 1], Y[r + 2], Y[r + 3]);
        const uint32_t yAd = pick4(R0, Y[r + 1], Y[r + 2], Y[r + 3], Y4);
        const uint32_t xb = pick4(R0, X[r + 1], X[r + 2], X[r + 3], X4);
        const uint32_t yB = pick4(R0, Y[r + 1], Y[r + 2], Y[r + 3], Yb4);
        const uint32_t yBd = pick4(R0, Y[r + 2], Y[r + 3], Y4, Y5);
        ca[m] &= (xa ^ __funnelshift_r(xa, E >> ya, 1)) & (yA ^ yAd) & ~(xa ^ yA);
        cb[m] &= (xb ^ __funnelshift_r(xb, E >> yb, 1)) & (yB ^ yBd) & ~(xb ^ yB);
        xa_[m] = xa;
        xb_[m] = xb;
        if (RANDOM) {
            cw |= ((ca[m] & ~xa & 1u) << ya) | ((ca[m] & xa & 1u) << (ya + 16u));
            cw |= ((cb[m] & ~xb & 1u) << yb) | ((cb[m] & xb & 1u) << (yb + 16u));
        }
    }
    pmin = 0u;
    pmax = 0u;
    if (RANDOM) {
        uint32_t cwR = 0u, cwBR = 0u;
        if (PACKED || SX) cwR = __shfl_sync(kFull, cw, n.lR);
        if (PACKED || (SX && SY)) cwBR = __shfl_sync(kFull, cw, n.lBR);
        if (PACKED && !SX) cwR = cwBR = 0u;
        uint32_t bmin = 0u, bmax = 0u;  // row 0 of the lane below (used with R0 = 3)
        if (PACKED || SY) {
            bmin = __shfl_sync(kFull, cb[3] & ~X[0], n.lB);
            bmax = __shfl_sync(kFull, cb[3] & X[0], n.lB);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t ya = 4u * m + R0, yb = ya + 1u;
            uint32_t mnl = ca[m] & ~xa_[m], mxl = ca[m] & xa_[m];
            uint32_t mnh = (cwR >> ya) & 1u, mxh = (cwR >> (ya + 16u)) & 1u;
            if (m == 3 && SY) {
                mnl |= bmin;
                mxl |= bmax;
                mnh |= cwBR & 1u;
                mxh |= (cwBR >> 16) & 1u;
            } else {
                mnl |= cb[m] & ~xb_[m];
                mxl |= cb[m] & xb_[m];
                mnh |= (cwR >> yb) & 1u;
                mxh |= (cwR >> (yb + 16u)) & 1u;
            }
            // align each cell's pair to bits 4j, 4j+1, then pack to bit 4j+m
            const uint32_t cmn = __funnelshift_r(mnl, mnh, c0) & c.p_random;
            const uint32_t cmx = __funnelshift_r(mxl, mxh, c0) & c.q_random;
            pmin |= ((cmn | (cmn >> 1)) & kNib) << m;
            pmax |= ((cmx | (cmx >> 1)) & kNib) << m;
        }
        // A lane outside the sub-tile can read a sub-tile lane's candidates
        // through the wrapped lane indices; it owns no thread cell.
        if (!c.active) {
            pmin = 0u;
            pmax = 0u;
        }
    }
}

// Phase 3: flips of the accepted candidates (acc: this lane's packed
// acceptance bits), then the exchange of the neighbour copies.  The flips of
// row r come from TC row m = r / 4 when r % 4 is R0 (row a) or R0 + 1 (row b),
// and from TC row m - 1 (mod 4: row 0 takes the wrapped row of TC row 3) when
// r % 4 = 0 and R0 = 3.
template <bool RANDOM, bool PACKED, class Ctx>
__device__ __forceinline__ void dtr_apply(uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D,
                                          uint32_t c0, uint32_t R0, uint32_t acc, const uint32_t (&ca)[4],
                                          const uint32_t (&cb)[4], const Ctx &c, const DtrLanes &n,
                                          int &net) {
    const bool SX = c0 == 3u;
    const bool SY = R0 == 3u;
    uint32_t accL = 0u, accA = 0u, accAL = 0u;
    if (RANDOM) {
        // (read only by the columns and rows that wrap)
        if (PACKED || SX) accL = __shfl_sync(kFull, acc, n.lL);
        if (PACKED || SY) accA = __shfl_sync(kFull, acc, n.lA);
        if (PACKED || (SX && SY)) accAL = __shfl_sync(kFull, acc, n.lAL);
    }
    // accepted candidates of rows a and b of every TC row (fb[3] with R0 = 3: row 0)
    uint32_t fa[4], fb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int r = 4 * m;
        const uint32_t xa = pick4(R0, X[r], X[r + 1], X[r + 2], X[r + 3]);
        const uint32_t xb = pick4(R0, X[r + 1], X[r + 2], X[r + 3], m < 3 ? X[(r + 4) & 15] : X[0]);
        uint32_t amin = c.p_always, amax = c.q_always, bmin = c.p_always, bmax = c.q_always;
        if (RANDOM) {
            const uint32_t own = ((acc >> m) & kNib) * 0xFu;
            const uint32_t left = ((accL >> m) & kNib) * 0xFu;
            const uint32_t cols = __funnelshift_l(left, own, c0);
            // row 0 with R0 = 3: thread cells of the lanes above
            const uint32_t cols0 = __funnelshift_l(((accAL >> 3) & kNib) * 0xFu, ((accA >> 3) & kNib) * 0xFu, c0);
            const uint32_t colb = (m == 3 && SY) ? cols0 : cols;
            amin |= cols & c.p_random;
            amax |= cols & c.q_random;
            bmin |= colb & c.p_random;
            bmax |= colb & c.q_random;
        }
        fa[m] = ca[m] & ((~xa & amin) | (xa & amax));
        fb[m] = cb[m] & ((~xb & bmin) | (xb & bmax));
        net += always_net<RANDOM>(fa[m], xa, c) + always_net<RANDOM>(fb[m], xb, c);
    }
    uint32_t F_prev = 0u, dE = 0u, dB0 = 0u;  // gathered as in gather_lsb; dE in reverse order
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int m = r >> 2;
        const uint32_t k = static_cast<uint32_t>(r & 3);
        uint32_t F = (R0 == k ? fa[m] : 0u) | (R0 + 1u == k ? fb[m] : 0u);
        if (k == 0u && SY) F |= fb[(m + 3) & 3];
        X[r] ^= F * 3u;      // F ^ (F << 1): the row's flips are at least three columns apart
        Y[r] ^= F ^ F_prev;  // its own Y, and Y(s+y) of the row above
        dE = __funnelshift_l(F, dE, 1);
        dB0 = __funnelshift_r(dB0, F, 1);
        F_prev = F;
    }
    dE = __brev(dE) >> 16;
    dB0 >>= 16;
    D ^= F_prev;  // Y(s+y) of row 15
    const uint32_t dD = F_prev;
    const uint32_t dY0 = (R0 == 0u ? fa[0] : 0u) | (SY ? fb[3] : 0u);  // the flips of row 0
    E ^= dE;
    const uint32_t vr = __shfl_up_sync(kFull, dE, 1);
    const uint32_t vl = __shfl_down_sync(kFull, dB0, 1);
    if (c.gx > 0) {
#pragma unroll
        for (int r = 0; r < 16; ++r) X[r] ^= (vr >> r) & 1u;
    }
    if (c.gx < c.GX - 1) E ^= vl;
    const uint32_t vd = __shfl_up_sync(kFull, dD, c.GX);
    const uint32_t vu = __shfl_down_sync(kFull, dY0, c.GX);
    if (c.gy > 0) Y[0] ^= vd;
    if (c.gy < c.GY - 1) D ^= vu;
}

// Where a lane's group lies in the planar lattice: the two words wA, wB of
// every row that hold its 32 sites (from bit sh of wA), and its first row ybase.
struct LaneGeom {
    uint32_t *Xp, *Yp;
    uint32_t sh, wA, wB, ybase;
};

// (y0 in buffer rows; the Y plane follows plane_rows rows of X.)
template <class Ctx>
__device__ __forceinline__ LaneGeom lane_geom(uint32_t *lat, uint32_t L, uint32_t plane_rows, uint32_t wpr,
                                              uint32_t x0, uint32_t y0, const Ctx &c) {
    LaneGeom q;
    q.Xp = lat;
    q.Yp = lat + static_cast<size_t>(plane_rows) * wpr;
    q.sh = x0 & 31u;
    q.wA = ((x0 >> 5) + static_cast<uint32_t>(c.gx)) % wpr;
    q.wB = (q.wA + 1u == wpr) ? 0u : q.wA + 1u;
    q.ybase = y0 + 16u * static_cast<uint32_t>(c.gy);
    if (q.ybase >= L) q.ybase -= L;
    return q;
}

// The staging and the write-back of a lane, 33 rows' words each, were a ninth
// of the instructions of a device step when every row's address was formed
// anew: one MCS at L=2^17 (1024x16, p=0.95, q=0.05) went from 11.15 to 10.1 ms
// with running addresses, and with E and D taken from the words read instead
// of by shuffles and loads of the edge lanes.
//
// Row r of the lane's group in words from the planes' start.  STRAIGHT: neither
// the rows nor the two words of any lane of the warp wrap around the lattice,
// so a row is one addition from the last and word wB follows wA; a warp that
// wraps (one in about L/32 by words, L/16 by rows) takes the general form.
template <bool STRAIGHT>
struct LaneRows {
    const LaneGeom &q;
    uint32_t L, wpr;
    size_t at;     // word wA of the current row
    uint32_t row;  // the current row
    __device__ __forceinline__ LaneRows(const LaneGeom &g, uint32_t L_, uint32_t wpr_)
        : q(g), L(L_), wpr(wpr_), at(static_cast<size_t>(g.ybase) * wpr_ + g.wA), row(g.ybase) {}
    __device__ __forceinline__ void next() {
        at += wpr;
        if (!STRAIGHT && ++row == L) {
            row = 0u;
            at = q.wA;
        }
    }
    __device__ __forceinline__ size_t a() const { return at; }
    __device__ __forceinline__ size_t b() const { return STRAIGHT ? at + 1u : at - q.wA + q.wB; }
};

// Stage the lane's group: 16 rows of X and Y, funnel-shifted to local bit 0;
// E: column 32 of its rows (column 0 of the right neighbour, or the sub-tile's
// halo column); D: its row 16 of Y (row 0 of the lane below, or the halo row).
template <bool STRAIGHT>
__device__ __forceinline__ void load_lane_rows(const LaneGeom &q, uint32_t L, uint32_t wpr, uint32_t (&X)[16],
                                               uint32_t (&Y)[16], uint32_t &E, uint32_t &D) {
    LaneRows<STRAIGHT> w(q, L, wpr);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const uint32_t xb = q.Xp[w.b()];
        X[r] = __funnelshift_r(q.Xp[w.a()], xb, q.sh);
        Y[r] = __funnelshift_r(q.Yp[w.a()], q.Yp[w.b()], q.sh);
        E = __funnelshift_r(E, xb >> q.sh, 1);
        w.next();
    }
    E >>= 16;
    D = __funnelshift_r(q.Yp[w.a()], q.Yp[w.b()], q.sh);
}

__device__ __forceinline__ bool lane_straight(const LaneGeom &q, uint32_t L, bool active) {
    return __all_sync(kFull, !active || (q.ybase + 17u <= L && q.wB == q.wA + 1u));
}

__device__ __forceinline__ void stage_lane(const LaneGeom &q, uint32_t L, uint32_t wpr, bool straight, bool active,
                                           uint32_t (&X)[16], uint32_t (&Y)[16], uint32_t &E, uint32_t &D) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        X[r] = 0u;
        Y[r] = 0u;
    }
    E = 0u;
    D = 0u;
    if (active) {
        if (straight)
            load_lane_rows<true>(q, L, wpr, X, Y, E, D);
        else
            load_lane_rows<false>(q, L, wpr, X, Y, E, D);
    }
}

// Write back.  Global word wA of a row receives the high bits of the left lane
// and the low bits of this lane; the leftmost lane shares word wA with the
// bits left of x0, the rightmost lane also owns the low bits of word wB (its
// own high bits, and for X the halo-column bit).  The bits of those shared
// words outside the sub-tile belong to neighbouring sub-tiles, which this
// device step does not update, and no other warp writes these words (active
// sub-tiles are at least 32 sites apart).  Full words are stored.  Shared words
// are merged in one of two ways:
//  * a warp holding one sub-tile (few shared words per lane): an AND/OR
//    reduction pair, which returns nothing, so the warp does not wait;
//  * a warp holding several small sub-tiles (many shared words per lane): a
//    fresh read of the outside bits, all reads of eight rows before their
//    stores (one wait for memory per eight rows), and one plain store per
//    word; there the reductions' throughput would bind the step.
template <bool LANE_SETS, bool STRAIGHT, class Ctx>
__device__ __forceinline__ void store_lane_rows(const LaneGeom &q, uint32_t L, uint32_t wpr, bool active,
                                                const Ctx &c, const uint32_t (&X)[16], const uint32_t (&Y)[16],
                                                uint32_t E, uint32_t D) {
    uint32_t *const Xp = q.Xp;
    uint32_t *const Yp = q.Yp;
    const uint32_t sh = q.sh;
    const bool left_edge = active && c.gx == 0 && sh != 0u;
    const bool right_edge = active && c.gx == c.GX - 1;
    const uint32_t lo_mask = (1u << sh) - 1u;  // bits [0, sh): left of x0 in word wA
    const uint32_t xb_mask = (2u << sh) - 1u;  // bits [0, sh]: ours in word wB of X (halo bit at sh)
    LaneRows<STRAIGHT> w(q, L, wpr);
#pragma unroll
    for (int h = 0; h < 16; h += 8) {
        uint32_t oX[8], oY[8];  // outside bits of the lane's edge words (wA's in lo_mask, wB's above)
        if (LANE_SETS) {
            LaneRows<STRAIGHT> v = w;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                oX[i] = 0u;
                oY[i] = 0u;
                if (left_edge) {
                    oX[i] = Xp[v.a()] & lo_mask;
                    oY[i] = Yp[v.a()] & lo_mask;
                }
                if (right_edge) {
                    oX[i] |= Xp[v.b()] & ~xb_mask;
                    oY[i] |= Yp[v.b()] & ~lo_mask;
                }
                v.next();
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = h + i;
            const uint32_t leftX = __shfl_up_sync(kFull, X[r], 1);
            const uint32_t leftY = __shfl_up_sync(kFull, Y[r], 1);
            if (active) {
                const size_t A = w.a(), B = w.b();
                if (left_edge) {
                    if (LANE_SETS) {
                        Xp[A] = (oX[i] & lo_mask) | (X[r] << sh);
                        Yp[A] = (oY[i] & lo_mask) | (Y[r] << sh);
                    } else {
                        reduce_bits(&Xp[A], X[r] << sh, ~lo_mask);
                        reduce_bits(&Yp[A], Y[r] << sh, ~lo_mask);
                    }
                } else {
                    Xp[A] = __funnelshift_l(leftX, X[r], sh);
                    Yp[A] = __funnelshift_l(leftY, Y[r], sh);
                }
                if (right_edge) {
                    const uint32_t hiX = (sh ? (X[r] >> (32u - sh)) : 0u) | (((E >> r) & 1u) << sh);
                    const uint32_t hiY = sh ? (Y[r] >> (32u - sh)) : 0u;
                    if (LANE_SETS) {
                        Xp[B] = (oX[i] & ~xb_mask) | hiX;
                        if (sh) Yp[B] = (oY[i] & ~lo_mask) | hiY;
                    } else {
                        reduce_bits(&Xp[B], hiX, xb_mask);
                        if (sh) reduce_bits(&Yp[B], hiY, lo_mask);
                    }
                }
            }
            w.next();
        }
    }
    {
        const bool d_row = active && c.gy == c.GY - 1;  // the halo row, below the sub-tile's last lanes
        const size_t A = w.a(), B = w.b();
        uint32_t oD = 0u;
        if (LANE_SETS && d_row) {
            if (left_edge) oD = Yp[A] & lo_mask;
            if (right_edge && sh) oD |= Yp[B] & ~lo_mask;
        }
        const uint32_t leftD = __shfl_up_sync(kFull, D, 1);
        if (d_row) {
            if (left_edge) {
                if (LANE_SETS)
                    Yp[A] = (oD & lo_mask) | (D << sh);
                else
                    reduce_bits(&Yp[A], D << sh, ~lo_mask);
            } else {
                Yp[A] = __funnelshift_l(leftD, D, sh);
            }
            if (right_edge && sh) {
                if (LANE_SETS)
                    Yp[B] = (oD & ~lo_mask) | (D >> (32u - sh));
                else
                    reduce_bits(&Yp[B], D >> (32u - sh), lo_mask);
            }
        }
    }
}

template <bool LANE_SETS, class Ctx>
__device__ __forceinline__ void write_back(const LaneGeom &q, uint32_t L, uint32_t wpr, bool straight, bool active,
                                           const Ctx &c, const uint32_t (&X)[16], const uint32_t (&Y)[16],
                                           uint32_t E, uint32_t D) {
    if (straight)
        store_lane_rows<LANE_SETS, true>(q, L, wpr, active, c, X, Y, E, D);
    else
        store_lane_rows<LANE_SETS, false>(q, L, wpr, active, c, X, Y, E, D);
}

// Device step on one sub-tile (Bx x By sites at (x0, y0)) held by the lanes of
// one warp that share it: stage the lane's group from the planar lattice,
// run the 16 single-hit collective steps, write back.  LANE_SETS: lanes of the
// warp may belong to different sub-tiles (each with its own set draws).
// SCHEME: 0 DTrDT, 1 DTrDB with all attempts of a step together, 2 DTrDB with
// delayed borders, 3 DTrDTr, 4 DTrDT with deposition only (p = 1, q = 0),
// 5 DTrDT with both rates strictly inside (0, 1), 6 DTrDB with deposition only,
// 7 DTrDB with delayed borders and both rates random, 8 and 9 as 5 and 7 with
// rates for which every tie is refused, 10 as 5 for rates of either kind.
template <bool RANDOM, bool LANE_SETS, int SCHEME = 0, class Ctx>
__device__ __forceinline__ void run_subtile(uint32_t *lat, uint32_t L, uint32_t plane_rows, uint32_t wpr,
                                            uint32_t x0, uint32_t y0, bool active, const Ctx &c, uint32_t *ring, int &net, int &draws,
                                            int &tails) {
    TailPool tp;
    tp.ring = ring + static_cast<uint32_t>(kRingWordsPerLane) * c.g;  // the lane's own slot
    tp.head = 0u;
    tp.end = 0u;
    tp.rounds = 0u;
    const LaneGeom q = lane_geom(lat, L, plane_rows, wpr, x0, y0, c);
    uint32_t X[16], Y[16], E, D;
    wait_for_previous_grid();  // nothing above reads the lattice
    const bool straight = lane_straight(q, L, active);
    stage_lane(q, L, wpr, straight, active, X, Y, E, D);

    const FlipConsts flips;
    uint32_t E0 = 0u;  // X bits of the lane's own column 0 (for column_fields)
    if (LANE_SETS && (SCHEME == 0 || SCHEME == 5 || SCHEME == 8 || SCHEME == 10)) E0 = gather_lsb(X);

    // Block layer: 16 single-hit collective steps.
    const uint4 setw = c.draw(c.k, kTagSet << 28);
    uint4 site = make_uint4(0u, 0u, 0u, 0u);
    uint4 borg = make_uint4(0u, 0u, 0u, 0u);
    if (SCHEME == 3) borg = c.draw(c.k, kTagBorg << 28);
    for (uint32_t s = 0; s < 16u; ++s) {
        if (SCHEME == 3) {
            // DTrDTr: the set, plus a block-layer origin (ax, ay) per step
            if ((s & 1u) == 0u)
                site = c.draw(c.k | ((s >> 1) << 2), (kTagSite << 28) | c.g);
            const uint32_t d = (setw.x >> (2u * s)) & 3u;
            const uint32_t bw = (s < 4u) ? borg.x : (s < 8u) ? borg.y : (s < 12u) ? borg.z : borg.w;
            const uint32_t byte = (bw >> (8u * (s & 3u))) & 0xFFu;
            const uint32_t c0 = ((byte & 3u) + 2u * (d & 1u)) & 3u;
            const uint32_t r0 = (((byte >> 4) & 3u) + 2u * (d >> 1)) & 3u;
            const DtrLanes n = dtr_lanes(c);
            uint32_t ca[4], cb[4], pmin, pmax;
            dtr_candidates<RANDOM, LANE_SETS>(X, Y, E, D, site, s, c0, r0, c, n, ca, cb, pmin, pmax);
            uint32_t acc = 0u;
            if (RANDOM) {
                draws += __popc(pmin | pmax);
                acc = accept_candidates<SCHEME == 3 ? kPreDtr : (LANE_SETS ? kPrePacked : kPreDt)>(pmin, pmax, level_words(s, c), c, tp);
                net += random_net(acc, pmin, pmax);
            }
            dtr_apply<RANDOM, LANE_SETS>(X, Y, E, D, c0, r0, acc, ca, cb, c, n, net);
            continue;
        }
        if (SCHEME == 1 || SCHEME == 2 || SCHEME == 6 || SCHEME == 7 || SCHEME == 9) {
            // DB: one site word per TC row and step, 4 bits per cell
            site = c.draw(c.k | (s << 2), (kTagSiteDb << 28) | c.g);
            if (SCHEME == 2)
                db_step_delayed<RANDOM>(X, Y, E, D, site, s, c, tp, net, draws);
            else if (SCHEME == 7)
                db_step_delayed<RANDOM, 2, kTiesCount>(X, Y, E, D, site, s, c, tp, net, draws);
            else if (SCHEME == 9)
                db_step_delayed<RANDOM, 2, kTiesRefused>(X, Y, E, D, site, s, c, tp, net, draws);
            else if (SCHEME == 6)
                db_step<RANDOM, 1>(X, Y, E, D, site, s, c, tp, net, draws);
            else
                db_step<RANDOM>(X, Y, E, D, site, s, c, tp, net, draws);
            continue;
        }
        if ((s & 1u) == 0u)
            site = c.draw(c.k | ((s >> 1) << 2), (kTagSite << 28) | c.g);
        else
            site = make_uint4(site.x >> 2, site.y >> 2, site.z >> 2, site.w >> 2);
        // the set (every lane of a one-sub-tile warp drew the same one; the broadcast
        // from lane 0 lets the compiler treat the branches on it as warp-uniform)
        const uint32_t d_own = (setw.x >> (2u * s)) & 3u;
        const uint32_t d = LANE_SETS ? d_own : __shfl_sync(kFull, d_own, 0);
        uint32_t cnd0[4], cnd1[4], pmin, pmax;
        constexpr int kSpec = SCHEME == 4 ? 1 : (SCHEME == 5 || SCHEME == 8 || SCHEME == 10) ? 2 : 0;
        constexpr int kTies = (SCHEME == 0 || SCHEME == 5) ? kTiesCount : SCHEME == 8 ? kTiesRefused : kTiesAsk;
        if (LANE_SETS)
            step_candidates_rt<RANDOM, kSpec>(X, Y, E, D, site, d & 1u, d >> 1, c, cnd0, cnd1, pmin, pmax);
        // the candidate phase with the set's column offset as a constant as well
        // (the flip phase stays specialised on the row offset alone: four copies
        // of it measured slower, from instruction-cache pressure)
        else if (d == 3u)
            step_candidates<1, RANDOM, kSpec>(X, Y, E, D, site, 1u, c, cnd0, cnd1, pmin, pmax);
        else if (d == 2u)
            step_candidates<1, RANDOM, kSpec>(X, Y, E, D, site, 0u, c, cnd0, cnd1, pmin, pmax);
        else if (d == 1u)
            step_candidates<0, RANDOM, kSpec>(X, Y, E, D, site, 1u, c, cnd0, cnd1, pmin, pmax);
        else
            step_candidates<0, RANDOM, kSpec>(X, Y, E, D, site, 0u, c, cnd0, cnd1, pmin, pmax);
        uint32_t acc = 0u;
        if (RANDOM) {
            draws += __popc(pmin | pmax);
            acc = accept_candidates<LANE_SETS ? kPrePacked : kPreDt, kTies>(pmin, pmax, level_words(s, c), c, tp);
            net += random_net(acc, pmin, pmax);
        }
        if (LANE_SETS)
            step_apply_rt<RANDOM, kSpec>(X, Y, E, D, d >> 1, acc, cnd0, cnd1, c, flips, E0, net);
        else if (d & 2u)
            step_apply<1, RANDOM, kSpec>(X, Y, E, D, d & 1u, acc, cnd0, cnd1, c, flips, net);
        else
            step_apply<0, RANDOM, kSpec>(X, Y, E, D, d & 1u, acc, cnd0, cnd1, c, flips, net);
    }

    launch_dependents();  // the next step's head overlaps this one's write-back
    write_back<LANE_SETS>(q, L, wpr, straight, active, c, X, Y, E, D);
    tails = static_cast<int>(tp.rounds);
}

}  // namespace oct
