// One device step of DTrDT with 4 x 4-site thread cells on a quarter of the
// registers and a quarter of the chain: a lane holds one TC row of a band (32
// x 4 sites: 4 X-row and 4 Y-row words) where subtile.cuh gives it a group of
// four TC rows.  Same sites, uniforms and tie order (reading of the streams in
// dtrdt.cu), so the same lattice bit for bit.
//
// Why: a device step of a small lattice has fewer warps than the chip has
// schedulers (L=4096 with 64 x 64 sub-tiles: 256 warps of four sub-tiles on 608),
// so it lasts as long as one warp's chain of instructions, 9-11 thousand for 512
// sites per lane.  With a TC row per lane a 64 x 64 sub-tile fills a warp of its
// own: four times the warps, each with a quarter of the rows, and the set draw
// is warp-uniform.  The four lanes of a group share its Philox blocks instead
// of repeating them: lane m generates every fourth block of the device step and
// leaves it (of the acceptance draws, their comparison with P32) in shared
// memory, before the step's first access to the lattice.  8 MCS and a W^2, us on
// packed groups and here: L=256 KPZ 266, 132; L=3136 p=0.95 (32 x 16 sub-tiles)
// 492, 290; L=4096 p=0.95 554, 346, p=q=0.5 387, 257.
//
// Lanes of a sub-tile: gx + GX * tr, TC row tr = 0 .. By/4 - 1 (group row tr/4,
// m = tr % 4), a power-of-two number of band columns GX, at most 32 lanes.
#pragma once
#include <cstdint>

#include "oct_internal.h"
#include "subtile.cuh"

namespace oct {

constexpr uint32_t kRowGroups = 8;  // groups of a warp: four lanes each
constexpr uint32_t kRowRing = 64;   // tail words kept per group
// 32-bit words of shared memory per warp: site blocks of 8 step pairs, and with
// draws the comparisons of 16 steps and the tail rings
template <bool RANDOM>
__host__ __device__ constexpr uint32_t row_smem_words() {
    return kRowGroups * (8u * 4u + (RANDOM ? 16u * 4u + kRowRing : 0u));
}

struct RowLane {
    uint32_t m, gw;        // TC row in its group; the group's place among the warp's
    int gx, tr, GX, TR;    // band column, TC row, and their numbers in the sub-tile
    bool active;
};

// Lanes of a sub-tile, rounded up to a power of two.
__host__ __device__ inline uint32_t row_segment(uint32_t GX, uint32_t By) {
    uint32_t s = 1u;
    while (s < GX * (By / 4u)) s <<= 1;
    return s;
}

// Device steps of more warps than this keep the chip busy either way, and then
// the lane of four TC rows needs fewer instructions per attempt (64 x 64
// sub-tiles, us per MCS here and there):
//   L                   4096        6144        7168        8192        8704         9216         16384
//   KPZ                 23.8, 34.7  38.1, 37.0  55.2, 51.8  54.2, 57.7  61.4, 62.7   69.8, 67.4   178, 131
//   p=q=0.5             28.9, 44.8  47.2, 47.0  64.8, 67.4  68.7, 73.9  75.4, 77.9   82.1, 90.7   224, 184
//   p=0.95, q=0.05      40.1, 65.7  59.8, 68.4  80.9, 89.2  86.6, 98.4  103, 109     113, 111     293, 227
constexpr uint32_t kRowWarpsMax = 152u * 32u;

// ONE: one sub-tile per warp (the set is warp-uniform); otherwise the rows of
// the set are picked per lane with selects.  `ready` waits for the device step
// before this one; everything ahead of it does not read the lattice.  `done` is
// called before the write-back.
// SHARED: lat lies in shared memory.
template <bool RANDOM, int SPEC, bool ONE, bool SHARED, class Ctx, class Ready, class Done>
__device__ __forceinline__ void run_rows(uint32_t *lat, uint32_t L, uint32_t plane_rows, uint32_t wpr, uint32_t x0,
                                         uint32_t y0, const Ctx &c, const RowLane &rl, uint32_t *sm, int &net,
                                         int &draws, int &tails, Ready ready, Done done) {
    uint4 *const site_w = reinterpret_cast<uint4 *>(sm);
    uint4 *const lvl_w = site_w + 8u * kRowGroups;
    uint32_t *const ring = sm + kRowGroups * 96u + rl.gw * kRowRing;
    const uint32_t m = rl.m, gw = rl.gw;
    // the draws of the whole device step, over those of the step before (in the one
    // launch of a whole run), which every lane has read
    if (SHARED) __syncwarp();
    const uint4 setw = c.draw(c.k, kTagSet << 28);
#pragma unroll
    for (uint32_t i = 0; i < 2u; ++i) {
        const uint32_t b = 4u * i + m;
        site_w[b * kRowGroups + gw] = c.draw(c.k | (b << 2), (kTagSite << 28) | c.g);
    }
    uint32_t head = 0u, end = 0u;  // words of the group's tail stream used, generated
    // see ties_matter: with SPEC 3 none does, with SPEC -1 (general) the replica's rates say
    const bool ties_count = SPEC == 0 || SPEC == 2 || (SPEC == -1 && __any_sync(kFull, ties_matter(c.thr_p, c.thr_q)));
    if (RANDOM) {
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            const uint32_t s = 4u * i + m;
            const uint4 B = c.draw(c.k | ((s * 8u) << 2), (kTagAcc << 28) | c.g);
            // the four leading bits of every cell's uniform (bit 4j+m of the four
            // words) against P32's: below, and equal, for p and for q
            const uint32_t lw[4] = {B.x, B.y, B.z, B.w};
            uint4 v = make_uint4(0u, kFull, 0u, kFull);
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                const uint32_t tp = (c.thr_p >> (31 - l)) & 1u ? kFull : 0u, tq = (c.thr_q >> (31 - l)) & 1u ? kFull : 0u;
                v.x |= v.y & tp & ~lw[l];
                v.y &= ~(tp ^ lw[l]);
                v.z |= v.w & tq & ~lw[l];
                v.w &= ~(tq ^ lw[l]);
            }
            lvl_w[s * kRowGroups + gw] = v;
        }
        if (ties_count) {
            *reinterpret_cast<uint4 *>(ring + 4u * m) = c.draw(c.k | (m << 2), (kTagTail << 28) | c.g);
            end = 16u;
            ++tails;
        }
    }
    __syncwarp();
    ready();

    // stage rows 0..3 and row 4 of Y (D: row 0 of the lane below, or the halo
    // row), and the bits of the edge words that are not the sub-tile's, which
    // nobody changes during the step.  Loads bypass the L1 cache: another SM may
    // have written the words in the step before, in the same launch or one whose
    // tail overlaps this one's head.
    const uint32_t sh = x0 & 31u;
    const uint32_t wA = ((x0 >> 5) + static_cast<uint32_t>(rl.gx)) % wpr, wB = (wA + 1u == wpr) ? 0u : wA + 1u;
    const bool left_edge = rl.active && rl.gx == 0 && sh != 0u, right_edge = rl.active && rl.gx == rl.GX - 1;
    const bool last_row = rl.active && rl.tr == rl.TR - 1;
    const uint32_t lo_mask = (1u << sh) - 1u, xb_mask = (2u << sh) - 1u;
    uint32_t *const Xp = lat;
    uint32_t *const Yp = lat + static_cast<size_t>(plane_rows) * wpr;
    auto load = [](const uint32_t *p) { return SHARED ? *p : __ldcg(p); };
    uint32_t X[4], Y[4], oX[4], oY[4], E = 0u, D = 0u, oD = 0u;
    size_t ro[5];
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        uint32_t yr = y0 + 4u * static_cast<uint32_t>(rl.tr) + static_cast<uint32_t>(r);
        if (yr >= L) yr -= L;
        ro[r] = static_cast<size_t>(yr) * wpr;
    }
    if (rl.active) {
        uint32_t xa[4], xb[4], ya[5], yb[5];
#pragma unroll
        for (int r = 0; r < 5; ++r) {
            if (r < 4) {
                xa[r] = load(Xp + ro[r] + wA);
                xb[r] = load(Xp + ro[r] + wB);
            }
            ya[r] = load(Yp + ro[r] + wA);
            yb[r] = load(Yp + ro[r] + wB);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            X[r] = __funnelshift_r(xa[r], xb[r], sh);
            Y[r] = __funnelshift_r(ya[r], yb[r], sh);
            E |= ((xb[r] >> sh) & 1u) << r;
            oX[r] = (left_edge ? xa[r] & lo_mask : 0u) | (right_edge ? xb[r] & ~xb_mask : 0u);
            oY[r] = (left_edge ? ya[r] & lo_mask : 0u) | (right_edge ? yb[r] & ~lo_mask : 0u);
        }
        D = __funnelshift_r(ya[4], yb[4], sh);
        oD = (left_edge ? ya[4] & lo_mask : 0u) | (right_edge ? yb[4] & ~lo_mask : 0u);
    } else {
#pragma unroll
        for (int r = 0; r < 4; ++r) X[r] = Y[r] = oX[r] = oY[r] = 0u;
    }

    const uint32_t low_p = c.thr_p << 4, low_q = c.thr_q << 4;
    const bool has_l = rl.gx > 0, has_r = rl.gx < rl.GX - 1, has_a = rl.tr > 0, has_b = rl.tr < rl.TR - 1;
    const uint32_t *const sw = reinterpret_cast<const uint32_t *>(site_w + gw) + m;
    const uint4 *const lvl = lvl_w + gw;

    // one collective step, rows of the set at ro2 = 0 or 2 (dy a constant when ONE)
    auto step = [&](uint32_t u, const uint4 &V, uint32_t dx, bool dy) {
        const uint32_t sh2 = 2u * dx, r0 = dy ? 2u : 0u;
        const uint32_t col = ((u & kNib) + kNib) << sh2;  // see step_candidates
        const uint32_t yoff = ((u >> 1) & kNib) * 0xFu;
        const uint32_t xa = dy ? X[2] : X[0], xb = dy ? X[3] : X[1];
        const uint32_t ya = dy ? Y[2] : Y[0], yb = dy ? Y[3] : Y[1], yc = dy ? D : Y[2];
        const uint32_t xra = __funnelshift_r(xa, E >> r0, 1), xrb = __funnelshift_r(xb, E >> (r0 + 1u), 1);
        uint32_t f0, f1;
        if (SPEC == 1) {
            f0 = col & ~yoff & ~xa & xra & ~ya & yb;
            f1 = col & yoff & ~xb & xrb & ~yb & yc;
            net += __popc(f0 | f1);
        } else {
            f0 = col & ~yoff & (xa ^ xra) & (ya ^ yb) & ~(xa ^ ya);
            f1 = col & yoff & (xb ^ xrb) & (yb ^ yc) & ~(xb ^ yb);
            uint32_t acc = 0u;
            if (RANDOM) {
                const uint32_t cc = f0 | f1, mx = (f0 & xa) | (f1 & xb);
                const uint32_t cmx = SPEC >= 2 ? mx : mx & c.q_random, cmn = SPEC >= 2 ? cc : (cc & ~mx) & c.p_random;
                const uint32_t pmax = ((cmx * 3u) >> (sh2 + 1u)) & kNib;
                uint32_t pmin = ((cmn * 3u) >> (sh2 + 1u)) & kNib;
                if (SPEC >= 2) pmin &= ~pmax;
                draws += __popc(pmin | pmax);
                const uint32_t mn = pmin << m, mx4 = pmax << m;  // bit 4j+m
                acc = (mn & V.x) | (mx4 & V.z);
                if (ties_count) {
                    uint32_t und = (mn & V.y) | (mx4 & V.w);
                    // ties of the whole group, so that a tie's place in the tail stream is the
                    // number of lower ones
                    uint32_t gt = und;
                    gt |= __shfl_xor_sync(kFull, gt, rl.GX);
                    gt |= __shfl_xor_sync(kFull, gt, 2 * rl.GX);
                    const uint32_t nt = static_cast<uint32_t>(__popc(gt));
                    while (__any_sync(kFull, end - head < nt)) {
                        __syncwarp();  // the words about to be overwritten have been read
                        const uint4 B = c.draw(c.k | (((end >> 2) + m) << 2), (kTagTail << 28) | c.g);
                        if (end - head <= kRowRing - 16u) {
                            *reinterpret_cast<uint4 *>(ring + ((end + 4u * m) & (kRowRing - 1u))) = B;
                            end += 16u;
                            ++tails;
                        }
                        __syncwarp();
                    }
                    while (und) {
                        const uint32_t bit = und & (0u - und);
                        und ^= bit;
                        const uint32_t at = head + static_cast<uint32_t>(__popc(gt & (bit - 1u)));
                        acc |= (ring[at & (kRowRing - 1u)] < ((mn & bit) ? low_p : low_q)) ? bit : 0u;
                    }
                    head += nt;
                }
                acc = (acc >> m) & kNib;
                net += random_net(acc, pmin, pmax);
            }
            if (SPEC >= 2) {
                const uint32_t spread = acc * 0xFu;
                f0 &= spread;
                f1 &= spread;
            } else {
                uint32_t amin = c.p_always, amax = c.q_always;
                if (RANDOM) {
                    const uint32_t spread = acc * 0xFu;
                    amin |= spread & c.p_random;
                    amax |= spread & c.q_random;
                }
                f0 &= (~xa & amin) | (xa & amax);
                f1 &= (~xb & amin) | (xb & amax);
                net += always_net<RANDOM>(f0, xa, c) + always_net<RANDOM>(f1, xb, c);
            }
        }
        // flips (3f: see step_apply) and the neighbours' copies.  Flips at column 31
        // occur for dx = 1 only and change the right lane's column 0, those at
        // column 0 for dx = 0 only, mirrored in the left lane's E.
        uint32_t g0 = f0 * 3u, g1 = f1 * 3u;
        const uint32_t e = (f0 >> 31) | ((f1 >> 31) << 1);
        E ^= e << r0;
        if (rl.GX > 1) {  // warp-uniform
            if (!ONE || dx) {
                const uint32_t v = __shfl_up_sync(kFull, e, 1);
                if (has_l) {
                    g0 ^= v & 1u;
                    g1 ^= v >> 1;
                }
            }
            if (!ONE || !dx) {
                const uint32_t v = __shfl_down_sync(kFull, (f0 & 1u) | ((f1 & 1u) << 1), 1);
                if (has_r) E ^= v << r0;
            }
        }
        const uint32_t f01 = f0 ^ f1;
        if (ONE) {
            if (dy) {
                X[2] ^= g0;
                X[3] ^= g1;
                Y[2] ^= f0;
                Y[3] ^= f01;
                D ^= f1;
                const uint32_t v = __shfl_up_sync(kFull, f1, rl.GX);
                if (has_a) Y[0] ^= v;
            } else {
                X[0] ^= g0;
                X[1] ^= g1;
                Y[0] ^= f0;
                Y[1] ^= f01;
                Y[2] ^= f1;
                const uint32_t v = __shfl_down_sync(kFull, f0, rl.GX);
                if (has_b) D ^= v;
            }
        } else {
            const uint32_t dym = dy ? 0xFFFFFFFFu : 0u;
            X[0] ^= g0 & ~dym;
            X[1] ^= g1 & ~dym;
            X[2] ^= g0 & dym;
            X[3] ^= g1 & dym;
            Y[0] ^= f0 & ~dym;
            Y[1] ^= f01 & ~dym;
            Y[2] ^= dy ? f0 : f1;
            Y[3] ^= f01 & dym;
            D ^= f1 & dym;
            const uint32_t vd = __shfl_up_sync(kFull, f1 & dym, rl.GX);
            const uint32_t vu = __shfl_down_sync(kFull, f0 & ~dym, rl.GX);
            if (has_a) Y[0] ^= vd;
            if (has_b) D ^= vu;
        }
    };
    auto site_of = [&](uint32_t s) { return sw[(s >> 1) * (kRowGroups * 4u)] >> (2u * (s & 1u)); };
    auto level_of = [&](uint32_t s) { return RANDOM ? lvl[s * kRowGroups] : make_uint4(0u, 0u, 0u, 0u); };
    if (ONE) {
        // the sets from lane 0: warp-uniform to the compiler too.  The next step's
        // draws are read before this step's chain (L=256 KPZ, 8 MCS and a W^2: 145
        // to 136 us).
        const uint32_t sets = __shfl_sync(kFull, setw.x, 0);
        uint32_t u = site_of(0u);
        uint4 V = level_of(0u);
        for (uint32_t s = 0; s < 16u; ++s) {
            const uint32_t us = u, nx = (s + 1u) & 15u, d = (sets >> (2u * s)) & 3u;
            const uint4 Vs = V;
            u = site_of(nx);
            V = level_of(nx);
            if (d & 2u)
                step(us, Vs, d & 1u, true);
            else
                step(us, Vs, d & 1u, false);
        }
    } else {
        for (uint32_t s = 0; s < 16u; ++s) {
            const uint32_t d = (setw.x >> (2u * s)) & 3u;
            step(site_of(s), level_of(s), d & 1u, (d & 2u) != 0u);
        }
    }

    done();
    // write back (see store_lane_rows): the edge words' outside bits are those staged
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        const uint32_t y = r < 4 ? Y[r & 3] : D, oy = r < 4 ? oY[r & 3] : oD;
        const uint32_t leftY = __shfl_up_sync(kFull, y, 1);
        if (r < 4) {
            const uint32_t leftX = __shfl_up_sync(kFull, X[r & 3], 1);
            if (rl.active) {
                Xp[ro[r] + wA] = left_edge ? (oX[r & 3] & lo_mask) | (X[r & 3] << sh) : __funnelshift_l(leftX, X[r & 3], sh);
                if (right_edge)
                    Xp[ro[r] + wB] = (oX[r & 3] & ~xb_mask) | (sh ? (X[r & 3] >> (32u - sh)) : 0u) | (((E >> r) & 1u) << sh);
            }
        }
        if (r < 4 ? rl.active : last_row) {
            Yp[ro[r] + wA] = left_edge ? (oy & lo_mask) | (y << sh) : __funnelshift_l(leftY, y, sh);
            if (right_edge && sh) Yp[ro[r] + wB] = (oy & ~lo_mask) | (y >> (32u - sh));
        }
    }
}

}  // namespace oct
