// Block layer of DTrDT with coarse thread cells, one lane per cell: cx x cy
// sites, cx in {8, 16, 32}, cy in {4, 8, 16}.
//
// A collective step makes one attempt per cell, so a lane that holds 32 x 16
// sites bit-parallel (cells.cuh) reads all eight rows that an attempt can fall
// on for the sake of its 512 / (cx cy) attempts: two for 16 x 16 cells.  Here
// the sub-tile lies in shared memory and a lane makes one attempt at a time,
// three loads and up to three stores of it, whatever the cell.  Bound by fixed
// latency and shared-memory round trips, issue slots 53 % (16 x 16 cells in 64 x
// 64 sub-tiles, p=0.95, q=0.05: one MCS at L=8192 from 2.31 to 0.56 ms at 171
// instructions per 32 attempts, then to 0.48 ms with the draws' places constant
// in loops over the steps of a level block).  A warp takes the cells of a
// sub-tile in turns of 32 (NC of them), or several sub-tiles of fewer than 32
// cells at once.
//
// Cells and random streams are those of cells.cuh (same sites, uniforms and tie
// order).  A group of four TC rows x 32 columns has 128/cx cells, which are
// consecutive lanes in order of position 4j+m, so the rank of a tied candidate
// among its group's ties is a population count.
//
// Shared-memory layout.  The unit is a half row of a cell, the cx/2 sites of
// one of its row halves: X bits below, Y bits above, in 1, 2 or 4 bytes.  The
// units of a cell fill words of its lane's own bank (word (ly / RPW) * 2 +
// half of lane l at 4 l + 128 times that, RPW rows to a word), so loads at
// random rows do not conflict.  In one step the units that two attempts write
// are distinct, and nobody else writes what an attempt reads: with dx = 1 a
// flip reaches the first column of the next cell, in its half 0, while that
// cell's own attempt stays in half 1; with dy = 1 the first row of the cell
// below, while that cell's stays in its lower rows.  So a step needs no
// ordering inside, and one warp barrier after it.
//
// The site words and the acceptance prefixes of several steps are generated at
// once, a block per lane; the four level words of a block are transposed so
// that a cell finds the four leading bits of its uniform in one nibble.
#pragma once
#include <cstdint>

#include "cells.cuh"

namespace oct {

template <int CX, int CY>
struct LaneCells {
    using S = CellShape<CX, CY>;
    static constexpr int UX = S::UX, UY = S::UY;
    static constexpr int GSZ = 128 / CX;            // cells of a group
    static constexpr int GPI = 32 / GSZ;            // groups per turn of 32 cells
    static constexpr int NCMAX = 512 / (CX * CY);   // turns of the largest sub-tile (16384 sites)
    static constexpr int RPW = 16 / UX;             // rows of a half in one word
    static constexpr int HB = 4 / RPW;              // bytes of a half row
    static constexpr int WR = CY / RPW;             // word rows of a cell
    static constexpr int TURN = (WR + 1) * 256;     // bytes of a turn: its cells and a halo row below
    static constexpr int P = CX == 8 ? 4 : 16;      // steps whose draws are generated at once
    static constexpr int RING = 32;                 // tail words kept per group
    static_assert(P % S::SPW == 0 && P % S::SPL == 0 && S::STEPS % P == 0, "whole blocks of draws");
    // byte offset of row ly of a half: word row ly / RPW (256 bytes), place ly % RPW in the word
    static constexpr uint32_t KMUL = 256u / RPW + (RPW > 1 ? static_cast<uint32_t>(HB) : 0u);
    static constexpr uint32_t KMASK = 0xFF00u | static_cast<uint32_t>((RPW - 1) * HB);
};

// How a launch's sub-tiles lie in warps (host and device).
struct LaneSplit {
    uint32_t nr;        // TC rows of a sub-tile
    uint32_t ng;        // groups of a sub-tile
    uint32_t ngp;       // lanes' groups per sub-tile when several share a warp
    uint32_t pk;        // sub-tiles per warp
    uint32_t nc;        // turns
    uint32_t ngw;       // groups per warp
    uint32_t hx, site, lvl, ring, tab, bytes;  // shared-memory offsets of a warp's areas, and their total
};

template <int CX, int CY, bool RANDOM>
__host__ __device__ inline LaneSplit lane_split(uint32_t GX, uint32_t By) {
    using C = LaneCells<CX, CY>;
    using S = CellShape<CX, CY>;
    LaneSplit q;
    q.nr = By / CY;
    q.ng = GX * ((q.nr + 3u) / 4u);
    q.ngp = 1u;
    while (q.ngp < q.ng && q.ngp < static_cast<uint32_t>(C::GPI)) q.ngp <<= 1;
    q.pk = C::GPI / q.ngp;
    q.nc = (q.ng + C::GPI - 1u) / C::GPI;
    q.ngw = q.nc * C::GPI;
    q.hx = q.nc * C::TURN;
    q.site = q.hx + ((q.nc + 1u) / 2u) * C::WR * 256u;
    q.lvl = q.site + (C::P / S::SPW) * q.ngw * 16u;
    q.ring = q.lvl + (RANDOM ? (C::P / S::SPL) * q.ngw * 16u : 0u);
    q.tab = q.ring + (RANDOM ? q.ngw * C::RING * 4u : 0u);
    q.bytes = q.tab + q.ngw * 8u;
    return q;
}

// Loads and stores of one half row (HB bytes) in shared memory.
template <int HB>
__device__ __forceinline__ uint32_t half_load(const unsigned char *p) {
    if (HB == 1) return *p;
    if (HB == 2) return *reinterpret_cast<const uint16_t *>(p);
    return *reinterpret_cast<const uint32_t *>(p);
}
template <int HB>
__device__ __forceinline__ void half_store(unsigned char *p, uint32_t v) {
    if (HB == 1) *p = static_cast<unsigned char>(v);
    else if (HB == 2) *reinterpret_cast<uint16_t *>(p) = static_cast<uint16_t>(v);
    else *reinterpret_cast<uint32_t *>(p) = v;
}

// Between the planar lattice and a sub-tile's half rows.  A lane takes the 32
// sites of one row and band at a time, 32 / GX whole rows per pass.  first: the
// lane group (of its group 0) that the sub-tile's cells start at.  STORE false:
// lattice to shared memory, with the halo column and row; true: back.
template <int CX, int CY, bool STORE>
__device__ __forceinline__ void move_subtile(uint32_t *lat, uint32_t L, uint32_t plane_rows, uint32_t wpr,
                                             uint32_t GX, uint32_t By, uint32_t x0, uint32_t y0, uint32_t nr,
                                             uint32_t first, unsigned char *sm, uint32_t hx, bool valid) {
    using C = LaneCells<CX, CY>;
    using S = CellShape<CX, CY>;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t per = 32u / GX, r = lane / GX, col = lane % GX;
    uint32_t *const Xp = lat;
    uint32_t *const Yp = lat + static_cast<size_t>(plane_rows) * wpr;
    const uint32_t sh = x0 & 31u;
    const uint32_t wA = ((x0 >> 5) + col) % wpr, wB = (wA + 1u == wpr) ? 0u : wA + 1u;
    constexpr uint32_t kHalf = (C::UX == 32) ? 0xFFFFFFFFu : ((1u << C::UX) - 1u);
    for (uint32_t yy = 0; yy <= By; yy += per) {
        const uint32_t y = yy + r;
        const bool on = valid && r < per && y <= By;
        const bool halo = y == By;
        const uint32_t yc = halo ? nr - 1u : y / CY, ly = halo ? static_cast<uint32_t>(CY) : y % CY;
        uint32_t yr = y0 + y;
        if (yr >= L) yr -= L;
        const size_t ro = static_cast<size_t>(yr) * wpr;
        const uint32_t G = first + (yc >> 2) * GX + col;  // lane group of the row's cells in this band
        const uint32_t turn = G / C::GPI, l0 = (G % C::GPI) * C::GSZ + (yc & 3u);
        const uint32_t off = (ly * C::KMUL) & C::KMASK;
        unsigned char *const cell = sm + turn * C::TURN + l0 * 4u + off;
        unsigned char *const edge = sm + hx + (turn >> 1) * (C::WR * 256u) + (turn & 1u) * 128u +
                                    (l0 + 4u * (S::TPB - 1)) * 4u + off;
        if (!STORE) {
            if (!on) continue;
            const uint32_t xB = Xp[ro + wB];
            const uint32_t x = __funnelshift_r(Xp[ro + wA], xB, sh);
            const uint32_t yv = __funnelshift_r(Yp[ro + wA], Yp[ro + wB], sh);
#pragma unroll
            for (int j = 0; j < S::TPB; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int s = CX * j + C::UX * h;
                    half_store<C::HB>(cell + 16 * j + 128 * h,
                                      ((x >> s) & kHalf) | (((yv >> s) & kHalf) << C::UX));
                }
            if (col == GX - 1u && !halo) half_store<C::HB>(edge, (xB >> sh) & 1u);
            continue;
        }
        uint32_t x = 0u, yv = 0u, ex = 0u;
        if (on) {
#pragma unroll
            for (int j = 0; j < S::TPB; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int s = CX * j + C::UX * h;
                    const uint32_t u = half_load<C::HB>(cell + 16 * j + 128 * h);
                    x |= (u & kHalf) << s;
                    yv |= ((u >> C::UX) & kHalf) << s;
                }
            if (col == GX - 1u && !halo) ex = half_load<C::HB>(edge) & 1u;
        }
        // as in write_back: full words are stored, the two edge words of a row
        // shared with neighbouring sub-tiles are merged by reductions
        const uint32_t leftX = __shfl_up_sync(kFull, x, 1), leftY = __shfl_up_sync(kFull, yv, 1);
        if (!on) continue;
        const uint32_t lo_mask = (1u << sh) - 1u, xb_mask = (2u << sh) - 1u;
        if (col == 0u && sh != 0u) {
            if (!halo) reduce_bits(&Xp[ro + wA], x << sh, ~lo_mask);
            reduce_bits(&Yp[ro + wA], yv << sh, ~lo_mask);
        } else {
            if (!halo) Xp[ro + wA] = __funnelshift_l(leftX, x, sh);
            Yp[ro + wA] = __funnelshift_l(leftY, yv, sh);
        }
        if (col == GX - 1u) {
            if (!halo) reduce_bits(&Xp[ro + wB], (sh ? (x >> (32u - sh)) : 0u) | (ex << sh), xb_mask);
            if (sh) reduce_bits(&Yp[ro + wB], yv >> (32u - sh), lo_mask);
        }
    }
}

template <int CX, int CY, bool RANDOM, int SPEC>
__global__ void __launch_bounds__(kStepWarpsPerBlock * 32) lane_cells_kernel(const StepArgs a, const LaneSplit q) {
    using C = LaneCells<CX, CY>;
    using S = CellShape<CX, CY>;
    extern __shared__ __align__(256) unsigned char lane_cells_smem[];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = blockIdx.x * kStepWarpsPerBlock + (threadIdx.x >> 5);
    const uint32_t n_tiles = work_tiles(a);
    if (warp * q.pk >= n_tiles) return;  // the whole warp leaves together
    unsigned char *const sm = lane_cells_smem + (threadIdx.x >> 5) * q.bytes;
    uint4 *const site_w = reinterpret_cast<uint4 *>(sm + q.site);
    uint4 *const lvl_w = reinterpret_cast<uint4 *>(sm + q.lvl);
    uint32_t *const ring = reinterpret_cast<uint32_t *>(sm + q.ring);
    uint2 *const tab = reinterpret_cast<uint2 *>(sm + q.tab);  // (T, group) of every lane group

    // the lane's sub-tile, and its cell in every turn
    const uint32_t gl = lane / C::GSZ, i = lane % C::GSZ, j = i >> 2, m = i & 3u;
    const uint32_t seg = q.pk > 1u ? gl / q.ngp : 0u;
    const uint32_t w = warp * q.pk + seg;
    const uint32_t t = *a.t_ptr + a.dt;
    const TilePlace pl = place_tile(a, w < n_tiles ? w : 0u, t, a.k);
    const uint32_t T = pl.T;
    uint32_t rb[C::NCMAX], db[C::NCMAX];  // half 0 of the next cell's row 0; row 0 of the cell below
    uint32_t on = 0u;                     // turns in which the lane holds a cell
    uint32_t hd[C::NCMAX], gen[C::NCMAX];  // tail words of the lane's group: used, generated
#pragma unroll
    for (int c = 0; c < C::NCMAX; ++c) {
        rb[c] = db[c] = hd[c] = gen[c] = 0u;
        if (c >= static_cast<int>(q.nc)) continue;
        const uint32_t base = q.pk > 1u ? seg * q.ngp : 0u;  // the sub-tile's first lane group
        const uint32_t gw = static_cast<uint32_t>(c) * C::GPI + gl, G = gw - base;
        const uint32_t gcol = G % a.GX, row = 4u * (G / a.GX) + m;
        if (w < n_tiles && G < q.ng && row < q.nr) on |= 1u << c;
        auto at = [&](uint32_t g, uint32_t l) {  // word row 0 of the cell at lane l of lane group g
            return (g / C::GPI) * C::TURN + ((g % C::GPI) * C::GSZ + l) * 4u;
        };
        const uint32_t own = at(gw, i);
        rb[c] = db[c] = own;  // a lane without a cell stays in its own words
        if (!((on >> c) & 1u)) {
            if (i == 0u) tab[gw] = make_uint2(T, G);
            continue;
        }
        rb[c] = j + 1u < static_cast<uint32_t>(S::TPB) ? own + 16u
                : gcol + 1u < a.GX ? at(gw + 1u, m)
                : q.hx + (static_cast<uint32_t>(c) >> 1) * (C::WR * 256u) + (static_cast<uint32_t>(c) & 1u) * 128u + lane * 4u;
        db[c] = row + 1u >= q.nr ? own + C::WR * 256u : m < 3u ? own + 4u : at(gw + a.GX, i - 3u);
        if (i == 0u) tab[gw] = make_uint2(T, G);
    }
    for (uint32_t sg = 0; sg < q.pk; ++sg) {
        const int src = static_cast<int>(sg * q.ngp * C::GSZ);
        const uint32_t x0 = __shfl_sync(kFull, pl.x0, src), y0 = __shfl_sync(kFull, pl.y0, src);
        move_subtile<CX, CY, false>(a.lat, a.L, a.plane_rows, a.wpr, a.GX, a.By, x0, y0, q.nr, sg * q.ngp, sm, q.hx,
                                    warp * q.pk + sg < n_tiles);
    }
    __syncwarp();

    int net = 0;
    uint32_t draws = 0u, tails = 0u;
    const uint32_t tie_mask = ties_matter(a.thr_p, a.thr_q) ? kFull : 0u;
    const uint32_t tp4 = a.thr_p >> 28, tq4 = a.thr_q >> 28, low_p = a.thr_p << 4, low_q = a.thr_q << 4;
    constexpr uint32_t kM = 1u | (1u << C::UX);  // X(s) and Y(s) of a half row, at the site's place
    constexpr int U = C::NCMAX < 4 ? C::NCMAX : 4;  // turns in flight
    // One step: the site word's field at sub, the level word's nibbles at lev.
    auto step = [&](const uint32_t *sw, uint32_t sub, const uint32_t *lw, uint32_t lev, uint32_t dx, uint32_t dy) {
#pragma unroll
        for (int c0 = 0; c0 < C::NCMAX; c0 += U) {
            if (c0 >= static_cast<int>(q.nc)) break;
            uint32_t h0[U], h1[U], he[U], rx[U], p0[U], p1[U], pe[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + u;
                if (c >= static_cast<int>(q.nc)) break;
                const uint32_t f = (sw[c * C::GPI * 4] >> (CX * j) >> sub) & ((1u << S::BPT) - 1u);
                rx[u] = f & static_cast<uint32_t>(C::UX - 1);
                const uint32_t ly = dy * C::UY + (f >> S::BXB);
                const uint32_t own = static_cast<uint32_t>(c) * C::TURN + lane * 4u;
                const uint32_t o0 = (ly * C::KMUL) & C::KMASK, o1 = (ly * C::KMUL + C::KMUL) & C::KMASK;
                p0[u] = own + 128u * dx + o0;
                p1[u] = (ly + 1u == static_cast<uint32_t>(CY) ? db[c] : own + o1) + 128u * dx;
                pe[u] = (dx ? rb[c] : own + 128u) + o0;
                h0[u] = half_load<C::HB>(sm + p0[u]);
                h1[u] = half_load<C::HB>(sm + p1[u]);
                he[u] = half_load<C::HB>(sm + pe[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + u;
                if (c >= static_cast<int>(q.nc)) break;
                const bool last = rx[u] == static_cast<uint32_t>(C::UX - 1);
                const uint32_t tt = h0[u] >> rx[u];
                const uint32_t xr = last ? he[u] << 1 : tt;                  // bit 1: X(s+x)
                const uint32_t yd = (h1[u] >> rx[u]) << 1;                   // bit UX + 1: Y(s+y)
                const uint32_t pat = (tt & kM) | (xr & 2u) | (yd & (2u << C::UX));
                const bool held = (on >> c) & 1u;
                const bool mn = held && pat == 2u * kM, mx = held && pat == kM;  // Eq. (1)
                bool acc;
                if (SPEC == 1) {
                    acc = mn;
                } else if (!RANDOM) {
                    acc = (mn && a.p_always) || (mx && a.q_always);
                } else {
                    const bool drw = SPEC >= 2 ? mn || mx : (mn && a.p_random) || (mx && a.q_random);
                    const uint32_t u4 = (lw[c * C::GPI * 4] >> (4u * j) >> lev) & 15u, t4 = mn ? tp4 : tq4;
                    acc = drw && u4 < t4;
                    if (SPEC < 2) acc = acc || (mn && a.p_always) || (mx && a.q_always);
                    draws += drw ? 1u : 0u;
                    const bool tie = drw && u4 == t4;
                    const uint32_t ties = SPEC == 3 ? 0u : SPEC == 2 ? __ballot_sync(kFull, tie) : __ballot_sync(kFull, tie) & tie_mask;
                    if (ties) {
                        // the ties of the lane's group, in order of position, take the next
                        // words of its tail stream
                        const uint32_t gt = C::GSZ == 32 ? ties : (ties >> (gl * C::GSZ)) & ((1u << C::GSZ) - 1u);
                        const uint32_t nt = static_cast<uint32_t>(__popc(gt));
                        uint32_t head = hd[c], end = gen[c];
                        uint32_t *const rg = ring + (static_cast<uint32_t>(c) * C::GPI + gl) * C::RING;
                        while (__any_sync(kFull, head + nt > end)) {
                            // one block per lane of the group, as many as fit above the live words
                            const uint32_t room = min((C::RING - (end - head)) / 4u, static_cast<uint32_t>(C::GSZ));
                            if (i < room) {
                                const uint2 tg = tab[static_cast<uint32_t>(c) * C::GPI + gl];
                                const uint4 B = philox4x32_10(t, a.k | (((end >> 2) + i) << 2), tg.x,
                                                              (kTagTail << 28) | tg.y, a.k0, a.k1);
                                *reinterpret_cast<uint4 *>(rg + ((end + 4u * i) & (C::RING - 1u))) = B;
                                ++tails;
                            }
                            end += 4u * room;
                            __syncwarp();
                        }
                        if (tie) {
                            const uint32_t at = head + static_cast<uint32_t>(__popc(gt & ((1u << i) - 1u)));
                            // (word >> 4) < (P32 mod 2^28)
                            acc = rg[at & (C::RING - 1u)] < (mn ? low_p : low_q);
                        }
                        hd[c] = head + nt;
                        gen[c] = end;
                        __syncwarp();  // a later refill overwrites words read here
                    }
                }
                if (acc) {
                    half_store<C::HB>(sm + p0[u], h0[u] ^ ((last ? kM : kM | 2u) << rx[u]));
                    half_store<C::HB>(sm + p1[u], h1[u] ^ ((1u << C::UX) << rx[u]));
                    if (last) half_store<C::HB>(sm + pe[u], he[u] ^ 1u);
                    net += mn ? 1 : -1;
                }
            }
        }
        __syncwarp();
    };
    const uint32_t site_stride = 4u * q.ngw, lvl_stride = 4u * q.ngw;  // words between blocks of steps
    uint4 setw = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t s0 = 0; s0 < static_cast<uint32_t>(S::STEPS); s0 += C::P) {
        if ((s0 & 63u) == 0u) setw = philox4x32_10(t, a.k | ((s0 >> 6) << 2), T, kTagSet << 28, a.k0, a.k1);
        // the draws of the next P steps, one Philox block per lane at a time
        const uint32_t n_site = (C::P / S::SPW) * q.ngw, n_all = n_site + (RANDOM ? (C::P / S::SPL) * q.ngw : 0u);
        for (uint32_t v = lane; v < n_all; v += 32u) {
            const bool lv = v >= n_site;
            const uint32_t vv = lv ? v - n_site : v, blk = vv / q.ngw, gw = vv % q.ngw;
            const uint2 tg = tab[gw];
            const uint32_t index = lv ? (s0 / S::SPL + blk) * 8u : s0 / S::SPW + blk;
            const uint4 B = philox4x32_10(t, a.k | (index << 2), tg.x, ((lv ? kTagAcc : kTagSite) << 28) | tg.y, a.k0,
                                          a.k1);
            if (lv) {
                uint32_t pre[4];
                transpose_nibbles(make_uint4(B.w, B.z, B.y, B.x), pre);
                lvl_w[vv] = make_uint4(pre[0], pre[1], pre[2], pre[3]);
            } else {
                site_w[vv] = B;
            }
        }
        __syncwarp();
        uint32_t sets = word_of(setw, (s0 >> 4) & 3u) >> (2u * (s0 & 15u));
        if (q.pk == 1u) sets = __shfl_sync(kFull, sets, 0);
        const uint32_t *sw = reinterpret_cast<const uint32_t *>(site_w + gl) + m;
        const uint32_t *lw = reinterpret_cast<const uint32_t *>(lvl_w + gl) + m;
        for (int i0 = 0; i0 < C::P; i0 += S::SPL) {
#pragma unroll
            for (int e = 0; e < S::SPL; ++e) {  // the steps of one level block
                step(sw + (e / S::SPW) * site_stride, (e % S::SPW) * (CX / S::SPW), lw, 4u * (e * S::TPB), sets & 1u,
                     (sets >> 1) & 1u);
                sets >>= 2;
            }
            sw += (S::SPL / S::SPW) * site_stride;
            lw += lvl_stride;
        }
    }
    for (uint32_t sg = 0; sg < q.pk; ++sg) {
        const int src = static_cast<int>(sg * q.ngp * C::GSZ);
        const uint32_t x0 = __shfl_sync(kFull, pl.x0, src), y0 = __shfl_sync(kFull, pl.y0, src);
        move_subtile<CX, CY, true>(a.lat, a.L, a.plane_rows, a.wpr, a.GX, a.By, x0, y0, q.nr, sg * q.ngp, sm, q.hx,
                                   warp * q.pk + sg < n_tiles);
    }

    const int total = __reduce_add_sync(kFull, net);
    if (lane == 0 && total != 0)
        atomicAdd(&a.net[warp % kNetSlots], static_cast<unsigned long long>(static_cast<long long>(total)));
    if (RANDOM) {
        const unsigned nd = __reduce_add_sync(kFull, draws), nb = __reduce_add_sync(kFull, tails);
        if (lane == 0 && nd != 0u) atomicAdd(&a.draws[warp % kNetSlots], static_cast<unsigned long long>(nd));
        if (lane == 0 && nb != 0u) atomicAdd(&a.tails[warp % kNetSlots], static_cast<unsigned long long>(nb));
    }
}

template <int CX, int CY, bool RANDOM, int SPEC>
cudaError_t launch_lane_cells(const StepArgs &a, const LaneSplit &q, cudaStream_t st) {
    const uint32_t warps = (work_tiles(a) + q.pk - 1u) / q.pk, smem = kStepWarpsPerBlock * q.bytes;
    // The limit is that of the largest sub-tile for every launch: threads that
    // run different sub-tiles may pass here at the same time.
    using C = LaneCells<CX, CY>;
    const uint32_t most = kStepWarpsPerBlock * lane_split<CX, CY, RANDOM>(1u, C::NCMAX * C::GPI * 4u * CY).bytes;
    if (smem > most) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(lane_cells_kernel<CX, CY, RANDOM, SPEC>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
    if (e != cudaSuccess) return e;
    lane_cells_kernel<CX, CY, RANDOM, SPEC><<<(warps + kStepWarpsPerBlock - 1) / kStepWarpsPerBlock,
                                              kStepWarpsPerBlock * 32, smem, st>>>(a, q);
    return cudaSuccess;
}

// The lane-per-cell kernel costs about the same per attempt whatever the cell
// and the sub-tile; the bit-parallel one costs a step of a lane for 512 / (cx cy)
// attempts, with GX * GY of 32 lanes at work.  One MCS at L=8192, p=0.95, q=0.05
// (us, bit-parallel and lane per cell):
//   256x64 sub-tiles (32 groups): 8x8 267, 592; 16x8 443, 590; 8x16 499, 606;
//                                 32x8 807, 613; 16x16 801, 586; 32x16 1441, 633
//   64x64 (8 groups):             8x4 414, 524; 16x4 674, 547; 8x8 660, 436;
//                                 16x8 1123, 429; 16x16 2036, 481; 32x16 3756, 668
//   32x32 (2 groups):             8x4 1319, 679; 8x8 2136, 546; 16x16 6835, 703
// so the line lies at cx cy 32 / groups = 256.  Cells four columns wide (half
// rows of two sites) and sub-tiles whose last group row is so incomplete that
// they need more turns than the registers hold stay bit-parallel.
template <int CX, int CY, bool RANDOM, int SPEC>
cudaError_t launch_cells_variant(const StepArgs &a, cudaStream_t st) {
    if constexpr (CX >= 8) {
        const LaneSplit q = lane_split<CX, CY, RANDOM>(a.GX, a.By);
        if (q.nc <= static_cast<uint32_t>(LaneCells<CX, CY>::NCMAX) && CX * CY * 32u >= 256u * a.GX * a.GY)
            return launch_lane_cells<CX, CY, RANDOM, SPEC>(a, q, st);
    }
    const uint32_t n_tiles = work_tiles(a);
    cells_step_kernel<CX, CY, RANDOM, SPEC>
        <<<(n_tiles + kStepWarpsPerBlock - 1) / kStepWarpsPerBlock, kStepWarpsPerBlock * 32, 0, st>>>(a);
    return cudaSuccess;
}

template <int CX, int CY>
cudaError_t launch_cells_shape(const StepArgs &a, bool any_random, cudaStream_t st) {
    if (!any_random && a.p_always == 0xFFFFFFFFu && a.q_always == 0u)
        return launch_cells_variant<CX, CY, false, 1>(a, st);  // deposition only (p = 1, q = 0)
    if (any_random && a.p_random && a.q_random && !ties_matter(a.thr_p, a.thr_q))
        return launch_cells_variant<CX, CY, true, 3>(a, st);   // both inside, every tie refused
    if (any_random && a.p_random && a.q_random)
        return launch_cells_variant<CX, CY, true, 2>(a, st);   // both rates inside (0, 1)
    if (any_random) return launch_cells_variant<CX, CY, true, 0>(a, st);
    return launch_cells_variant<CX, CY, false, 0>(a, st);
}

}  // namespace oct
