// Lattice-wide kernels: flat start, exact roughness, layout conversion.
//
// Roughness (Eq. (3), mean over the L^2 sites): heights relative to h(0,0)=0,
//   h(0,y) = sum_{y'=1..y} (2 Y(0,y') - 1),
//   h(x,y) = h(0,y) + r(x,y),  r(x,y) = sum_{x'=1..x} (2 X(x',y) - 1).
// Pass 1 (one warp per row): with q(x) = sum_{x'=0..x} (2X(x',y)-1) and
// s0 = 2X(0,y)-1, r = q - s0, so the row sums of r and r^2 follow from those
// of q.  A warp takes the row in chunks of 512 words, 16 consecutive words per
// lane (16-byte coalesced loads); each lane reduces its words with a 256-entry
// byte table (per byte: the sum of the running step inside it, of its square,
// the net step and the extremes) and integer multiply-adds, and a warp scan of
// the lanes' net steps lifts the lane sums to the row.  Pass 2: a scan of the
// column bits gives h0 = h(0,y), and S1 = sum_y (L h0 + R1), S2 = sum_y (L h0^2 +
// 2 h0 R1 + R2) accumulate in 128-bit integers, per block of rows and then
// over the blocks.  Per-row terms are bounded by
// 4 L^3 < 2^63 for L <= 2^20, so only the cross-row sums need 128 bits.
#include <algorithm>

#include "oct_internal.h"
#include "overlap.cuh"

namespace oct {
namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;

__global__ void init_flat_kernel(uint32_t *lat, uint32_t rows, uint64_t n_words, uint32_t wpr) {
    // X = Y = (x+y) & 1: odd x set on even rows, even x set on odd rows (the
    // buffer's first row is an even lattice row).
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < n_words;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t row = (i / wpr) % rows;
        lat[i] = (row & 1u) ? 0x55555555u : 0xAAAAAAAAu;
    }
}

// Byte table of the row pass.  For byte value v, with the running step
// e_i = sum_{j<=i} (2 b_j - 1), i = 0..7, t1 = sum e_i, t2 = sum e_i^2, n = e_7:
//   .x = 2 t1 + t2 2^17 + n 2^27   (mod 2^32; |2 t1| <= 72 < 2^17 <= t2 2^17)
//   .y = (min e_i + kW2Bias) | (kW2Bias - max e_i) << 16
// The four .x of a word plus 512 hold sum 2 t1 + 512 in bits 0..16 and
// sum t2 <= 816 in bits 17..26; read as a signed word, floor(.x / 2^27) = n
// (t2 >= 4, so the part below bit 27 is positive).
constexpr uint32_t kW2Bias = 0x8000u;

__device__ __forceinline__ uint2 byte_entry(uint32_t v) {
    int e = 0, s1 = 0, s2 = 0, mn = 1 << 20, mx = -(1 << 20);
    for (int i = 0; i < 8; ++i) {
        e += ((v >> i) & 1u) ? 1 : -1;
        s1 += e;
        s2 += e * e;
        mn = min(mn, e);
        mx = max(mx, e);
    }
    uint2 r;
    r.x = static_cast<uint32_t>(2 * s1) + (static_cast<uint32_t>(s2) << 17) + (static_cast<uint32_t>(e) << 27);
    r.y = (kW2Bias + static_cast<uint32_t>(mn)) | ((kW2Bias - static_cast<uint32_t>(mx)) << 16);
    return r;
}

// Halfword-wise unsigned minimum of two packed pairs.
__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// hi32(a * b) + c, signed
__device__ __forceinline__ int mad_hi_s32(uint32_t a, int b, int c) {
    int d;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

constexpr int kW2Warps = 8;
constexpr int kW2BlocksPerSM = 3;
constexpr int kW2LaneWords = 16;                      // words per lane and chunk
constexpr uint32_t kW2ChunkWords = 32u * kW2LaneWords;  // words per warp and chunk
// Table entry v of copy c at byte offset 256 v + 8 c, c = lane % 16: the shared
// address of byte k of a word w is one byte permute (byte k of w above the
// copy offset).  The 16 lanes of a half-warp (one 8-byte shared-memory
// transaction) read banks 2c, 2c + 1, whatever bytes they look up.
constexpr int kW2TableBytes = 256 * 256;

// Running sums of one lane over the words of its chunk: P = running step
// before the current word (relative to the lane's first bit); M2, Mz and SPw
// accumulate the square sums, the linear sums and the word-start prefixes
// (with constant offsets removed once per chunk); ext is the packed pair of
// extremes of the lane's running step, biased by kW2Bias.
struct W2Lane {
    int P;
    uint32_t M2, Mz;
    int SPw;
    uint32_t ext;
    uint32_t St;  // sum of the words' S (see w2_word): the sums t2 are read off it once per chunk
};

// One 32-site word w.  With a_j the running step inside the word (j = 0..31)
// and P the lane's running step before it, the word adds
//   sum (P + a_j) = 32 P + A1,  sum (P + a_j)^2 = P (32 P + 2 A1) + A2.
// Byte k (P_k = running step before it inside the word, P_0 = 0) contributes
// 8 P_k + t1 to A1 and 8 P_k^2 + 2 P_k t1 + t2 to A2.  u = 8 P_k + .x is
// 8 P_k + 2 t1 in its low 17 bits (the t2 and n fields only add multiples of
// 2^17), so
//   acc2 = 2^16 + sum_{k>=1} u P_k = 2^16 + V (mod 2^17), |V| <= 3 * 264 * 24 < 2^16,
// with V = sum (8 P_k^2 + 2 P_k t1), A2 = V + sum t2 and 2 A1 = 16 sum P_k + sum 2 t1.
// P_{k+1} = P_k + n is one multiply-high of .x.
__device__ __forceinline__ void w2_word(const unsigned char *tab, uint32_t slot, uint32_t w, W2Lane &a) {
    const uint2 e0 = *reinterpret_cast<const uint2 *>(tab + __byte_perm(w, slot, 0x6504));
    const uint2 e1 = *reinterpret_cast<const uint2 *>(tab + __byte_perm(w, slot, 0x6514));
    const uint2 e2 = *reinterpret_cast<const uint2 *>(tab + __byte_perm(w, slot, 0x6524));
    const uint2 e3 = *reinterpret_cast<const uint2 *>(tab + __byte_perm(w, slot, 0x6534));
    // extremes: .y + P_k (1 - 2^16) = (min + bias + P_k) | (bias - max - P_k) << 16
    const int p1 = mad_hi_s32(e0.x, 32, 0);
    uint32_t u = static_cast<uint32_t>(p1) * 8u + e1.x;
    uint32_t acc2 = u * static_cast<uint32_t>(p1) + 0x10000u;
    const uint32_t c1 = e1.y + static_cast<uint32_t>(p1) * 0xFFFF0001u;
    const int p2 = mad_hi_s32(e1.x, 32, p1);
    u = static_cast<uint32_t>(p2) * 8u + e2.x;
    acc2 += u * static_cast<uint32_t>(p2);
    const uint32_t c2 = e2.y + static_cast<uint32_t>(p2) * 0xFFFF0001u;
    const int p3 = mad_hi_s32(e2.x, 32, p2);
    u = static_cast<uint32_t>(p3) * 8u + e3.x;
    acc2 += u * static_cast<uint32_t>(p3);
    const uint32_t c3 = e3.y + static_cast<uint32_t>(p3) * 0xFFFF0001u;
    const int p4 = mad_hi_s32(e3.x, 32, p3);
    const uint32_t ext = min_u16x2(min_u16x2(e0.y, c1), min_u16x2(c2, c3));
    // S = sum .x + 512: Sl = sum 2 t1 + 512, bits 17..26 sum t2
    const uint32_t S = e0.x + e1.x + e2.x + e3.x + 512u;
    const uint32_t Sl = S & 0x1FFFFu;
    a.St += S;
    const uint32_t SP = static_cast<uint32_t>(p1 + p2 + p3);
    const uint32_t tw = SP * 16u + Sl;  // 2 A1 + 512
    // lane sums: zp = 32 P + 2 A1 + 512, P zp + Vb + t2 = (word's square sum)
    // + 512 P + 2^16; the offsets are removed at the end of the chunk
    const uint32_t P = static_cast<uint32_t>(a.P);
    const uint32_t zp = P * 32u + tw;
    a.M2 = zp * P + a.M2 + (acc2 & 0x1FFFFu);
    a.Mz += zp;
    a.SPw += a.P;
    a.ext = min_u16x2(a.ext, ext + P * 0xFFFF0001u);
    a.P += p4;
}

// The lane's kW2LaneWords words of the chunk at word w0 of a row (16-byte
// loads where the row allows them); words past the row's end read as 0 and
// are not counted.
__device__ __forceinline__ void load_lane(const uint32_t *row, uint32_t w, uint32_t wpr, bool vec_ok,
                                          uint32_t (&v)[kW2LaneWords]) {
    if (vec_ok && w + kW2LaneWords <= wpr) {
#pragma unroll
        for (int i = 0; i < kW2LaneWords / 4; ++i) {
            const uint4 q = *reinterpret_cast<const uint4 *>(row + w + 4 * i);
            v[4 * i] = q.x;
            v[4 * i + 1] = q.y;
            v[4 * i + 2] = q.z;
            v[4 * i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kW2LaneWords; ++i) v[i] = (w + i < wpr) ? row[w + i] : 0u;
    }
}

__global__ void __launch_bounds__(kW2Warps * 32, kW2BlocksPerSM)
    w2_rows_kernel(const uint32_t *lat, uint32_t L, uint32_t nrows, uint32_t plane_rows, W2RowSums *rows) {
    extern __shared__ __align__(16) unsigned char w2_table[];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        const uint2 e = byte_entry(static_cast<uint32_t>(i));
#pragma unroll
        for (int c = 0; c < 16; ++c) *reinterpret_cast<uint2 *>(w2_table + 256 * i + 8 * c) = e;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t slot = 8u * static_cast<uint32_t>(lane & 15);
    const uint32_t wpr = L >> 5;
    const uint32_t *Yp = lat + static_cast<size_t>(plane_rows) * wpr;
    // 16-byte loads need every row to start on a 16-byte boundary
    const bool vec_ok = (wpr % 4u) == 0u && (reinterpret_cast<uintptr_t>(lat) % 16u) == 0u;
    // The warp's rows y0, y0 + stride, ... are taken chunk by chunk (chunks of
    // kW2ChunkWords words, lane i on words 16i..16i+15 of the chunk); the next
    // chunk's loads, across row ends too, are issued before the current chunk
    // is reduced.
    const uint32_t stride = gridDim.x * kW2Warps;
    const uint32_t nchunks = (wpr + kW2ChunkWords - 1) / kW2ChunkWords;
    uint32_t y = blockIdx.x * kW2Warps + (threadIdx.x >> 5), c = 0;
    uint32_t v[kW2LaneWords], vn[kW2LaneWords];
    if (y < nrows) load_lane(lat + static_cast<size_t>(y) * wpr, kW2LaneWords * lane, wpr, vec_ok, v);
    long long base = 0;  // q just before the current chunk
    long long q1 = 0, q2 = 0;
    int qmin = 1 << 30, qmax = -(1 << 30);
    while (y < nrows) {
        const uint32_t w0 = c * kW2ChunkWords;
        const uint32_t w = w0 + kW2LaneWords * lane;
        const bool last = c + 1 == nchunks;
        const uint32_t ny = last ? y + stride : y, nc = last ? 0u : c + 1;
        if (ny < nrows)
            load_lane(lat + static_cast<size_t>(ny) * wpr, nc * kW2ChunkWords + kW2LaneWords * lane, wpr, vec_ok, vn);
        W2Lane a{0, 0u, 0u, 0, 0xFFFFFFFFu, 0u};
        uint32_t nw = 0;
        if (w0 + kW2ChunkWords <= wpr) {
#pragma unroll
            for (int j = 0; j < kW2LaneWords; ++j) w2_word(w2_table, slot, v[j], a);
            nw = kW2LaneWords;
        } else {
#pragma unroll
            for (int j = 0; j < kW2LaneWords; ++j)
                if (w + j < wpr) {
                    w2_word(w2_table, slot, v[j], a);
                    ++nw;
                }
        }
        // lane-relative sums: sum q' and sum q'^2 over the lane's 32 nw sites
        // (|q'| <= 512, so both fit 32 bits), extremes and net step
        const int M2 = static_cast<int>(a.M2 + ((a.St - (static_cast<uint32_t>(a.P) << 27)) >> 17) -
                                        512u * static_cast<uint32_t>(a.SPw) - 65536u * nw);
        const int M1 = static_cast<int>(a.Mz + 32u * static_cast<uint32_t>(a.SPw) - 512u * nw) / 2;
        const int step = a.P;
        int incl = step;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += n;
        }
        // lift to the row: q = B + q' with B = q before this lane's first bit
        const long long B = base + (incl - step);
        const long long nbits = 32ll * nw;
        q1 += nbits * B + M1;
        q2 += nbits * B * B + 2 * B * M1 + M2;
        if (nw > 0) {
            const int lmn = static_cast<int>(a.ext & 0xFFFFu) - static_cast<int>(kW2Bias);
            const int lmx = static_cast<int>(kW2Bias) - static_cast<int>(a.ext >> 16);
            qmin = min(qmin, static_cast<int>(B) + lmn);
            qmax = max(qmax, static_cast<int>(B) + lmx);
        }
        base += __shfl_sync(kFull, incl, 31);
        if (last) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                q1 += __shfl_xor_sync(kFull, q1, o);
                q2 += __shfl_xor_sync(kFull, q2, o);
            }
            qmin = __reduce_min_sync(kFull, qmin);
            qmax = __reduce_max_sync(kFull, qmax);
            if (lane == 0) {
                const uint32_t *row = lat + static_cast<size_t>(y) * wpr;
                const long long s0 = (row[0] & 1u) ? 1 : -1;
                const long long Ll = L;
                W2RowSums o;
                o.r1 = q1 - Ll * s0;
                o.r2 = q2 - 2 * s0 * q1 + Ll * s0 * s0;
                o.rmin = qmin - static_cast<int>(s0);
                o.rmax = qmax - static_cast<int>(s0);
                o.c = static_cast<int>(Yp[static_cast<size_t>(y) * wpr] & 1u);
                o.pad = 0;
                rows[y] = o;
            }
            base = 0;
            q1 = q2 = 0;
            qmin = 1 << 30;
            qmax = -(1 << 30);
        }
        y = ny;
        c = nc;
#pragma unroll
        for (int j = 0; j < kW2LaneWords; ++j) v[j] = vn[j];
    }
}

// Pass 2 runs in two kernels.  Pass 2a: one block per kW2BlockRows rows
// computes, relative to the height h0 of its first row, the sums
//   A = sum_y (L h0l + R1),  Q = sum_y (L h0l^2 + 2 h0l R1 + R2)
// (h0l = h0(y) - h0(first row)), the extremes of h0l + r and the rise of h0l
// to its last row, and stores them in place of its first row record.  Pass 2b
// (one block) scans the rises for each block's first-row height H and adds
// S1 = sum (A + L n H), S2 = sum (Q + 2 H A + L n H^2) over the blocks
// (n rows each) in 128-bit integers.
constexpr int kW2BlockRows = 256;
constexpr int kW2CombineThreads = 1024;

// The record of one pass-2a block, stored over its first row record.
struct W2BlockSums {
    long long a;                 // A
    unsigned long long q_lo;     // Q (>= 0: a sum of squared heights), bits 0..63
    unsigned int q_hi;           // bits 64..95 (Q < 2^70 for L <= 2^20)
    int lo, hi;                  // extremes of h0l + r over the block's rows
    int ec;                      // 2 h0l(last row) + Y(0, first row)
};
static_assert(sizeof(W2BlockSums) == sizeof(W2RowSums), "a block record replaces one row record");

// 128-bit unsigned sum of (lo, hi) pairs over a warp, in lane 0.
__device__ __forceinline__ void warp_sum_u128(unsigned long long &lo, unsigned long long &hi) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l2 = __shfl_down_sync(kFull, lo, o);
        const unsigned long long h2 = __shfl_down_sync(kFull, hi, o);
        const unsigned long long nl = lo + l2;
        hi = hi + h2 + (nl < lo ? 1ull : 0ull);
        lo = nl;
    }
}

__global__ void __launch_bounds__(kW2BlockRows)
    w2_block_kernel(W2RowSums *rows, uint32_t L, uint32_t nrows) {
    __shared__ int wsum[kW2BlockRows / 32];
    __shared__ long long sa[kW2BlockRows / 32];
    __shared__ unsigned long long sqlo[kW2BlockRows / 32], sqhi[kW2BlockRows / 32];
    __shared__ int slo[kW2BlockRows / 32], shi[kW2BlockRows / 32];
    __shared__ int last_h0l;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t y0 = blockIdx.x * kW2BlockRows, y = y0 + tid;
    const uint32_t n = min(static_cast<uint32_t>(kW2BlockRows), nrows - y0);
    const bool valid = static_cast<uint32_t>(tid) < n;
    W2RowSums r{};
    if (valid) r = rows[y];
    // column step into row y from row y - 1 (none into the block's first row)
    int incl = (valid && tid > 0) ? (r.c ? 1 : -1) : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    const long long h = before + incl;  // h0l(y)
    if (static_cast<uint32_t>(tid) == n - 1) last_h0l = static_cast<int>(h);
    const long long Ll = L;
    long long a = 0;
    unsigned long long qlo = 0, qhi = 0;
    int lo = 1 << 30, hi = -(1 << 30);
    if (valid) {
        a = Ll * h + r.r1;
        // sum_x (h0l + r(x))^2 >= 0; |terms| < 2^63 for L <= 2^20
        const __int128 q = static_cast<__int128>(Ll * h * h) + static_cast<__int128>(2 * h * r.r1) +
                           static_cast<__int128>(r.r2);
        qlo = static_cast<unsigned long long>(q);
        qhi = static_cast<unsigned long long>(q >> 64);
        lo = static_cast<int>(h) + r.rmin;
        hi = static_cast<int>(h) + r.rmax;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(kFull, a, o);
    warp_sum_u128(qlo, qhi);
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if (lane == 0) {
        sa[warp] = a;
        sqlo[warp] = qlo;
        sqhi[warp] = qhi;
        slo[warp] = lo;
        shi[warp] = hi;
    }
    __syncthreads();
    if (tid == 0) {
        W2BlockSums b;
        b.a = 0;
        unsigned __int128 q = 0;
        b.lo = 1 << 30;
        b.hi = -(1 << 30);
        for (int w = 0; w < kW2BlockRows / 32; ++w) {
            b.a += sa[w];
            q += (static_cast<unsigned __int128>(sqhi[w]) << 64) | sqlo[w];
            b.lo = min(b.lo, slo[w]);
            b.hi = max(b.hi, shi[w]);
        }
        b.q_lo = static_cast<unsigned long long>(q);
        b.q_hi = static_cast<unsigned int>(q >> 64);
        b.ec = 2 * last_h0l + r.c;  // thread 0 holds the block's first row
        *reinterpret_cast<W2BlockSums *>(rows + y0) = b;
    }
}

__global__ void __launch_bounds__(kW2CombineThreads)
    w2_combine_kernel(const W2RowSums *rows, uint32_t L, uint32_t nrows, W2Result *out) {
    __shared__ long long part[kW2CombineThreads];
    __shared__ unsigned long long s2lo[kW2CombineThreads / 32], s2hi[kW2CombineThreads / 32];
    __shared__ long long s1w[kW2CombineThreads / 32], low[kW2CombineThreads / 32], hiw[kW2CombineThreads / 32];
    const int tid = threadIdx.x;
    const uint32_t nb = (nrows + kW2BlockRows - 1) / kW2BlockRows;
    const uint32_t per = (nb + kW2CombineThreads - 1) / kW2CombineThreads;
    const uint32_t b_begin = min(nb, tid * per), b_end = min(nb, (tid + 1) * per);
    auto rec = [&](uint32_t b) {
        return *reinterpret_cast<const W2BlockSums *>(rows + static_cast<size_t>(b) * kW2BlockRows);
    };
    // rise of h0 from the last row of block b - 1 to the last row of block b
    auto rise = [](const W2BlockSums &r, uint32_t b) {
        return static_cast<long long>(r.ec >> 1) + (b > 0 ? ((r.ec & 1) ? 1 : -1) : 0);
    };
    long long local = 0;
    for (uint32_t b = b_begin; b < b_end; ++b) local += rise(rec(b), b);
    part[tid] = local;
    __syncthreads();
    for (int o = 1; o < kW2CombineThreads; o <<= 1) {
        const long long v = (tid >= o) ? part[tid - o] : 0;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    long long last = part[tid] - local;  // h0 of the last row before b_begin
    __int128 S1 = 0, S2 = 0;
    long long lo = 1ll << 62, hi = -(1ll << 62);
    const long long Ll = L;
    for (uint32_t b = b_begin; b < b_end; ++b) {
        const W2BlockSums r = rec(b);
        const long long H = last + (b > 0 ? ((r.ec & 1) ? 1 : -1) : 0);  // h0 of the block's first row
        const long long n = min(static_cast<uint32_t>(kW2BlockRows), nrows - b * kW2BlockRows);
        const __int128 Q = static_cast<__int128>((static_cast<unsigned __int128>(r.q_hi) << 64) | r.q_lo);
        S1 += static_cast<__int128>(r.a) + static_cast<__int128>(Ll * n) * H;
        S2 += Q + static_cast<__int128>(2 * H) * r.a + static_cast<__int128>(Ll * n) * H * H;
        lo = min(lo, H + r.lo);
        hi = max(hi, H + r.hi);
        last = H + (r.ec >> 1);
    }
    if (b_end == nb && b_begin < b_end) out->e_last = last;  // h0 of the last row
    // block reduction of S1 (fits 64 bits for L <= 2^20), S2 (128 bits), extremes
    long long s1 = static_cast<long long>(S1);
    unsigned long long s2l = static_cast<unsigned long long>(S2);
    unsigned long long s2h = static_cast<unsigned long long>(S2 >> 64);
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_down_sync(kFull, s1, o);
        lo = min(lo, __shfl_down_sync(kFull, lo, o));
        hi = max(hi, __shfl_down_sync(kFull, hi, o));
    }
    warp_sum_u128(s2l, s2h);
    if ((tid & 31) == 0) {
        s1w[tid >> 5] = s1;
        s2lo[tid >> 5] = s2l;
        s2hi[tid >> 5] = s2h;
        low[tid >> 5] = lo;
        hiw[tid >> 5] = hi;
    }
    __syncthreads();
    if (tid == 0) {
        long long a1 = 0, amn = 1ll << 62, amx = -(1ll << 62);
        unsigned __int128 a2 = 0;
        for (int w = 0; w < kW2CombineThreads / 32; ++w) {
            a1 += s1w[w];
            a2 += (static_cast<unsigned __int128>(s2hi[w]) << 64) | s2lo[w];
            amn = min(amn, low[w]);
            amx = max(amx, hiw[w]);
        }
        out->s1 = a1;
        out->s2_lo = static_cast<unsigned long long>(a2);
        out->s2_hi = static_cast<unsigned long long>(a2 >> 64);
        out->lo = amn;
        out->hi = amx;
        out->hmax = max(amn < 0 ? -amn : amn, amx < 0 ? -amx : amx);
        out->f0 = (rec(0).ec & 1) ? 1 : -1;
    }
}

// Lattices of up to kW2SmallL sites a side: one or many of them in two
// launches.  A row of 16384 sites is 512 words, one warp's chunk, so a row is
// one step: 2^sl_log lanes take it, 2^lw_log words each, and a warp takes
// 32 / 2^sl_log rows at once (w2_rows_kernel gives a row to a warp at 16 words
// per lane: at L = 2048 four of its lanes have work).  Pass 2 is one block per
// lattice and writes the result, the counters and the time to where the job
// points (page-locked host memory: no copies).  Every sum of a lattice this
// small fits 64 bits: S2 <= 2^28 sites x (2^14)^2 = 2^56.
// Bound by launches and latency, not by work: one W^2 of L=256 went from four
// kernels and two copies (33 us with the wait) to two kernels (17 us), and the
// W^2 of 256 replicas (L = 64..2048, 375 M sites) from 256 such calls (8.3 ms)
// to 0.5 ms.  Both launches overlap the one before them: the tables are
// filled during the last device step (8 MCS of L=256 and their W^2: 132 to
// 128 us).
constexpr int kW2SmallThreads = 512;  // of the second launch
// Rows of one lattice that a single block may finish; a lattice alone with more
// takes the large passes, whose second one has a block per 256 rows (W^2 in two
// launches and in four, us: L=8192 41, 41; 12288 59, 44; 16384 70, 46).
constexpr uint32_t kW2FinishRows = 8192;

// Words j .. j+3 of the lane's nw, as one 16-byte load where allowed.
__device__ __forceinline__ void load_quad(const uint32_t *row, uint32_t j, uint32_t nw, bool vec_ok,
                                          uint32_t (&v)[4]) {
    if (vec_ok && j + 4u <= nw) {
        const uint4 q = *reinterpret_cast<const uint4 *>(row + j);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else {
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) v[i] = (j + i < nw) ? row[j + i] : 0u;
    }
}

// A job list passed by value; the kernels read it where no list in device
// memory is given.  Asynchronous measurements take it: a copy to the device
// would need staging that outlives the call.  Up to 32 lattices (2.8 KB of the
// 4 KB of arguments) share two launches; one by one the device idled in each:
// 24 served jobs with 192 W^2 went from 8.75 to 6.9 ms.
template <uint32_t N>
struct W2Pack {
    W2Job j[N];
};

template <uint32_t N>
__global__ void __launch_bounds__(kW2Warps * 32, kW2BlocksPerSM)
    w2_small_rows_kernel(const __grid_constant__ W2Pack<N> pack, const W2Job *jobs, uint32_t n, uint32_t n_tasks,
                         W2RowSums *rows) {
    launch_dependents();
    extern __shared__ __align__(16) unsigned char w2_table[];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        const uint2 e = byte_entry(static_cast<uint32_t>(i));
#pragma unroll
        for (int c = 0; c < 16; ++c) *reinterpret_cast<uint2 *>(w2_table + 256 * i + 8 * c) = e;
    }
    __syncthreads();
    wait_for_previous_grid();  // the table needs nothing of it
    const W2Job *list = jobs ? jobs : pack.j;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t slot = 8u * (lane & 15u);
    for (uint32_t task = blockIdx.x * kW2Warps + (threadIdx.x >> 5); task < n_tasks; task += gridDim.x * kW2Warps) {
        uint32_t a0 = 0, b0 = n;  // the last job whose first task is not past this one
        while (b0 - a0 > 1u) {
            const uint32_t m = (a0 + b0) >> 1;
            if (list[m].task_first <= task) a0 = m; else b0 = m;
        }
        const W2Job *J = list + a0;
        const uint32_t wpr = J->L >> 5, nrows = J->nrows, lw = 1u << J->lw_log, sl = 1u << J->sl_log;
        const uint32_t y = ((task - J->task_first) << (5u - J->sl_log)) + (lane >> J->sl_log);
        const uint32_t li = lane & (sl - 1u), w = li * lw;
        const uint32_t nw = (y < nrows && w < wpr) ? min(lw, wpr - w) : 0u;
        const uint32_t *row = J->lat + static_cast<size_t>(min(y, nrows - 1u)) * wpr;
        const bool vec_ok = lw >= 4u && (wpr & 3u) == 0u && (reinterpret_cast<uintptr_t>(J->lat) & 15u) == 0u;
        W2Lane a{0, 0u, 0u, 0, 0xFFFFFFFFu, 0u};
        uint32_t v[4], vn[4] = {0u, 0u, 0u, 0u};
        load_quad(row + w, 0u, nw, vec_ok, v);
        for (uint32_t j = 0; j < lw; j += 4u) {
            if (j + 4u < lw) load_quad(row + w, j + 4u, nw, vec_ok, vn);
#pragma unroll
            for (uint32_t i = 0; i < 4u; ++i)
                if (j + i < nw) w2_word(w2_table, slot, v[i], a);
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = vn[i];
        }
        // as in w2_rows_kernel: the lane's sums, lifted by the steps before it
        const int M2 = static_cast<int>(a.M2 + ((a.St - (static_cast<uint32_t>(a.P) << 27)) >> 17) -
                                        512u * static_cast<uint32_t>(a.SPw) - 65536u * nw);
        const int M1 = static_cast<int>(a.Mz + 32u * static_cast<uint32_t>(a.SPw) - 512u * nw) / 2;
        int incl = a.P;
        for (uint32_t o = 1; o < sl; o <<= 1) {
            const int x = __shfl_up_sync(kFull, incl, o, sl);
            if (li >= o) incl += x;
        }
        const long long B = incl - a.P, nbits = 32ll * nw;
        long long q1 = nbits * B + M1, q2 = nbits * B * B + 2 * B * M1 + M2;
        int qmin = 1 << 30, qmax = -(1 << 30);
        if (nw > 0) {
            qmin = static_cast<int>(B) + static_cast<int>(a.ext & 0xFFFFu) - static_cast<int>(kW2Bias);
            qmax = static_cast<int>(B) + static_cast<int>(kW2Bias) - static_cast<int>(a.ext >> 16);
        }
        for (uint32_t o = sl >> 1; o > 0; o >>= 1) {
            q1 += __shfl_xor_sync(kFull, q1, o);
            q2 += __shfl_xor_sync(kFull, q2, o);
            qmin = min(qmin, __shfl_xor_sync(kFull, qmin, o));
            qmax = max(qmax, __shfl_xor_sync(kFull, qmax, o));
        }
        if (li == 0 && y < nrows) {
            const long long s0 = (row[0] & 1u) ? 1 : -1;
            const long long Ll = J->L;
            W2RowSums o;
            o.r1 = q1 - Ll * s0;
            o.r2 = q2 - 2 * s0 * q1 + Ll;
            o.rmin = qmin - static_cast<int>(s0);
            o.rmax = qmax - static_cast<int>(s0);
            o.c = static_cast<int>(row[static_cast<size_t>(J->plane_rows) * wpr] & 1u);
            o.pad = 0;
            rows[J->row_first + y] = o;
        }
    }
}

// Pass 2: one block per lattice, a run of consecutive rows per thread.
template <uint32_t N>
__global__ void __launch_bounds__(kW2SmallThreads)
    w2_small_finish_kernel(const __grid_constant__ W2Pack<N> pack, const W2Job *jobs, const W2RowSums *all_rows) {
    wait_for_previous_grid();
    constexpr int kWarps = kW2SmallThreads / 32;
    __shared__ int wsum[kWarps];
    __shared__ long long red[6][kWarps];
    __shared__ long long last_h;
    const W2Job &J = (jobs ? jobs : pack.j)[N > 1u || jobs ? blockIdx.x : 0u];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nrows = J.nrows;
    const W2RowSums *rows = all_rows + J.row_first;
    const uint32_t per = (nrows + kW2SmallThreads - 1) / kW2SmallThreads;
    const uint32_t y0 = min(nrows, tid * per), y1 = min(nrows, y0 + per);
    // one pass over the thread's rows, relative to the height before its first one;
    // several rows' records are in flight at a time
    const long long Ll = J.L;
    long long v[4] = {0, 0, 0, 0};  // S1, S2, counters
    int hl = 0, rlo = 1 << 30, rhi = -(1 << 30);
#pragma unroll 8
    for (uint32_t y = y0; y < y1; ++y) {
        const W2RowSums r = rows[y];
        hl += y == 0 ? 0 : r.c ? 1 : -1;
        v[0] += Ll * hl + r.r1;
        v[1] += Ll * hl * hl + 2 * hl * r.r1 + r.r2;
        rlo = min(rlo, hl + r.rmin);
        rhi = max(rhi, hl + r.rmax);
    }
    int incl = hl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    long long h = incl - hl;  // before the thread's first row
    for (int w = 0; w < warp; ++w) h += wsum[w];
    const long long n = y1 - y0;
    v[1] += 2 * h * v[0] + Ll * n * h * h;
    v[0] += Ll * n * h;
    long long lo = 1ll << 40, hi = -(1ll << 40);
    if (n > 0) {
        lo = h + rlo;
        hi = h + rhi;
    }
    if (y0 < y1 && y1 == nrows) last_h = h + hl;
    if (J.cnt)
        for (uint32_t i = tid; i < J.cnt_n; i += kW2SmallThreads) {
            v[2] += static_cast<long long>(J.cnt[i]);
            v[3] += static_cast<long long>(J.cnt[J.cnt_off + i]);
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] += __shfl_down_sync(kFull, v[i], o);
        lo = min(lo, __shfl_down_sync(kFull, lo, o));
        hi = max(hi, __shfl_down_sync(kFull, hi, o));
    }
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) red[i][warp] = v[i];
        red[4][warp] = lo;
        red[5][warp] = hi;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kWarps; ++w) {
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] += red[i][w];
            lo = min(lo, red[4][w]);
            hi = max(hi, red[5][w]);
        }
        W2Result o;
        o.s1 = v[0];
        o.s2_lo = static_cast<unsigned long long>(v[1]);
        o.s2_hi = 0;
        o.hmax = max(lo < 0 ? -lo : lo, hi < 0 ? -hi : hi);
        o.lo = lo;
        o.hi = hi;
        o.e_last = last_h;
        o.f0 = rows[0].c ? 1 : -1;
        *J.res = o;
        if (J.cnt) {
            J.cnt_out[0] = v[2];
            J.cnt_out[1] = v[3];
        }
        if (J.t) *J.t_out = *J.t;
    }
}

// The counters and the time of a job whose sums the large passes took.
__global__ void w2_counters_kernel(const __grid_constant__ W2Job J) {
    __shared__ unsigned long long sum[2];
    if (threadIdx.x < 2u) sum[threadIdx.x] = 0ull;
    __syncthreads();
    if (J.cnt) {
        unsigned long long a = 0, b = 0;
        for (uint32_t i = threadIdx.x; i < J.cnt_n; i += blockDim.x) {
            a += J.cnt[i];
            b += J.cnt[J.cnt_off + i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(kFull, a, o);
            b += __shfl_down_sync(kFull, b, o);
        }
        if ((threadIdx.x & 31u) == 0u) {
            atomicAdd(&sum[0], a);
            atomicAdd(&sum[1], b);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2u && J.cnt) J.cnt_out[threadIdx.x] = static_cast<long long>(sum[threadIdx.x]);
    if (threadIdx.x == 0u && J.t) *J.t_out = *J.t;
}

// Interleave two 4-bit values: a0 b0 a1 b1 a2 b2 a3 b3 (LSB first).
__device__ __forceinline__ uint32_t interleave4(uint32_t a, uint32_t b) {
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) r |= (((a >> i) & 1u) << (2 * i)) | (((b >> i) & 1u) << (2 * i + 1));
    return r;
}

__global__ void pack_canonical_kernel(const uint32_t *lat, uint32_t L, uint32_t cy0, uint32_t ncy,
                                      uint32_t *out) {
    const uint32_t wpr = L >> 5, cpr = L >> 2;  // canonical words per canonical row
    const uint32_t *Yp = lat + static_cast<size_t>(L) * wpr;
    const uint64_t n = static_cast<uint64_t>(ncy) * cpr;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint32_t cy = cy0 + static_cast<uint32_t>(i / cpr), cx = static_cast<uint32_t>(i % cpr);
        const uint32_t w = (4u * cx) >> 5, b = (4u * cx) & 31u;
        uint32_t v = 0;
#pragma unroll
        for (int yy = 0; yy < 4; ++yy) {
            const size_t ro = static_cast<size_t>(4u * cy + yy) * wpr + w;
            v |= interleave4((lat[ro] >> b) & 0xFu, (Yp[ro] >> b) & 0xFu) << (8 * yy);
        }
        out[i] = v;
    }
}

__global__ void unpack_canonical_kernel(const uint32_t *in, uint32_t L, uint32_t cy0, uint32_t ncy,
                                        uint32_t *lat) {
    // one thread per planar word pair (X and Y) of lattice rows 4*cy0 .. 4*(cy0+ncy)-1
    const uint32_t wpr = L >> 5, cpr = L >> 2;
    uint32_t *Yp = lat + static_cast<size_t>(L) * wpr;
    const uint64_t n = static_cast<uint64_t>(ncy) * 4u * wpr;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint32_t lr = static_cast<uint32_t>(i / wpr), w = static_cast<uint32_t>(i % wpr);
        const uint32_t y = 4u * cy0 + lr, yy = y & 3u;
        uint32_t xv = 0, yv = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint32_t word = in[static_cast<size_t>(lr >> 2) * cpr + 8u * w + c] >> (8u * yy);
#pragma unroll
            for (int xx = 0; xx < 4; ++xx) {
                xv |= ((word >> (2 * xx)) & 1u) << (4 * c + xx);
                yv |= ((word >> (2 * xx + 1)) & 1u) << (4 * c + xx);
            }
        }
        lat[static_cast<size_t>(y) * wpr + w] = xv;
        Yp[static_cast<size_t>(y) * wpr + w] = yv;
    }
}

// One thread per counter slot (kNetSlots threads), then a block reduction.
__global__ void __launch_bounds__(kNetSlots)
    net_sum_kernel(const unsigned long long *net, const unsigned long long *draws, const unsigned long long *tails,
                   long long *out) {
    __shared__ long long part[3][kNetSlots / 32];
    const int i = threadIdx.x;
    long long s = static_cast<long long>(net[i]), d = static_cast<long long>(draws[i]),
              b = static_cast<long long>(tails[i]);
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_down_sync(kFull, s, o);
        d += __shfl_down_sync(kFull, d, o);
        b += __shfl_down_sync(kFull, b, o);
    }
    if ((i & 31) == 0) {
        part[0][i >> 5] = s;
        part[1][i >> 5] = d;
        part[2][i >> 5] = b;
    }
    __syncthreads();
    if (i < 3) {
        long long t = 0;
        for (int w = 0; w < kNetSlots / 32; ++w) t += part[i][w];
        out[i] = t;
    }
}

// SMs of the current device, with the shared-memory limit of a table kernel
// raised once per device.
cudaError_t table_kernel_setup(const void *kernel, int which, int *sm_count) {
    constexpr int kMaxDevices = 64;
    static int sms[kMaxDevices] = {};
    static bool smem_set[3][kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (sms[dev] <= 0) {
        e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    if (!smem_set[which][dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kW2TableBytes);
        if (e != cudaSuccess) return e;
        smem_set[which][dev] = true;
    }
    *sm_count = sms[dev];
    return cudaSuccess;
}

template <uint32_t N>
cudaError_t w2_small(const W2Pack<N> &pack, const W2Job *jobs, uint32_t n, uint32_t n_tasks, W2RowSums *rows,
                     cudaStream_t st) {
    int sms = 0;
    cudaError_t e = table_kernel_setup(reinterpret_cast<const void *>(w2_small_rows_kernel<N>), N > 1u ? 2 : 1, &sms);
    if (e != cudaSuccess) return e;
    const uint32_t want = (n_tasks + kW2Warps - 1) / kW2Warps, wave = static_cast<uint32_t>(sms) * kW2BlocksPerSM;
    e = launch_overlapped_smem(w2_small_rows_kernel<N>, dim3(std::min(want, wave)), dim3(kW2Warps * 32), kW2TableBytes,
                               true, st, pack, jobs, n, n_tasks, rows);
    if (e != cudaSuccess) return e;
    return launch_overlapped(w2_small_finish_kernel<N>, dim3(n), dim3(kW2SmallThreads), true, st, pack, jobs,
                             static_cast<const W2RowSums *>(rows));
}

// One lattice in the passes for large ones: a warp per row, then a block per
// kW2BlockRows rows, then one block.
cudaError_t w2_large(const uint32_t *lat, uint32_t L, uint32_t nrows, uint32_t plane_rows, W2RowSums *rows,
                     W2Result *out, cudaStream_t st) {
    // one wave of resident blocks (64 KB of table each), rows taken grid-stride
    int sms = 0;
    cudaError_t e = table_kernel_setup(reinterpret_cast<const void *>(w2_rows_kernel), 0, &sms);
    if (e != cudaSuccess) return e;
    const uint64_t want = (static_cast<uint64_t>(nrows) + kW2Warps - 1) / kW2Warps;
    const uint64_t wave = static_cast<uint64_t>(sms) * kW2BlocksPerSM;
    const int blocks = static_cast<int>(want < wave ? want : wave);
    w2_rows_kernel<<<blocks, kW2Warps * 32, kW2TableBytes, st>>>(lat, L, nrows, plane_rows, rows);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    w2_block_kernel<<<(nrows + kW2BlockRows - 1) / kW2BlockRows, kW2BlockRows, 0, st>>>(rows, L, nrows);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    w2_combine_kernel<<<1, kW2CombineThreads, 0, st>>>(rows, L, nrows, out);
    return cudaGetLastError();
}

int grid_for(uint64_t n, int threads) {
    const uint64_t b = (n + threads - 1) / threads;
    return static_cast<int>(b < 152ull * 32 ? (b ? b : 1) : 152ull * 32);
}

}  // namespace

cudaError_t launch_init_flat(uint32_t *lat, uint32_t L, cudaStream_t st) {
    return launch_init_flat_rows(lat, L, L, st);
}

cudaError_t launch_init_flat_rows(uint32_t *lat, uint32_t L, uint32_t rows, cudaStream_t st) {
    const uint32_t wpr = L >> 5;
    const uint64_t n = 2ull * rows * wpr;
    init_flat_kernel<<<grid_for(n, 256), 256, 0, st>>>(lat, rows, n, wpr);
    return cudaGetLastError();
}

cudaError_t launch_w2(const uint32_t *lat, uint32_t L, W2RowSums *rows, W2Result *out,
                      cudaStream_t st) {
    return launch_w2_rows(lat, L, L, L, rows, out, st);
}

cudaError_t launch_w2_rows(const uint32_t *lat, uint32_t L, uint32_t nrows, uint32_t plane_rows, W2RowSums *rows,
                           W2Result *out, cudaStream_t st) {
    if (L <= kW2SmallL) {
        W2Job j{};
        j.lat = lat;
        j.L = L;
        j.nrows = nrows;
        j.plane_rows = plane_rows;
        j.res = out;
        return launch_w2_small_pack(&j, 1, rows, st);
    }
    return w2_large(lat, L, nrows, plane_rows, rows, out, st);
}

uint32_t w2_small_split(W2Job *jobs, uint32_t n) {
    uint64_t words = 0;
    for (uint32_t i = 0; i < n; ++i) words += static_cast<uint64_t>(jobs[i].nrows) * (jobs[i].L >> 5);
    // As many words per lane (up to 16) as still leave a full device of
    // warps: the scan and the sums over the lanes of a row cost about three
    // words' work, but few warps leave the chip idle.
    uint32_t lw = 0;
    while (lw < 4u && (words >> (5u + lw + 1u)) >= 4096u) ++lw;
    uint32_t tasks = 0, rows = 0;
    for (uint32_t i = 0; i < n; ++i) {
        W2Job &j = jobs[i];
        const uint32_t wpr = j.L >> 5;
        j.lw_log = lw;
        while ((32u << j.lw_log) < wpr) ++j.lw_log;
        while (j.lw_log > 0u && (1u << (j.lw_log - 1u)) >= wpr) --j.lw_log;  // a row of few words
        j.sl_log = 0;
        while (((1u << j.sl_log) << j.lw_log) < wpr) ++j.sl_log;
        j.task_first = tasks;
        j.row_first = rows;
        const uint32_t per = 32u >> j.sl_log;
        tasks += (j.nrows + per - 1u) / per;
        rows += j.nrows;
    }
    return tasks;
}

cudaError_t launch_w2_small(const W2Job *jobs, uint32_t n, uint32_t n_tasks, W2RowSums *rows, cudaStream_t st) {
    return w2_small(W2Pack<1>{}, jobs, n, n_tasks, rows, st);
}

cudaError_t launch_w2_small_pack(W2Job *jobs, uint32_t n, W2RowSums *rows, cudaStream_t st) {
    if (n == 0 || n > kW2PackJobs) return cudaErrorInvalidValue;
    const uint32_t n_tasks = w2_small_split(jobs, n);
    const W2Job *none = nullptr;
    if (n == 1 && jobs[0].nrows > kW2FinishRows) {
        const W2Job &j = jobs[0];
        const cudaError_t e = w2_large(j.lat, j.L, j.nrows, j.plane_rows, rows, j.res, st);
        if (e != cudaSuccess || !(j.cnt || j.t)) return e;
        w2_counters_kernel<<<1, j.cnt_n > 256u ? 512 : 32, 0, st>>>(j);
        return cudaGetLastError();
    }
    if (n == 1) return w2_small(W2Pack<1>{{jobs[0]}}, none, 1, n_tasks, rows, st);
    W2Pack<kW2PackJobs> pack{};
    std::copy(jobs, jobs + n, pack.j);
    return w2_small(pack, none, n, n_tasks, rows, st);
}

cudaError_t launch_pack_canonical(const uint32_t *lat, uint32_t L, uint32_t cy0, uint32_t ncy,
                                  uint32_t *out, cudaStream_t st) {
    pack_canonical_kernel<<<grid_for(static_cast<uint64_t>(ncy) * (L >> 2), 256), 256, 0, st>>>(
        lat, L, cy0, ncy, out);
    return cudaGetLastError();
}

cudaError_t launch_unpack_canonical(const uint32_t *in, uint32_t L, uint32_t cy0, uint32_t ncy,
                                    uint32_t *lat, cudaStream_t st) {
    unpack_canonical_kernel<<<grid_for(static_cast<uint64_t>(ncy) * 4u * (L >> 5), 256), 256, 0,
                              st>>>(in, L, cy0, ncy, lat);
    return cudaGetLastError();
}

cudaError_t launch_net_sum(const unsigned long long *net, const unsigned long long *draws,
                           const unsigned long long *tails, long long *out, cudaStream_t st) {
    net_sum_kernel<<<1, kNetSlots, 0, st>>>(net, draws, tails, out);
    return cudaGetLastError();
}

}  // namespace oct
