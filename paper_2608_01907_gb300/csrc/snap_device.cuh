// snap_device.cuh -- device helpers of the epoch and objective kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "snap_internal.h"

namespace snap {

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel Random Numbers: As Easy
// as 1, 2, 3", SC'11): ten rounds of two 32x32->64 multiplies mixed with the
// other half of the counter and the round key; the key advances by the Weyl
// constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// Words 4g..4g+3 of the random stream of directed edge e in epoch t.
__device__ __forceinline__ uint4 edge_words(int64_t e, uint32_t t, uint32_t g, uint2 key) {
    return philox4x32_10(make_uint4((uint32_t)e, (uint32_t)((uint64_t)e >> 32), t, g), key);
}

// Uniform negative from V \ {i} (Algorithm 1): u = floor(w (n-1) / 2^32), s = u + (u >= i).
__device__ __forceinline__ int32_t negative_of(uint32_t w, int32_t i, uint32_t n_minus_1) {
    const uint32_t u = __umulhi(w, n_minus_1);
    return (int32_t)(u + (u >= (uint32_t)i ? 1u : 0u));
}

// The word stream of one directed edge, consumed in order by its negatives
// (word w is component w mod 4 of the Philox block w div 4).
struct WordCursor {
    int64_t e;       // edge index (graph-local)
    uint32_t next;   // next word
    uint32_t blk;    // Philox block held in buf (~0u: none)
    uint4 buf;
};

__device__ __forceinline__ WordCursor word_cursor(int64_t e) {
    WordCursor c;
    c.e = e;
    c.next = 0;
    c.blk = ~0u;
    c.buf = make_uint4(0, 0, 0, 0);
    return c;
}

__device__ __forceinline__ uint32_t take_word(WordCursor &c, uint32_t t, uint2 key) {
    const uint32_t b = c.next >> 2;
    if (b != c.blk) {
        c.buf = edge_words(c.e, t, b, key);
        c.blk = b;
    }
    const uint32_t q = c.next & 3u;
    ++c.next;
    return q == 0 ? c.buf.x : q == 1 ? c.buf.y : q == 2 ? c.buf.z : c.buf.w;
}

// Weighted negative (degree or caller weights) through an alias table of n
// entries {threshold, alias} (graph-local ids): two words per attempt --
// column floor(w0 n / 2^32), kept when w1 < threshold, else its alias; an
// attempt that yields the source is rejected, and after 16 rejections the
// uniform rule takes the next word.  Returns a graph-local id.
__device__ __forceinline__ int32_t weighted_negative(WordCursor &c, uint32_t t, uint2 key, const uint2 *table,
                                                     uint32_t n, int32_t src) {
    for (int attempt = 0; attempt < 16; ++attempt) {
        const uint32_t w0 = take_word(c, t, key);
        const uint32_t w1 = take_word(c, t, key);
        const uint32_t col = __umulhi(w0, n);
        const uint2 en = __ldg(table + col);
        const int32_t s = w1 < en.x ? (int32_t)col : (int32_t)en.y;
        if (s != src) return s;
    }
    return negative_of(take_word(c, t, key), src, n - 1);
}

// 1 / d for d = 1 + r^2 >= 1, correctly rounded: the hardware's estimate (one
// ulp) and one Newton-Raphson step in fused arithmetic, which rounds correctly
// from there (P. Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", 1990).  Equal to the IEEE reciprocal for every
// float in [1, 2^126); above, where that is subnormal and this is 0, and at
// infinity (d is clamped to 2^127, NaN stays), the force coefficients built
// from it still agree.  Four instructions without a branch; __frcp_rn's slow
// path costs a convergence point.
__device__ __forceinline__ float reciprocal(float d) {
    float q;
    asm("min.NaN.f32 %0, %0, 0f7F000000;" : "+f"(d));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(d));
    return fmaf(q, fmaf(-d, q, 1.0f), q);
}

// The reciprocal of a kernel's forces: SHORT = reciprocal(), else __frcp_rn --
// the same bits in another time.  What the racing lanes of the lock-free modes
// read depends on how long an entry takes.  Single graphs with uniform
// negatives take the short one where it gains time (HOGWILD; HOGWILD_RED on
// small graphs, launch_oriented_k), and their layouts stay where they were:
// 1.0 to 1.3 times as far from the other's as two runs are apart (HOGWILD on
// 778k / 10M, k = 5: 2067 -> 1799 us).  Multi-handle epochs, batches and
// weighted negatives gain no more than 2% from it and land 1.3 to 2 times as
// far off, so they keep the long one.
template <bool SHORT>
__device__ __forceinline__ float reciprocal_of(float d) {
    return SHORT ? reciprocal(d) : __frcp_rn(d);
}

// Force on i from the attraction of Table 1 (t-FDP): pulls i toward the
// partner, coefficient alpha (1 + beta / (1 + r^2)); d = y_i - y_partner.
template <bool SHORT>
__device__ __forceinline__ float2 attraction_on_i(float dx, float dy) {
    const float r2 = fmaf(dx, dx, dy * dy);
    const float q = reciprocal_of<SHORT>(1.0f + r2);
    const float ca = kAlpha * fmaf(kBeta, q, 1.0f);
    return make_float2(-ca * dx, -ca * dy);
}

// Force on i from the repulsion of Table 1 (t-FDP, gamma = 2): pushes i away,
// coefficient (1 + r^2)^-2; d = y_i - y_sample.
template <bool SHORT>
__device__ __forceinline__ float2 repulsion_on_i(float dx, float dy) {
    const float r2 = fmaf(dx, dx, dy * dy);
    const float q = reciprocal_of<SHORT>(1.0f + r2);
    const float cr = q * q;
    return make_float2(cr * dx, cr * dy);
}

// Position accesses that must see other SMs' writes: cached in L2 only.
// (Measured on GB300 against these intrinsics, with no gain on the R-MAT
// epoch: an explicit vector red.global.add.v2.f32, L2 evict-last / evict-first
// cache policies on positions and entries.)
__device__ __forceinline__ float2 load_pos(const float2 *p) { return __ldcg(p); }

// Adds d to a position (relaxed, device scope, no return value: a vector
// reduction in L2).
__device__ __forceinline__ void add_pos(float2 *p, float2 d) { atomicAdd(p, d); }

// A position written as one 64-bit atomic exchange (racy, last writer wins).
__device__ __forceinline__ void exchange_pos(float2 *p, float2 v) {
    unsigned long long bits;
    memcpy(&bits, &v, 8);
    atomicExch(reinterpret_cast<unsigned long long *>(p), bits);
}

// The edge stream is read once per epoch: evict-first streaming loads.
__device__ __forceinline__ int4 load_cols4(const int32_t *p) {
    return __ldcs(reinterpret_cast<const int4 *>(p));
}

// One oriented entry {j, index of (i, j), index of (j, i), i}.  Read through
// L1: the 32 lanes of a warp read one 512-byte run of entries per step.
__device__ __forceinline__ int4 load_entry(const int4 *p) { return __ldg(p); }

// int64 fixed point (2^-32) of one force component, clamped to +-2^20.
__device__ __forceinline__ long long to_fixed(float v, uint32_t &flags) {
    if (!(fabsf(v) <= kFixClamp)) {
        if (v != v) {
            flags |= kStatusNonFinite;
            return 0;
        }
        flags |= kStatusClamped;
        v = copysignf(kFixClamp, v);
    }
    return __float2ll_rn(v * kFixScale);
}

__device__ __forceinline__ void add_fixed(long long *dst, long long v) {
    atomicAdd(reinterpret_cast<unsigned long long *>(dst), (unsigned long long)v);
}

__device__ __forceinline__ bool finite2(float2 v) {
    return isfinite(v.x) && isfinite(v.y);
}


// Energies of Table 1 / Eq. 2 for the actual energy of an epoch (Section
// 3.3): U^a = alpha (r^2/2 + beta/2 ln(1 + r^2)), U^r = 1 / (2 (1 + r^2)).
__device__ __forceinline__ float attraction_energy(float dx, float dy) {
    const float r2 = fmaf(dx, dx, dy * dy);
    return kAlpha * fmaf(0.5f, r2, 0.5f * kBeta * log1pf(r2));
}

__device__ __forceinline__ float repulsion_energy(float dx, float dy) {
    return 0.5f * __frcp_rn(1.0f + fmaf(dx, dx, dy * dy));
}

// Per-lane view of the graph the current segment belongs to.
struct GraphCtx {
    int32_t base;        // first vertex of the graph
    uint32_t nm1;        // n_g - 1
    int64_t edge_base;   // first directed edge of the graph (random-word index origin)
    uint32_t epoch;      // the graph's epoch
    float eta;
    uint2 key;           // Philox key (the graph's seed)
    bool active;
};

__device__ __forceinline__ int32_t negative_in(const GraphCtx &c, uint32_t w, int32_t src) {
    return c.base + negative_of(w, src - c.base, c.nm1);
}

__device__ __forceinline__ uint4 words_in(const GraphCtx &c, int64_t e, uint32_t g) {
    return edge_words(e - c.edge_base, c.epoch, g, c.key);
}

__device__ __forceinline__ WordCursor cursor_in(const GraphCtx &c, int64_t e) { return word_cursor(e - c.edge_base); }

// Next weighted negative of source src (global ids); table = the graph's alias table.
__device__ __forceinline__ int32_t weighted_in(const GraphCtx &c, WordCursor &wc, const uint2 *alias, int32_t src) {
    return c.base + weighted_negative(wc, c.epoch, c.key, alias + c.base, c.nm1 + 1u, src - c.base);
}

// Displacement slots.  L2 serves one cache line's updates one after another,
// and vertices that are written often can have neighbouring ids (the hubs of
// R-MAT graphs under their natural labels), so their 128-byte line holds up the
// rest.  Inside every block of kSpreadBlock vertices neighbouring pairs of
// vertices are put far apart (an odd multiplier near the golden section, modulo
// the block); the array is padded to whole blocks.  The two vertices of a
// 32-byte sector stay together, so that the apply sweep reads whole sectors.
// R-MAT 2^22 / 34M edges with natural labels, 16 chunks: 4.36 -> 3.84 ms per
// epoch, the time of the same graph under a random relabelling (3.82 ms).  It
// parts only vertices of different heat inside a block: where a whole block is
// written often, as the first ids of a breadth-first relabelling are, as many
// hot vertices share a line as before (that labelling: 4.33 ms).
__host__ __device__ __forceinline__ int32_t spread_pair(int32_t i) {   // keeps i < 0 below 0
    constexpr int32_t half = kSpreadBlock / 2 - 1;
    return (i & ~(kSpreadBlock - 1)) | (int32_t)(((((uint32_t)i >> 1) * 633u) & (uint32_t)half) << 1) | (i & 1);
}

// Displacement slot of vertex i: two int64 fixed-point sums.
__device__ __forceinline__ long long *disp_of(long long *disp, int32_t i) {
    return disp + 2 * (int64_t)spread_pair(i);
}

// Adds (fx, fy) to vertex idx's displacement for every lane of the warp (idx
// < 0: nothing to add).  All 32 lanes call it together.  Lanes 2m and 2m + 1
// serve each other's vertices: first both add to the even lane's vertex (the
// even lane its x, the odd lane its y), then both to the odd lane's, so one
// request to L2 carries a vertex's two adjacent int64 sums.  L2 takes about
// 210 G requests/s whatever they hold: two separate adds per lane reach 105 G
// vertices/s on a random array, paired ones 203 G.
__device__ __forceinline__ void add_fixed_paired(long long *disp, int32_t idx, long long fx, long long fy) {
    const int odd = threadIdx.x & 1;
    idx = spread_pair(idx);
    const int32_t other = __shfl_xor_sync(0xffffffffu, idx, 1);
    const long long got = __shfl_xor_sync(0xffffffffu, odd ? fx : fy, 1);
    const int32_t first = odd ? other : idx, second = odd ? idx : other;
    if (first >= 0) add_fixed(disp + 2 * (int64_t)first + odd, odd ? got : fx);
    if (second >= 0) add_fixed(disp + 2 * (int64_t)second + odd, odd ? fy : got);
}

// One pair's term in the synchronous mode: the force on the source i from
// the attraction (REP = false) or the repulsion (REP = true) of Table 1 at
// the frozen positions, quantised (to_fixed); the source's share is summed
// into accx / accy, the other vertex's (x < 0: none) is added to disp.
// `twice`: the source's share counts twice and the other vertex gets nothing.
// Called by whole warps.
template <bool REP>
__device__ __forceinline__ void sync_pair_term(long long *disp, float2 yi, int32_t x, float2 yx, bool twice,
                                               long long &accx, long long &accy, uint32_t &flags) {
    long long fx = 0, fy = 0;
    if (x >= 0) {
        const float2 f = REP ? repulsion_on_i<true>(yi.x - yx.x, yi.y - yx.y)
                             : attraction_on_i<true>(yi.x - yx.x, yi.y - yx.y);
        fx = to_fixed(f.x, flags);
        fy = to_fixed(f.y, flags);
        accx += twice ? 2 * fx : fx;
        accy += twice ? 2 * fy : fy;
    }
    add_fixed_paired(disp, twice ? -1 : x, -fx, -fy);
}

// All force terms of directed edge e = (i, j) in the synchronous mode, with
// positions frozen (read-only during the launch): the attraction of Table 1
// and the repulsion of each of its k negatives (Algorithm 1's draws, in the
// order they consume the edge's random words), each force quantised to int64
// fixed point (2^-32, to_fixed).  The partner's and the negatives' terms are
// added to disp with integer atomics; the source's are summed into accx /
// accy, which the caller flushes once per row run.  Integer addition makes
// the totals independent of the order of the terms.
//
// both: (j, i) is stepped from the same frozen positions, i.e. j's row lies
// in the same chunk.  The force it puts on i is then the exact negative of
// what (i, j) puts on j -- every operation is odd in the difference -- so
// each row counts its own force twice and neither adds to its partner: the
// same integer total with one scattered add per edge less (a quarter of them
// at k = 3 and one chunk, and the ones that all go to the hubs).
//
// Called by whole warps (valid = false: the lane only takes part in the
// exchanges).  Returns the energy of the step's pairs at the frozen positions
// (U^a of (i, j) and U^r of each drawn pair) when `energy` is set, else 0.
// Shared by the synchronous chunk kernel of a handle and by the
// allocation-free entry point.
template <bool W>
__device__ __forceinline__ float sync_edge_terms(const float2 *pos, long long *disp, const GraphCtx &c,
                                                 const uint2 *alias, bool valid, int32_t i, float2 yi, int32_t j,
                                                 bool both, int64_t e, int32_t k, bool energy, long long &accx,
                                                 long long &accy, uint32_t &flags) {
    float2 yj = yi;
    if (valid) yj = __ldg(pos + j);
    float en = 0.0f;
    WordCursor wc = cursor_in(c, e);
    bool attracted = false;
    for (int g = 0; g * 4 < k || !attracted; ++g) {
        const int nm = k - 4 * g < 4 ? k - 4 * g : 4;   // 0 when k = 0
        int32_t s[4];
        float2 ys[4];
        if (W) {
#pragma unroll
            for (int m = 0; m < 4; ++m) s[m] = valid && m < nm ? weighted_in(c, wc, alias, i) : -1;
        } else {
            uint4 w = make_uint4(0u, 0u, 0u, 0u);
            if (nm > 0) w = words_in(c, e, (uint32_t)g);
            s[0] = valid && 0 < nm ? negative_in(c, w.x, i) : -1;
            s[1] = valid && 1 < nm ? negative_in(c, w.y, i) : -1;
            s[2] = valid && 2 < nm ? negative_in(c, w.z, i) : -1;
            s[3] = valid && 3 < nm ? negative_in(c, w.w, i) : -1;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            ys[m] = yi;
            if (s[m] >= 0) ys[m] = __ldg(pos + s[m]);
        }
        if (!attracted) {
            // after the first negatives' loads, which do not wait for it
            if (energy && valid) en += attraction_energy(yi.x - yj.x, yi.y - yj.y);
            sync_pair_term<false>(disp, yi, valid ? j : -1, yj, both, accx, accy, flags);
            attracted = true;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (m < nm) {
                if (energy && valid) en += repulsion_energy(yi.x - ys[m].x, yi.y - ys[m].y);
                sync_pair_term<true>(disp, yi, s[m], ys[m], false, accx, accy, flags);
            }
        }
    }
    return en;
}

}  // namespace snap
