// np_kernels.cu -- neighbourhood preservation on the device (Section 4.1,
// "Metrics": NP with r = 2), for the autotuner's quality gate and the
// library's own quality report.
//
// For a sampled vertex i of a graph with vertices [lo, lo + len):
//   N_G(i) = the vertices within two hops of i, i excluded; k = |N_G(i)|;
//   N_L(i) = the k vertices of the same graph nearest to i in the layout, i
//            excluded, ordered by squared distance and then by smaller id;
//   NP_i   = |N_G(i) & N_L(i)| / |N_G(i) | N_L(i)| (a Jaccard index); vertices
//            with k = 0 are skipped.
// Squared distances are formed in FP64 from the FP32 positions,
// (x_i - x_v)^2 + (y_i - y_v)^2 with every operation rounded on its own, so
// the ranking equals that of an FP64 evaluation of the same positions.
//
// One block per sample.  N_G(i) is a bitmap over the graph (in shared memory
// for graphs of up to 2^18 vertices, else a global scratch row of the block's
// own); a warp marks each neighbour's row (so a hub's row is read by 32 lanes).
//
// The k-th nearest (squared distance, then id) is found exactly with one pass
// over the positions in FP32: FP64 runs at about a sixtieth of the FP32 rate
// here.  The FP32 distance is within kRel of the FP64 one, so a bracket
// [lo, hi] around the k-th distance, taken from a sorted sample of the
// vertices, splits them into surely nearer, surely farther and a few percent
// of candidates; the candidates' FP64 keys go to a list, an exact
// most-significant-digit radix select over it gives the threshold, and the
// members of N_G are compared with that.  The bracket is checked afterwards:
// the threshold must lie inside it by more than the FP32 error, else (and when
// too many vertices tie) the select runs over the FP64 distances of all
// vertices (select_over_all).  A candidate list that overflows is narrowed and the
// pass repeated.
//
// Bound by the pass (8 bytes a vertex and sample from L2, about a dozen FP32
// instructions) and, on power-law graphs, by the sample with the largest 2-hop
// set.  Power-law graph of 1M vertices / 8M edges, 256 samples: 8.16 -> 0.44
// ms against thirteen FP64 passes (two, above 2^18 vertices); planted, 200k
// vertices, 256 samples: 9.7 -> 0.23 ms; R-MAT 2^22, 1,024 samples: 462 -> 14
// ms.  Eight positions of a thread under way: 0.63 -> 0.44 ms on the first.
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include "snap_internal.h"

namespace snap {
namespace {

constexpr int kNpThreads = 512;
constexpr int kSample = 4096;    // sampled distances held in shared memory
constexpr int kLongRow = 1024;   // a row marked by the whole block
constexpr int kSample2 = 12 * kSample;   // vertices sampled to narrow the first bracket
// FP32 against FP64 squared distance: two differences, a product and a fused
// product-sum, each within 2^-24: below 2.5e-7 relative; underflow adds less
// than kAbs.  Coordinates beyond about 1.8e19 apart overflow to infinity:
// such a vertex is a candidate of every bracket without an upper end, and a
// member whose FP64 key decides.
constexpr double kRel = 1e-6, kAbs = 1e-37;

__device__ __forceinline__ uint64_t dist_key(float2 a, float2 b) {
    const double dx = __dsub_rn((double)a.x, (double)b.x);
    const double dy = __dsub_rn((double)a.y, (double)b.y);
    return (uint64_t)__double_as_longlong(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}

__device__ __forceinline__ float dist32(float2 a, float2 b) {
    const float dx = a.x - b.x, dy = a.y - b.y;
    return fmaf(dx, dx, dy * dy);
}

// Shared state of one block.
struct NpShared {
    uint32_t value[kSample];   // sampled FP32 distances (bit patterns order like the values)
    uint32_t hist[256];
    uint32_t part[kNpThreads / 32];
    uint32_t total, rank, bin, ties, count;
    unsigned long long prefix, lowest, highest;
    float lo, hi;
};

// Sum of v over the block, on every thread.
__device__ uint32_t block_total(uint32_t v, NpShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) sh.part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < kNpThreads / 32 ? sh.part[lane] : 0u;
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) sh.total = v;
    }
    __syncthreads();
    v = sh.total;
    __syncthreads();
    return v;
}

// Ascending bitonic sort of sh.value.
__device__ void sort_values(NpShared &sh) {
    for (int size = 2; size <= kSample; size <<= 1) {
        for (int half = size >> 1; half > 0; half >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < kSample / 2; t += kNpThreads) {
                const int a = ((t & ~(half - 1)) << 1) | (t & (half - 1)), b = a | half;
                const uint32_t x = sh.value[a], y = sh.value[b];
                if ((x > y) == ((a & size) == 0)) {
                    sh.value[a] = y;
                    sh.value[b] = x;
                }
            }
        }
    }
    __syncthreads();
}

// One digit of the select: the bin of sh.hist that holds the sh.rank-th item
// (1-based); sh.rank becomes its rank inside the bin, sh.ties the bin's size.
__device__ void pick_digit(NpShared &sh) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        uint32_t h[8], sum = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            h[q] = sh.hist[8 * lane + q];
            sum += h[q];
        }
        uint32_t upto = sum;   // inclusive over the lanes
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += x;
        }
        const uint32_t rank = sh.rank;
        __syncwarp();
        uint32_t before = upto - sum;
        if (rank > before && rank <= upto) {
            for (int q = 0; q < 8; ++q) {
                if (rank <= before + h[q]) {
                    sh.bin = 8u * lane + q;
                    sh.rank = rank - before;
                    sh.ties = h[q];
                    break;
                }
                before += h[q];
            }
        }
    }
    __syncthreads();
}

// The rank-th smallest (key, id) among the items each() visits (each thread
// calls f(key, id) for its share): *dstar, *idstar on every thread.  The keys
// agree above bit `top` (63 when nothing is known).
template <typename Each>
__device__ void radix_select(Each each, uint32_t rank, unsigned long long agreed, int top, NpShared &sh,
                             uint64_t &dstar, uint32_t &idstar) {
    if (threadIdx.x == 0) {
        sh.rank = rank;
        sh.prefix = agreed;   // the bits above `top`
        sh.ties = 0;
    }
    __syncthreads();
    for (int shift = top & ~7; shift >= 0; shift -= 8) {
        for (int b = threadIdx.x; b < 256; b += kNpThreads) sh.hist[b] = 0u;
        __syncthreads();
        const uint64_t prefix = sh.prefix;
        each([&](uint64_t key, uint32_t) {
            if (shift == 56 || (key >> (shift + 8)) == (prefix >> (shift + 8)))
                atomicAdd(&sh.hist[(key >> shift) & 255u], 1u);
        });
        pick_digit(sh);
        if (threadIdx.x == 0) sh.prefix = prefix | ((uint64_t)sh.bin << shift);
        __syncthreads();
    }
    dstar = sh.prefix;
    if (sh.rank == sh.ties) {   // all items at this distance are taken
        idstar = 0xffffffffu;
        __syncthreads();
        return;
    }
    __syncthreads();   // every thread holds dstar before the prefix is reused
    if (threadIdx.x == 0) sh.prefix = 0ull;
    __syncthreads();
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = threadIdx.x; b < 256; b += kNpThreads) sh.hist[b] = 0u;
        __syncthreads();
        const uint32_t prefix = (uint32_t)sh.prefix;
        each([&](uint64_t key, uint32_t id) {
            if (key != dstar) return;
            if (shift == 24 || (id >> (shift + 8)) == (prefix >> (shift + 8)))
                atomicAdd(&sh.hist[(id >> shift) & 255u], 1u);
        });
        pick_digit(sh);
        if (threadIdx.x == 0) sh.prefix = prefix | (sh.bin << shift);
        __syncthreads();
    }
    idstar = (uint32_t)sh.prefix;
    __syncthreads();
}

// N_G(i) as a bitmap over [lo, lo + len) (cleared first), i excluded; returns
// k = |N_G(i)| on every thread.
__device__ uint32_t two_hop_bitmap(const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col_idx,
                                   int32_t i, int32_t lo, int32_t len, uint32_t *bits, NpShared &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t words = (len + 31) >> 5;
    for (int32_t w = threadIdx.x; w < words; w += kNpThreads) bits[w] = 0u;
    __syncthreads();
    // neighbours and their neighbours: a warp reads the bounds of 32 rows at
    // once and marks row after row, the whole block a long row (sh.value lists
    // them); four loads of a thread are under way at a time
    auto mark = [&](int32_t v) { atomicOr(&bits[(v - lo) >> 5], 1u << ((v - lo) & 31)); };
    auto mark_row = [&](int64_t f, int64_t f1, int32_t stride) {
        for (; f + 3 * (int64_t)stride < f1; f += 4 * (int64_t)stride) {
            const int32_t a = col_idx[f], b = col_idx[f + stride];
            const int32_t c = col_idx[f + 2 * (int64_t)stride], d = col_idx[f + 3 * (int64_t)stride];
            mark(a);
            mark(b);
            mark(c);
            mark(d);
        }
        for (; f < f1; f += stride) mark(col_idx[f]);
    };
    if (threadIdx.x == 0) sh.count = 0;
    __syncthreads();
    const int64_t b0 = row_ptr[i], b1 = row_ptr[i + 1];
    for (int64_t e = b0 + 32 * warp; e < b1; e += kNpThreads) {
        int32_t u = 0;
        int64_t f0 = 0, f1 = 0;
        bool inline_row = e + lane < b1;
        if (inline_row) {
            u = col_idx[e + lane];
            f0 = row_ptr[u];
            f1 = row_ptr[u + 1];
            mark(u);
            if (f1 - f0 > kLongRow) {
                const uint32_t at = atomicAdd(&sh.count, 1u);
                if (at < kSample) {
                    sh.value[at] = (uint32_t)u;
                    inline_row = false;
                }
            }
        }
        uint32_t rows = __ballot_sync(0xffffffffu, inline_row);
        while (rows) {
            const int t = __ffs(rows) - 1;
            rows &= rows - 1;
            const int64_t g0 = __shfl_sync(0xffffffffu, f0, t), g1 = __shfl_sync(0xffffffffu, f1, t);
            mark_row(g0 + lane, g1, 32);
        }
    }
    __syncthreads();
    const uint32_t longs = sh.count < kSample ? sh.count : kSample;
    for (uint32_t t = 0; t < longs; ++t) {
        const int32_t u = (int32_t)sh.value[t];
        mark_row(row_ptr[u] + threadIdx.x, row_ptr[u + 1], kNpThreads);
    }
    __syncthreads();
    if (threadIdx.x == 0) bits[(i - lo) >> 5] &= ~(1u << ((i - lo) & 31));
    __syncthreads();
    uint32_t kl = 0;
    for (int32_t w = threadIdx.x; w < words; w += kNpThreads) kl += __popc(bits[w]);
    return block_total(kl, sh);
}

// The graph of vertex i: [lo, lo + len).
__device__ __forceinline__ void graph_of(int32_t i, const int32_t *node_graph, const GraphInfo *graphs, int32_t n,
                                         int32_t &lo, int32_t &len) {
    lo = 0;
    len = n;
    if (graphs) {
        const GraphInfo gi = graphs[node_graph[i]];
        lo = gi.node_base;
        len = gi.n;
    }
}

// Members of the bitmap (k of them) at or before (dstar, idstar): |N_G & N_L|.
__device__ uint32_t members_within(const float2 *__restrict__ pos, const uint32_t *bits, float2 yi, int32_t lo,
                                   int32_t len, uint32_t k, uint64_t dstar, uint32_t idstar, NpShared &sh) {
    const double d = __longlong_as_double((long long)dstar);
    const double nearer = d * (1.0 - kRel) - kAbs, farther = d * (1.0 + kRel) + kAbs;
    auto within = [&](int32_t v) -> uint32_t {
        const float2 yv = pos[v];
        const double near32 = (double)dist32(yi, yv);
        if (near32 < nearer) return 1u;
        if (near32 > farther && near32 <= (double)FLT_MAX) return 0u;   // an overflow says nothing
        const uint64_t key = dist_key(yi, yv);
        return key < dstar || (key == dstar && (uint32_t)v <= idstar);
    };
    uint32_t inter = 0;
    if (k > (uint32_t)len / 16u) {   // many members: vertex by vertex, coalesced
#pragma unroll 4
        for (uint32_t x = threadIdx.x; x < (uint32_t)len; x += kNpThreads)
            if ((bits[x >> 5] >> (x & 31)) & 1u) inter += within(lo + (int32_t)x);
    } else {
        const int32_t words = (len + 31) >> 5;
        for (int32_t w = threadIdx.x; w < words; w += kNpThreads)
            for (uint32_t m = bits[w]; m; m &= m - 1) inter += within(lo + 32 * w + __ffs(m) - 1);
    }
    return block_total(inter, sh);
}

// The threshold from the FP64 distances of all vertices of [lo, lo + len)
// except i.
__device__ void select_over_all(const float2 *__restrict__ pos, int32_t i, int32_t lo, int32_t len, uint32_t k,
                                NpShared &sh, uint64_t &dstar, uint32_t &idstar) {
    const float2 yi = pos[i];
    auto all = [&](auto f) {
        for (int32_t v = lo + threadIdx.x; v < lo + len; v += kNpThreads)
            if (v != i) f(dist_key(yi, pos[v]), (uint32_t)v);
    };
    radix_select(all, k, 0ull, 63, sh, dstar, idstar);
}

// Sorted sample -> bracket: of `m` sampled vertices the `before` nearest lie
// below sh.lo and sh.value holds the next `held` in order; the vertex of
// share q of all has about rank q m among them, give or take four standard
// deviations.
__device__ __forceinline__ void bracket(NpShared &sh, double q, double m, double before, int held) {
    if (threadIdx.x == 0) {
        const double r = q * m - before, s = 4.0 * sqrt(m * q * (1.0 - q)) + 4.0;
        const double a = r - s, b = r + s;
        if (a >= 1.0 && a < (double)held) sh.lo = __uint_as_float(sh.value[(int)a - 1]);
        if (b < (double)held) sh.hi = __uint_as_float(sh.value[b < 0.0 ? 0 : (int)b]);
    }
    __syncthreads();
}

// Collects into sh.value the FP32 distances inside [sh.lo, sh.hi] of m
// vertices spread evenly over the graph, sorted; returns how many of the m lie
// below, and in `held` how many are held (more than kSample: not all are).
__device__ uint32_t sample_bracket(const float2 *__restrict__ pos, float2 yi, int32_t i, int32_t lo, int32_t len,
                                   int32_t m, NpShared &sh, uint32_t &held) {
    const float blo = sh.lo, bhi = sh.hi;
    for (int t = threadIdx.x; t < kSample; t += kNpThreads) sh.value[t] = 0xffffffffu;
    if (threadIdx.x == 0) sh.count = 0;
    __syncthreads();
    uint32_t below = 0;
    for (int32_t t = threadIdx.x; t < m; t += kNpThreads) {
        const int32_t v = lo + (int32_t)(((2 * (int64_t)t + 1) * len) / (2 * (int64_t)m));
        const float d = dist32(yi, pos[v]);
        if (v == i) continue;
        if (d < blo) {
            ++below;
        } else if (d <= bhi) {
            const uint32_t at = atomicAdd(&sh.count, 1u);
            if (at < kSample) sh.value[at] = __float_as_uint(d);
        }
    }
    below = block_total(below, sh);
    held = sh.count;
    if (held <= kSample) sort_values(sh);
    return below;
}

// NP of one sample: the threshold by the bracketed pass, or over all vertices
// where the bracket does not hold; NP_i on thread 0.
__device__ double np_of_sample(const float2 *__restrict__ pos, const uint32_t *bits, int32_t i, int32_t lo,
                               int32_t len, uint32_t k, uint64_t *ck, uint32_t *ci, uint32_t cap, NpShared &sh) {
    const float2 yi = pos[i];
    const double q = (double)k / (double)(len - 1);
    if (threadIdx.x == 0) {
        sh.lo = 0.0f;
        sh.hi = __int_as_float(0x7f800000);
    }
    __syncthreads();
    if ((uint32_t)len > cap) {
        uint32_t held;
        uint32_t before = sample_bracket(pos, yi, i, lo, len, kSample, sh, held);
        bracket(sh, q, kSample, before, (int)held);
        if (len > 2 * kSample2) {
            before = sample_bracket(pos, yi, i, lo, len, kSample2, sh, held);
            if (held <= kSample) bracket(sh, q, kSample2, before, (int)held);
        }
    }
    uint64_t dstar = 0;
    uint32_t idstar = 0;
    bool found = false;
    for (int round = 0; round < 4 && !found; ++round) {
        const float blo = sh.lo, bhi = sh.hi;
        __syncthreads();
        if (threadIdx.x == 0) {
            sh.count = 0;
            sh.lowest = ~0ull;
            sh.highest = 0ull;
        }
        __syncthreads();
        uint32_t below = 0;
        const int lane = threadIdx.x & 31;
        constexpr int kBatch = 8;   // positions a thread has under way
        for (uint32_t b = 0; b < (uint32_t)len; b += kBatch * kNpThreads) {
            float2 yv[kBatch];
#pragma unroll
            for (int m = 0; m < kBatch; ++m) {
                const uint32_t x = b + m * kNpThreads + threadIdx.x;
                yv[m] = x < (uint32_t)len ? pos[lo + (int32_t)x] : make_float2(NAN, NAN);
            }
#pragma unroll
            for (int m = 0; m < kBatch; ++m) {
                const int32_t v = lo + (int32_t)(b + m * kNpThreads + threadIdx.x);
                const float d = dist32(yi, yv[m]);   // NaN past the end: neither below nor a candidate
                const bool other = v != i;
                below += other && d < blo;
                const bool cand = other && d >= blo && d <= bhi;
                const uint32_t mask = __ballot_sync(0xffffffffu, cand);
                if (mask) {
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(&sh.count, (uint32_t)__popc(mask));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(mask & ((1u << lane) - 1u));
                    if (cand && at < cap) ci[at] = (uint32_t)v;
                }
            }
        }
        below = block_total(below, sh);
        const uint32_t ncand = sh.count;
        __syncthreads();
        if (k <= below || k - below > ncand) break;   // the bracket misses the rank
        const uint32_t rank = k - below;
        if (ncand > cap) {
            // too many: a sample of the bracket alone, with the exact rank inside it
            const double share = (double)ncand / (double)len;
            const double want = 0.7 * kSample / share;
            uint32_t held;
            sample_bracket(pos, yi, i, lo, len, (int32_t)(want < (double)len ? want : (double)len), sh, held);
            if (held > kSample || held == 0) break;
            bracket(sh, (double)rank / (double)ncand, (double)held, 0.0, (int)held);
            if (sh.lo == blo && sh.hi == bhi) break;   // ties: nothing to narrow
            continue;
        }
        // the candidates' FP64 keys, and the bits they agree in
        unsigned long long least = ~0ull, most = 0ull;
        for (uint32_t t = threadIdx.x; t < ncand; t += kNpThreads) {
            const unsigned long long key = dist_key(yi, pos[ci[t]]);
            ck[t] = key;
            least = key < least ? key : least;
            most = key > most ? key : most;
        }
        atomicMin(&sh.lowest, least);
        atomicMax(&sh.highest, most);
        __syncthreads();
        const unsigned long long differ = sh.lowest ^ sh.highest;
        const int top = differ ? 63 - __clzll((long long)differ) : 0;
        const int shift = top & ~7;
        const unsigned long long agreed = shift == 56 ? 0ull : (sh.lowest >> (shift + 8)) << (shift + 8);
        __syncthreads();
        auto cands = [&](auto f) {
            for (uint32_t t = threadIdx.x; t < ncand; t += kNpThreads) f(ck[t], ci[t]);
        };
        radix_select(cands, rank, agreed, top, sh, dstar, idstar);
        const double d = __longlong_as_double((long long)dstar);
        found = (blo == 0.0f || d > (double)blo * (1.0 + kRel) + kAbs) && d < (double)bhi * (1.0 - kRel) - kAbs;
        break;
    }
    if (!found) select_over_all(pos, i, lo, len, k, sh, dstar, idstar);
    const uint32_t total = members_within(pos, bits, yi, lo, len, k, dstar, idstar, sh);
    return (double)total / (double)(2u * k - total);
}

// gbits == null: the bitmap in dynamic shared memory.  Candidate keys and ids:
// `cap` of each per block.
__global__ void __launch_bounds__(kNpThreads) np_sample_kernel(const int64_t *__restrict__ row_ptr,
                                                               const int32_t *__restrict__ col_idx,
                                                               const float2 *__restrict__ pos,
                                                               const int32_t *__restrict__ nodes, int32_t count,
                                                               const int32_t *__restrict__ node_graph,
                                                               const GraphInfo *__restrict__ graphs, int32_t n,
                                                               double *__restrict__ out, uint32_t *gbits,
                                                               int64_t gbits_words, uint64_t *ckeys, uint32_t *cids,
                                                               uint32_t cap) {
    extern __shared__ uint32_t sbits[];
    __shared__ NpShared sh;
    uint32_t *bits = gbits ? gbits + (int64_t)blockIdx.x * gbits_words : sbits;
    uint64_t *ck = ckeys + (int64_t)blockIdx.x * cap;
    uint32_t *ci = cids + (int64_t)blockIdx.x * cap;
    for (int32_t q = blockIdx.x; q < count; q += gridDim.x) {
        const int32_t i = nodes[q];
        int32_t lo, len;
        graph_of(i, node_graph, graphs, n, lo, len);
        const uint32_t k = two_hop_bitmap(row_ptr, col_idx, i, lo, len, bits, sh);
        double np = -1.0;   // skipped
        if (k > 0) np = np_of_sample(pos, bits, i, lo, len, k, ck, ci, cap, sh);
        if (threadIdx.x == 0) out[q] = np;
        __syncthreads();
    }
}

}  // namespace

int np_blocks_per_sm(int32_t max_graph) {
    const size_t smem = max_graph > kNpMaxGraph ? 0 : sizeof(uint32_t) * (size_t)((max_graph + 31) / 32);
    int nb = 0;
    cudaFuncSetAttribute(np_sample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNpMaxGraph / 8);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, np_sample_kernel, kNpThreads, smem);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_np_samples(const int64_t *row_ptr, const int32_t *col_idx, const float2 *pos, const int32_t *nodes,
                              int32_t count, const int32_t *node_graph, const GraphInfo *graphs, int32_t n,
                              int32_t max_graph, double *out, int grid, const NpScratch &s, cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    const size_t smem = s.bits ? 0 : sizeof(uint32_t) * (size_t)((max_graph + 31) / 32);
    np_sample_kernel<<<grid, kNpThreads, smem, stream>>>(row_ptr, col_idx, pos, nodes, count, node_graph, graphs, n,
                                                         out, s.bits, s.bits_words, s.keys, s.ids, s.cap);
    return cudaGetLastError();
}

}  // namespace snap
