// graph_kernels.cu -- segment table, CSR validation and the objective of
// Eq. 4 (weight realised by uniform sampling, Section 3.3).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cub/device/device_scan.cuh>

#include "snap_device.cuh"
#include "snap_internal.h"

namespace snap {

namespace {

// seg_row[s] = the row holding edge s * seg_len: the largest r with
// row_ptr[r] <= e (then row_ptr[r+1] > e, so the row is not empty).
__global__ void segment_rows_kernel(const int64_t *__restrict__ row_ptr, int32_t n, int32_t seg_len,
                                    int32_t *__restrict__ seg_row, int64_t num_segs) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < num_segs; s += stride) {
        const int64_t e = s * seg_len;
        int32_t lo = 0, hi = n;   // invariant: row_ptr[lo] <= e < row_ptr[hi]
        while (hi - lo > 1) {
            const int32_t mid = lo + (hi - lo) / 2;
            if (row_ptr[mid] <= e)
                lo = mid;
            else
                hi = mid;
        }
        seg_row[s] = lo;
    }
}

// src[e] = the row of directed edge e.  Runs beside the validation, so row_ptr
// may be anything: rows stay below n.
__global__ void edge_sources_kernel(const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ seg_row,
                                    int32_t n, int64_t nnz, int32_t seg_len, int32_t *__restrict__ src) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q * 4 < nnz; q += stride) {
        int32_t row = seg_row[q * 4 / seg_len];   // seg_len is a multiple of 4
        int64_t row_end = row_ptr[row + 1];
        int32_t out[4] = {0, 0, 0, 0};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (q * 4 + t < nnz) {
                while (row_end <= q * 4 + t && row < n - 1) {
                    ++row;
                    row_end = row_ptr[row + 1];
                }
                out[t] = row;
            }
        }
        reinterpret_cast<int4 *>(src)[q] = make_int4(out[0], out[1], out[2], out[3]);
    }
}

// deg[i] = row_ptr[i+1] - row_ptr[i] (row_ptr checked non-decreasing by
// check_row_ptr_kernel before anything uses it as a rank).
__global__ void degrees_kernel(const int64_t *__restrict__ row_ptr, int32_t n, int32_t *__restrict__ deg) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        deg[i] = (int32_t)(row_ptr[i + 1] - row_ptr[i]);
}

// Orientation of the undirected edges: {i, j} belongs to the bundle of the
// endpoint that ranks higher by (degree, then smaller id).  That endpoint's
// lane processes both directed copies (i, j) and (j, i), so a vertex is a
// partner only of its higher-ranked neighbours.
__device__ __forceinline__ bool ranks_higher(int32_t di, int32_t dj, int32_t i, int32_t j) {
    return di > dj || (di == dj && i < j);
}

// row_ptr non-decreasing inside [0, nnz] (row_ptr[0] = 0 and row_ptr[n] =
// nnz are checked on the host).  Every kernel that runs before this result
// is read clamps the offsets it uses as indices.
__global__ void check_row_ptr_kernel(const int64_t *__restrict__ row_ptr, int32_t n, int64_t nnz,
                                     uint32_t *flags_out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t lo = row_ptr[i], hi = row_ptr[i + 1];
        if (lo < 0 || hi < lo || hi > nnz) bad = true;
    }
    if (bad) atomicOr(flags_out, kBadRowPtr);
}

// Columns in [0, n), no self-loop, rows strictly ascending, no edge across
// two graphs of a batch.  upper_count != null (the synchronous mode, which
// has no orientation pass): also symmetry, checked on half of the edges --
// every (i, j) with j < i must have (j, i) in row j (binary search), and the
// number of such edges must be nnz / 2 (the caller compares): reversal maps
// them one-to-one into the edges with j > i, so equal counts mean every edge
// has its reverse.  (The HOGWILD modes check symmetry the same way in the
// orientation pass, which searches the reverse of half of the edges anyway.)
// orient != null (the HOGWILD modes): also orient[e] = 1 when edge e's
// source ranks higher than its partner (ranks_higher; deg = row lengths),
// else 0, and orient[nnz] = 0 -- the input of the orientation scan.
//
// One thread per edge, so that a warp reads 32 consecutive columns at a time;
// its row is found from the segment table (a segment is at most a warp wide).
// LFR-shaped graph of 13.8M directed edges: 218 -> 108 us (a thread per
// 32-edge segment before).
__global__ void __launch_bounds__(256) validate_csr_kernel(const int64_t *__restrict__ row_ptr,
                                                           const int32_t *__restrict__ col_idx,
                                                           const int32_t *__restrict__ seg_row, int32_t n, int64_t nnz,
                                                           int32_t seg_len, uint32_t *flags_out,
                                                           const int32_t *__restrict__ node_graph,
                                                           unsigned long long *upper_count,
                                                           const int32_t *__restrict__ deg,
                                                           int32_t *__restrict__ orient) {
    if (orient && blockIdx.x == 0 && threadIdx.x == 0) orient[nnz] = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint32_t flags = 0;
    uint32_t upper = 0;   // at most nnz / threads + 1 of a thread's edges
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) {
        int32_t row = seg_row[e / seg_len];
        while (row < n - 1 && e >= row_ptr[row + 1]) ++row;
        const int32_t j = col_idx[e];
        if (j < 0 || j >= n) {
            flags |= kBadColumn;
            if (orient) orient[e] = 0;
            continue;
        }
        if (orient) orient[e] = ranks_higher(deg[row], deg[j], row, j) ? 1 : 0;
        if (j == row) flags |= kSelfLoop;
        if (node_graph && node_graph[j] != node_graph[row]) flags |= kCrossGraph;
        if (e > 0 && e > row_ptr[row] && col_idx[e - 1] >= j) flags |= kUnsorted;
        if (upper_count && j < row) {
            ++upper;
            // binary search for `row` in row j (offsets clamped to [0, nnz])
            int64_t lo = max(row_ptr[j], (int64_t)0), hi = min(row_ptr[j + 1], nnz);
            bool found = false;
            while (lo < hi) {
                const int64_t mid = lo + (hi - lo) / 2;
                const int32_t v = col_idx[mid];
                if (v == row) {
                    found = true;
                    break;
                }
                if (v < row)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            if (!found) flags |= kAsymmetric;
        }
    }
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (flags && (threadIdx.x & 31) == 0) atomicOr(flags_out, flags);
    if (upper_count) {
        upper = __reduce_add_sync(0xffffffffu, upper);
        if (upper && (threadIdx.x & 31) == 0) atomicAdd(upper_count, (unsigned long long)upper);
    }
}

// Entry of an oriented edge {i, j}: {j, index of (i, j), index of (j, i), i}
// -- the CSR indices of both directed copies (a handle holds fewer than 2^32
// directed edges) and the source, so an entry names its own row.
__device__ __forceinline__ int4 make_entry(int32_t i, int32_t j, int64_t fwd, int64_t rev) {
    return make_int4(j, (int32_t)(uint32_t)fwd, (int32_t)(uint32_t)rev, i);
}

// Order of the entries inside an oriented row of length L: the entry of
// rank q (ascending partner id) is stored at (a q) mod L, a the odd number
// nearest above 0.618 L that is coprime with L.  Consecutive stored entries
// -- the steps a lane runs back to back -- then belong to partners far apart
// in the row.  (Under a locality relabelling, partners with close ids are
// close in the graph; running them back to back pulls the source along one
// direction many times in a row.  Sequential FP64 emulation on R-MAT 2^22,
// 4-entry chunks: objective +1.5% / NP -2.0% against the shuffled order of
// Algorithm 1 in ascending order, +0.9% / -0.7% with the rows permuted.)
// (32-bit arithmetic: a row has fewer than 2^31 entries, and 64-bit
// remainders cost several times as much on the GPU.)
__device__ __forceinline__ uint32_t gcd_dev(uint32_t a, uint32_t b) {
    while (b) {
        const uint32_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

__device__ __forceinline__ int64_t row_multiplier(int32_t L) {
    uint32_t a = (uint32_t)(int64_t)(0.6180339887498949 * (double)L) | 1u;
    while (gcd_dev(a, (uint32_t)L) != 1u) a += 2u;
    return (int64_t)a;
}

__device__ __forceinline__ int32_t row_position(int32_t q, int32_t L) {
    if (L <= 2) return q;
    return (int32_t)((row_multiplier(L) * (int64_t)q) % L);
}

// Rank (ascending partner id) of the entry stored at offset o of a row of
// length L in the affine order: the inverse of row_position.
__device__ __forceinline__ int32_t row_rank(int32_t o, int32_t L) {
    if (L <= 2) return o;
    // inverse of a mod L by the extended Euclidean algorithm
    int64_t r0 = L, r1 = row_multiplier(L) % L, t0 = 0, t1 = 1;
    while (r1 != 0) {
        const int64_t qt = r0 / r1;
        int64_t tmp = r0 - qt * r1;
        r0 = r1;
        r1 = tmp;
        tmp = t0 - qt * t1;
        t0 = t1;
        t1 = tmp;
    }
    const int64_t inv = t0 < 0 ? t0 + L : t0;
    return (int32_t)((inv * (int64_t)o) % L);
}

// Per row, from the orientation scan: the row's place in the oriented list,
// the chunks of T entries it spans (0: empty row) and, in the affine order,
// its multiplier (row_multiplier, which searches).
__global__ void __launch_bounds__(256) oriented_rows_kernel(const int64_t *__restrict__ row_ptr,
                                                            const int32_t *__restrict__ pos, int32_t n, int32_t T,
                                                            int32_t order, int64_t *__restrict__ act_row_ptr,
                                                            int32_t *__restrict__ pieces,
                                                            int32_t *__restrict__ multiplier) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t b = pos[row_ptr[i]], e = pos[row_ptr[i + 1]];
        act_row_ptr[i] = b;
        if (i == n - 1) act_row_ptr[n] = e;
        pieces[i] = e > b ? (int32_t)((e - 1) / T - b / T + 1) : 0;
        const int32_t L = (int32_t)(e - b);
        multiplier[i] = order == 0 && L > 2 ? (int32_t)row_multiplier(L) : 1;
    }
}

// Builds the oriented list directly in its chunked, slot-interleaved layout
// `to` (both row orders), one thread per edge: owned edge e of row i (the
// orientation scan goes up at it) has rank r = pos[e] - pos[row_ptr[i]] among
// its row's owned edges (ascending partner id), sits at row position r
// (ascending order) or (a r) mod L (affine order, row_position), hence at list
// index pt = pos[row_ptr[i]] + that, in chunk pt / T; the entry is written to
// its slot's place and the chunk's first entry writes the slot descriptor
// {i, chunk}.
// Also the symmetry check of the HOGWILD modes: the reverse (j, i) of every
// owned edge must exist (else kAsymmetric), and the caller compares the
// number of owned edges with nnz / 2 -- reversal maps the owned edges one-to-
// one into the others (rows hold no duplicates), so equal counts mean every
// edge has its reverse.  Entries are written only for pt < capacity (the
// count is checked after the pass).
// Bound by the search for the reverse, log2 of the partner's degree random
// reads, and the scattered 16-byte writes: LFR-shaped graph of 13.8M directed
// edges 527 -> 289 us (a thread walked 32 edges, searches one after
// another, with the multiplier's search between them).
__global__ void __launch_bounds__(256) orient_scatter_kernel(const int64_t *__restrict__ row_ptr,
                                                             const int32_t *__restrict__ col_idx,
                                                             const int32_t *__restrict__ seg_row, int64_t nnz,
                                                             int32_t seg_len, const int32_t *__restrict__ pos,
                                                             const int64_t *__restrict__ act_row_ptr,
                                                             const int32_t *__restrict__ multiplier,
                                                             const ChunkLayout to, int4 *__restrict__ ent,
                                                             int2 *__restrict__ meta, int64_t capacity,
                                                             uint32_t *flags_out) {
    uint32_t flags = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) {
        const int32_t at = pos[e];
        if (pos[e + 1] == at) continue;   // the partner's row owns this edge
        int32_t i = seg_row[e / seg_len];
        while (e >= row_ptr[i + 1]) ++i;
        const int32_t j = col_idx[e];
        const int64_t start = act_row_ptr[i];
        const uint32_t L = (uint32_t)(act_row_ptr[i + 1] - start), r = (uint32_t)((int64_t)at - start);
        const uint32_t a = (uint32_t)multiplier[i];
        const uint32_t o = L < 65536u ? (a * r) % L : (uint32_t)(((uint64_t)a * r) % L);
        // index of the reverse copy (j, i): binary search for i in row j
        const int64_t re = row_ptr[j + 1];
        int64_t lo = row_ptr[j], hi = re - 1;
        while (lo < hi) {
            const int64_t mid = lo + (hi - lo) / 2;
            if (col_idx[mid] < i)
                lo = mid + 1;
            else
                hi = mid;
        }
        if (lo >= re || col_idx[lo] != i) {
            flags |= kAsymmetric;
            continue;
        }
        const int64_t pt = start + o;
        if (pt < 0 || pt >= capacity) continue;
        const int64_t c = pt / to.T;
        const int64_t t = pt - c * to.T;
        const int64_t slot = chunk_slot(to, c);
        ent[chunk_entry_index(slot, to.S, to.T, t)] = make_entry(i, j, e, lo);
        if (t == 0) meta[slot] = make_int2(i, (int32_t)c);
    }
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (flags && (threadIdx.x & 31) == 0) atomicOr(flags_out, flags);
}

// Chunks of T entries that each vertex's oriented row spans (0: empty row),
// when a list is cut anew.
__global__ void row_pieces_kernel(const int64_t *__restrict__ act_rp, int32_t n, int32_t T,
                                  int32_t *__restrict__ pieces) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t b = act_rp[v], e = act_rp[v + 1];
        pieces[v] = e > b ? (int32_t)((e - 1) / T - b / T + 1) : 0;
    }
}

// Chunk layout of the oriented list (the stored order is described with
// ChunkLayout).  One thread per entry p of the row-major list copies it from
// its place under `from` to its place under `to`; the thread of a chunk's
// first entry also writes the slot's {row, chunk}.
__global__ void chunk_layout_kernel(const int4 *__restrict__ src, const ChunkLayout from, int4 *__restrict__ dst,
                                    const ChunkLayout to, int2 *__restrict__ meta, const int64_t *__restrict__ act_rp,
                                    int32_t n, int64_t nnz) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride) {
        int64_t q = p;
        if (from.T > 0) {
            const int64_t c = p / from.T;
            q = chunk_entry_index(chunk_slot(from, c), from.S, from.T, p - c * from.T);
        }
        // p is the entry's row-major index in `from`'s row order; pt its index
        // in `to`'s (the same row, another place when the orders differ)
        const int4 en = src[q];
        int64_t pt = p;
        if (from.order != to.order) {
            const int32_t row = en.w;   // the entry names its row
            const int64_t b = act_rp[row];
            const int32_t L = (int32_t)(act_rp[row + 1] - b), o = (int32_t)(p - b);
            const int32_t rank = from.order == 0 ? row_rank(o, L) : o;
            pt = b + (to.order == 0 ? row_position(rank, L) : rank);
        }
        const int64_t c = pt / to.T;
        const int64_t t = pt - c * to.T;
        const int64_t slot = chunk_slot(to, c);
        dst[chunk_entry_index(slot, to.S, to.T, t)] = en;
        if (t == 0) meta[slot] = make_int2(en.w, (int32_t)c);
    }
}

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double warp_part[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warp_part[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        t = lane < nw ? warp_part[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;   // valid in thread 0
}

// U^a summed over undirected edges, each counted once (from its i < j copy).
// U^a(r) = alpha (r^2 / 2 + beta/2 ln(1 + r^2)), Eq. 2 with Table 1's attraction.
__global__ void objective_edges_kernel(const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col_idx,
                                       const int32_t *__restrict__ seg_row, const float2 *__restrict__ pos,
                                       int64_t nnz, int32_t seg_len, double *partial) {
    const int64_t num_segs = (nnz + seg_len - 1) / seg_len;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    double acc = 0.0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < num_segs; s += stride) {
        const int64_t e0 = s * seg_len;
        const int64_t e1 = min(e0 + (int64_t)seg_len, nnz);
        int32_t row = seg_row[s];
        int64_t row_end = row_ptr[row + 1];
        float2 yi = pos[row];
        float part = 0.0f;
        for (int64_t e = e0; e < e1; ++e) {
            if (e >= row_end) {
                do {
                    ++row;
                    row_end = row_ptr[row + 1];
                } while (row_end <= e);
                yi = pos[row];
            }
            const int32_t j = col_idx[e];
            if (row < j) {
                const float2 yj = pos[j];
                const float dx = yi.x - yj.x, dy = yi.y - yj.y;
                const float r2 = fmaf(dx, dx, dy * dy);
                part += kAlpha * (0.5f * r2 + 0.5f * kBeta * log1pf(r2));
            }
        }
        acc += (double)part;
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// U^a over an oriented list (each undirected edge once).  An entry names both
// endpoints, so a warp reads the 32 chunks of a slot group step by step, 512
// contiguous bytes each, and gathers two positions per entry; nothing else is
// looked up.  Each lane sums up to 32 entries of its chunk in FP32 (a chunk may
// hold 4096), those sums in FP64.  With 16M
// sampled pairs the objective of 2M vertices / 16M edges takes 353 us (973 us
// when this walked the row offsets and the samples came one by one).
__global__ void __launch_bounds__(256) objective_oriented_kernel(const int4 *__restrict__ ent, const ChunkLayout L,
                                                                 int64_t nnz, const float2 *__restrict__ pos,
                                                                 double *partial) {
    const int64_t groups = (L.S + 31) >> 5;
    const int64_t last_slot = chunk_slot(L, L.S - 1);
    const int32_t last_len = (int32_t)(nnz - (L.S - 1) * (int64_t)L.T);
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < groups; g += warps) {
        const int64_t slot = (g << 5) | lane;
        if (slot >= L.S) continue;
        const int64_t step = chunk_group_width(slot, L.S);
        const int32_t len = slot == last_slot ? last_len : L.T;
        const int4 *p = ent + chunk_entry_index(slot, L.S, L.T, 0);
        for (int32_t t0 = 0; t0 < len; t0 += 32) {
            const int32_t t1 = min(t0 + 32, len);
            float part = 0.0f;
#pragma unroll 4
            for (int32_t t = t0; t < t1; ++t) {
                const int4 e = p[t * step];
                const float2 yi = pos[e.w], yj = pos[e.x];
                const float dx = yi.x - yj.x, dy = yi.y - yj.y;
                const float r2 = fmaf(dx, dx, dy * dy);
                part += kAlpha * (0.5f * r2 + 0.5f * kBeta * log1pf(r2));
            }
            acc += (double)part;
        }
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// sum over ordered pairs i != j of (d_i + d_j) U^r(r_ij), U^r = 1 / (2 (1 + r^2)).
// The host halves it (unordered pairs) and applies k / (2 (n-1)).
constexpr int kPairTile = 256;
constexpr int32_t kWideRows = 14000;

// Pair coefficient of the objective: uniform negatives (d_i + d_j); weighted
// negatives c_ij = d_i P(j|i) + d_j P(i|j) = x_i z_j + y_i + x_j z_i + y_j from
// the per-vertex factors {x, y, z} (Section 3.3's derivation with P(s|i)).
__device__ __forceinline__ float pair_coef(float di, float dj, const float4 &wi, const float4 &wj, bool weighted) {
    return weighted ? fmaf(wi.x, wj.z, wi.y) + fmaf(wj.x, wi.z, wj.y) : di + dj;
}

// Work items: a tile of kPairTile * R rows (R per thread, in registers)
// against kPairTile columns in shared memory, for the column tiles from the
// rows' own on: U^r is symmetric, so pairs above the diagonal tiles count
// twice, and the diagonal tiles hold both orders of theirs.  Item `it` of the
// triangle belongs to row tile I when first_item(I) <= it < first_item(I + 1).
// Each row's 256 terms of an item are summed in FP32, then in FP64.
// Bound by issue: about eleven instructions a pair (the reciprocal unit, an
// eighth of the FP32 rate, is close behind).  The whole exact objective of
// 16,000 vertices / 120k edges takes 98 us, of which about 42 are launches and
// the copy back (1,138 us with every ordered pair, a thread a row and 63
// blocks); 24,000 vertices 147 us (1,676 us).
template <bool WT, int R>
__global__ void __launch_bounds__(kPairTile) objective_pairs_exact_kernel(const float2 *__restrict__ pos,
                                                                          const int32_t *__restrict__ deg,
                                                                          const float4 *__restrict__ wt,
                                                                          int32_t n, double *partial) {
    __shared__ float4 tile[kPairTile];           // x, y, degree
    __shared__ float4 tw[WT ? kPairTile : 1];
    const int64_t cols = ((int64_t)n + kPairTile - 1) / kPairTile, rows = (cols + R - 1) / R;
    auto first_item = [&](int64_t I) { return I * cols - R * (I * (I - 1) / 2); };   // sum of cols - R J for J < I
    const int64_t items = first_item(rows);
    double acc = 0.0;
    int64_t I = 0;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        while (it >= first_item(I + 1)) ++I;   // items ascend, so does I
        const int64_t J = I * R + (it - first_item(I));
        const int64_t jb = J * kPairTile, ib = I * R * kPairTile;
        __syncthreads();
        const int64_t jl = jb + threadIdx.x;
        float2 yj = make_float2(0.f, 0.f);
        if (jl < n) yj = pos[jl];
        tile[threadIdx.x] = make_float4(yj.x, yj.y, jl < n ? (float)deg[jl] : 0.f, 0.f);
        if (WT) tw[threadIdx.x] = jl < n ? wt[jl] : make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        float2 yi[R];
        float di[R], part[R];
        float4 wi[R];
        int self[R];   // this row's column in the tile (none: -1)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = ib + r * kPairTile + threadIdx.x;
            yi[r] = i < n ? pos[i] : make_float2(0.f, 0.f);
            di[r] = i < n ? (float)deg[i] : 0.f;
            wi[r] = (WT && i < n) ? wt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            part[r] = 0.f;
            self[r] = J == I * R + r ? (int)threadIdx.x : -1;
        }
        const int cnt = (int)min((int64_t)kPairTile, n - jb);
        auto column = [&](int q, bool diagonal) {
            const float4 t = tile[q];
            const float4 wj = tw[WT ? q : 0];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float dx = yi[r].x - t.x, dy = yi[r].y - t.y;
                const float u = reciprocal(fmaf(dx, dx, fmaf(dy, dy, 1.0f)));
                const float c = pair_coef(di[r], t.z, wi[r], wj, WT);
                if (diagonal)
                    part[r] = q == self[r] ? part[r] : fmaf(c, u, part[r]);
                else
                    part[r] = fmaf(c, u, part[r]);
            }
        };
        const bool diagonal = J < (I + 1) * R;
        if (diagonal) {
            for (int q = 0; q < cnt; ++q) column(q, true);
        } else {
#pragma unroll 4
            for (int q = 0; q < cnt; ++q) column(q, false);
        }
        double sum = 0.0;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (ib + r * kPairTile + threadIdx.x < n) sum += (double)part[r];
        acc += diagonal ? 0.5 * sum : sum;   // 0.5: U^r = u / 2, and twice that above the diagonal tiles
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// Batch: per vertex i, the sum over j != i of its graph of w_ij U^r(r_ij),
// w_ij = (d_i + d_j) / (2 (n_g - 1)) for uniform negatives or c_ij / 2 for
// weighted ones; one thread per vertex, the graph's vertices in turn.
__global__ void objective_pairs_batch_kernel(const float2 *__restrict__ pos, const int32_t *__restrict__ deg,
                                             const float4 *__restrict__ wt, const int32_t *__restrict__ node_graph,
                                             const GraphInfo *__restrict__ graphs, int32_t n, double *partial) {
    double acc = 0.0;
    const bool weighted = wt != nullptr;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const GraphInfo gi = graphs[node_graph[i]];
        if (gi.n < 2) continue;
        const float2 yi = pos[i];
        const float di = (float)deg[i];
        const float4 wi = weighted ? wt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        double sum = 0.0;
        float part = 0.0f;
        int cnt = 0;
        for (int32_t j = gi.node_base; j < gi.node_base + gi.n; ++j) {
            if (j == i) continue;
            const float2 yj = pos[j];
            const float dx = yi.x - yj.x, dy = yi.y - yj.y;
            const float r2 = fmaf(dx, dx, dy * dy);
            const float4 wj = weighted ? wt[j] : make_float4(0.f, 0.f, 0.f, 0.f);
            part += pair_coef(di, (float)deg[j], wi, wj, weighted) * (0.5f * reciprocal(1.0f + r2));
            if (++cnt == 256) {
                sum += (double)part;
                part = 0.0f;
                cnt = 0;
            }
        }
        sum += (double)part;
        acc += weighted ? 0.5 * sum : sum / (2.0 * (double)(gi.n - 1));
    }
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// Sampled unordered pairs: p -> Philox(ctr = (p_lo, p_hi, 0xFFFFFFFD, 0), key = seed);
// i = floor(w0 n / 2^32), j = negative(w1) of i.  Returns the sum of coef * U^r.
__global__ void objective_pairs_sampled_kernel(const float2 *__restrict__ pos, const int32_t *__restrict__ deg,
                                               const float4 *__restrict__ wt, int32_t n, int64_t pairs,
                                               uint64_t seed, double *partial) {
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    const bool weighted = wt != nullptr;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    double acc = 0.0;
    float part = 0.0f;
    int cnt = 0;
#pragma unroll 4
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < pairs; p += stride) {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)p, (uint32_t)((uint64_t)p >> 32), 0xFFFFFFFDu, 0u), key);
        const int32_t i = (int32_t)__umulhi(w.x, (uint32_t)n);
        const int32_t j = negative_of(w.y, i, (uint32_t)(n - 1));
        const float2 yi = pos[i], yj = pos[j];
        const float dx = yi.x - yj.x, dy = yi.y - yj.y;
        const float r2 = fmaf(dx, dx, dy * dy);
        const float4 wi = weighted ? wt[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 wj = weighted ? wt[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        part += pair_coef((float)deg[i], (float)deg[j], wi, wj, weighted) * (0.5f * reciprocal(1.0f + r2));
        if (++cnt == 256) {
            acc += (double)part;
            part = 0.0f;
            cnt = 0;
        }
    }
    acc += (double)part;
    const double t = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

}  // namespace

cudaError_t launch_segment_rows(const int64_t *row_ptr, int32_t n, int64_t nnz, int32_t seg_len,
                                int32_t *seg_row, int64_t num_segs, cudaStream_t s) {
    if (num_segs <= 0) return cudaSuccess;
    const int block = 256;
    const int64_t want = (num_segs + block - 1) / block;
    const int grid = (int)(want < 65536 ? want : 65536);
    segment_rows_kernel<<<grid, block, 0, s>>>(row_ptr, n, seg_len, seg_row, num_segs);
    (void)nnz;
    return cudaGetLastError();
}

cudaError_t launch_edge_sources(const int64_t *row_ptr, const int32_t *seg_row, int32_t n, int64_t nnz,
                                int32_t seg_len, int32_t *src, cudaStream_t s) {
    if (nnz <= 0) return cudaSuccess;
    const int64_t want = ((nnz + 3) / 4 + 255) / 256;
    edge_sources_kernel<<<(int)(want < 65536 ? want : 65536), 256, 0, s>>>(row_ptr, seg_row, n, nnz, seg_len, src);
    return cudaGetLastError();
}

cudaError_t launch_degrees(const int64_t *row_ptr, int32_t n, int32_t *deg, cudaStream_t s) {
    const int block = 256;
    const int64_t want = ((int64_t)n + block - 1) / block;
    const int grid = (int)(want < 65536 ? (want > 0 ? want : 1) : 65536);
    degrees_kernel<<<grid, block, 0, s>>>(row_ptr, n, deg);
    return cudaGetLastError();
}

cudaError_t launch_validate_csr(const int64_t *row_ptr, const int32_t *col_idx, const int32_t *seg_row,
                                int32_t n, int64_t nnz, int32_t seg_len, uint32_t *flags, cudaStream_t s,
                                const int32_t *node_graph, unsigned long long *upper_count, const int32_t *deg,
                                int32_t *orient) {
    const int block = 256;
    {
        const int64_t want = ((int64_t)n + block - 1) / block;
        const int grid = (int)(want < 65536 ? (want > 0 ? want : 1) : 65536);
        check_row_ptr_kernel<<<grid, block, 0, s>>>(row_ptr, n, nnz, flags);
    }
    if (nnz <= 0) return cudaGetLastError();
    const int64_t want = (nnz + block - 1) / block;
    const int grid = (int)(want < 65536 ? want : 65536);
    validate_csr_kernel<<<grid, block, 0, s>>>(row_ptr, col_idx, seg_row, n, nnz, seg_len, flags, node_graph,
                                               upper_count, deg, orient);
    return cudaGetLastError();
}

cudaError_t launch_objective_edges(const int64_t *row_ptr, const int32_t *col_idx, const int32_t *seg_row,
                                   const float2 *pos, int64_t nnz, int32_t seg_len, double *partial, int grid,
                                   cudaStream_t s) {
    objective_edges_kernel<<<grid, 256, 0, s>>>(row_ptr, col_idx, seg_row, pos, nnz, seg_len, partial);
    return cudaGetLastError();
}

static int grid_for(int64_t items, int block) {
    const int64_t want = (items + block - 1) / block;
    return (int)(want < 65536 ? (want > 0 ? want : 1) : 65536);
}


cudaError_t exclusive_scan_i32(void *temp, size_t *temp_bytes, const int32_t *in, int32_t *out, int64_t count,
                               cudaStream_t s) {
    return cub::DeviceScan::ExclusiveSum(temp, *temp_bytes, in, out, count, s);
}

cudaError_t launch_oriented_rows(const int64_t *row_ptr, const int32_t *pos, int32_t n, const ChunkLayout &to,
                                 int64_t *act_row_ptr, int32_t *pieces, int32_t *multiplier, cudaStream_t s) {
    oriented_rows_kernel<<<grid_for(n, 256), 256, 0, s>>>(row_ptr, pos, n, to.T, to.order, act_row_ptr, pieces,
                                                         multiplier);
    return cudaGetLastError();
}

cudaError_t launch_orient_scatter(const int64_t *row_ptr, const int32_t *col_idx, const int32_t *seg_row, int64_t nnz,
                                  int32_t seg_len, const int32_t *pos, const int64_t *act_row_ptr,
                                  const int32_t *multiplier, const ChunkLayout &to, int4 *ent, int2 *meta,
                                  int64_t capacity, uint32_t *flags, cudaStream_t s) {
    orient_scatter_kernel<<<grid_for(nnz, 256), 256, 0, s>>>(row_ptr, col_idx, seg_row, nnz, seg_len, pos, act_row_ptr,
                                                            multiplier, to, ent, meta, capacity, flags);
    return cudaGetLastError();
}

cudaError_t launch_row_pieces(const int64_t *act_rp, int32_t n, int32_t T, int32_t *pieces, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    row_pieces_kernel<<<grid_for(n, 256), 256, 0, s>>>(act_rp, n, T, pieces);
    return cudaGetLastError();
}

cudaError_t launch_chunk_layout(const int4 *src, const ChunkLayout &from, int4 *dst, const ChunkLayout &to,
                                int2 *meta, const int64_t *act_rp, int32_t n, int64_t nnz, cudaStream_t s) {
    if (nnz == 0) return cudaSuccess;
    chunk_layout_kernel<<<grid_for(nnz, 256), 256, 0, s>>>(src, from, dst, to, meta, act_rp, n, nnz);
    return cudaGetLastError();
}

cudaError_t launch_objective_oriented(const int4 *ent, const ChunkLayout &L, int64_t nnz, const float2 *pos,
                                      double *partial, int grid, cudaStream_t s) {
    objective_oriented_kernel<<<grid, 256, 0, s>>>(ent, L, nnz, pos, partial);
    return cudaGetLastError();
}

cudaError_t launch_objective_pairs_exact(const float2 *pos, const int32_t *deg, const float4 *wt, int32_t n,
                                         double *partial, int grid, cudaStream_t s) {
    // four rows a thread reuse a column's shared-memory read, one row a thread
    // gives a small graph four times as many work items (one against four, us:
    // 3,000 vertices 43 / 56, 12,000 77 / 82, 16,000 103 / 94)
    const bool wide = n >= kWideRows;
    if (wt && wide)
        objective_pairs_exact_kernel<true, 4><<<grid, kPairTile, 0, s>>>(pos, deg, wt, n, partial);
    else if (wt)
        objective_pairs_exact_kernel<true, 1><<<grid, kPairTile, 0, s>>>(pos, deg, wt, n, partial);
    else if (wide)
        objective_pairs_exact_kernel<false, 4><<<grid, kPairTile, 0, s>>>(pos, deg, nullptr, n, partial);
    else
        objective_pairs_exact_kernel<false, 1><<<grid, kPairTile, 0, s>>>(pos, deg, nullptr, n, partial);
    return cudaGetLastError();
}

cudaError_t launch_objective_pairs_batch(const float2 *pos, const int32_t *deg, const float4 *wt,
                                         const int32_t *node_graph, const GraphInfo *graphs, int32_t n,
                                         double *partial, int grid, cudaStream_t s) {
    objective_pairs_batch_kernel<<<grid, 256, 0, s>>>(pos, deg, wt, node_graph, graphs, n, partial);
    return cudaGetLastError();
}

cudaError_t launch_objective_pairs_sampled(const float2 *pos, const int32_t *deg, const float4 *wt, int32_t n,
                                           int64_t pairs, uint64_t seed, double *partial, int grid,
                                           cudaStream_t s) {
    objective_pairs_sampled_kernel<<<grid, 256, 0, s>>>(pos, deg, wt, n, pairs, seed, partial);
    return cudaGetLastError();
}

}  // namespace snap
