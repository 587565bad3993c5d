// Input validation and renumbering of the graph by rank position.
//
// The paper's input is an undirected graph with positive edge weights
// (Sec. 2) and a total order R (Sec. 1). chl_build checks the CSR on the GPU
// (row bounds, ids, weights >= 1, sorted rows without duplicates or
// self-loops, an equal-weight reverse for every arc) and that R is a
// permutation, then renumbers vertices by rank position p = n-1-R(v): the
// vertex with the highest rank becomes 0. In that numbering the ancestor with
// the highest rank is the smallest id, so "highest-ranked ancestor" in
// Algorithm 3 becomes an unsigned min inside the packed search key, and the
// trees of the most important roots (the largest ones, Sec. 5.1 label counts
// per tree) come first in the claim order.
#include <algorithm>
#include <cstdio>

#include "chl_common.cuh"

namespace chl {

// ------------------------------------------------------------------ scan
namespace {

constexpr int SCAN_TPB = 1024;

__global__ void scan_blocks_kernel(const uint64_t *in, uint64_t *out, uint64_t *block_sums,
                                   uint64_t n) {
    __shared__ uint64_t warp_tot[32];
    const uint64_t i = uint64_t(blockIdx.x) * SCAN_TPB + threadIdx.x;
    const uint64_t x = i < n ? in[i] : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint64_t t = warp_tot[lane];
        uint64_t s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        warp_tot[lane] = s - t;  // exclusive prefix of warp totals
        if (lane == 31 && block_sums) block_sums[blockIdx.x] = s;
    }
    __syncthreads();
    if (i < n) out[i] = incl - x + warp_tot[warp];
}

__global__ void scan_add_kernel(uint64_t *out, const uint64_t *block_prefix, uint64_t n) {
    const uint64_t i = uint64_t(blockIdx.x) * SCAN_TPB + threadIdx.x;
    if (i < n) out[i] += block_prefix[blockIdx.x];
}

}  // namespace

// exclusive scan of n uint64 values; out may alias in
cudaError_t exclusive_scan_u64(const uint64_t *in, uint64_t *out, uint64_t n, cudaStream_t s,
                               int *launches) {
    if (n == 0) return cudaSuccess;
    const uint64_t nb = (n + SCAN_TPB - 1) / SCAN_TPB;
    if (nb == 1) {
        scan_blocks_kernel<<<1, SCAN_TPB, 0, s>>>(in, out, nullptr, n);
        if (launches) *launches += 1;
        return cudaGetLastError();
    }
    uint64_t *sums = nullptr;
    cudaError_t e = dmalloc(&sums, nb * sizeof(uint64_t), s);
    if (e != cudaSuccess) return e;
    scan_blocks_kernel<<<unsigned(nb), SCAN_TPB, 0, s>>>(in, out, sums, n);
    if (launches) *launches += 1;
    e = exclusive_scan_u64(sums, sums, nb, s, launches);
    if (e == cudaSuccess) {
        scan_add_kernel<<<unsigned(nb), SCAN_TPB, 0, s>>>(out, sums, n);
        if (launches) *launches += 1;
        e = cudaGetLastError();
    }
    cudaFreeAsync(sums, s);
    return e;
}

// ------------------------------------------------------------------ validation
namespace {

enum : uint32_t {
    BAD_ROWPTR = 1u << 0,
    BAD_COL = 1u << 1,
    BAD_WEIGHT = 1u << 2,
    BAD_ORDER = 1u << 3,
    BAD_SELF = 1u << 4,
    BAD_SYMM = 1u << 5,
    BAD_RANK = 1u << 6,
};

struct Check {
    uint32_t bits;
    uint32_t where;  // a vertex where the first failure was seen (any)
    uint32_t deg_max;  // longest row
    uint32_t wmax, wmin;
    unsigned long long wsum;
    double wsq;             // sum of the squared weights
    unsigned long long gap; // sum of |u - v| over the arcs
    unsigned long long fp;  // symmetry fingerprint: sum of h(v, u, w) - h(u, v, w) over the arcs
};

__device__ void fail(Check *c, uint32_t bit, uint32_t v) {
    if (!(atomicOr(&c->bits, bit) & bit)) atomicExch(&c->where, v);
}

__global__ void check_rows_kernel(uint32_t n, uint64_t m2, const uint64_t *row, Check *c) {
    uint64_t dmax = 0;
    for (uint64_t v = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n;
         v += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t a = row[v], b = row[v + 1];
        if (a > b || b > m2 || (v == 0 && a != 0) || (v == n - 1 && b != m2)) fail(c, BAD_ROWPTR, uint32_t(v));
        else dmax = max(dmax, b - a);
    }
    const uint32_t d = __reduce_max_sync(0xffffffffu, uint32_t(min(dmax, uint64_t(0xFFFFFFFFu))));
    if ((threadIdx.x & 31) == 0 && d > *(volatile uint32_t *)&c->deg_max) atomicMax(&c->deg_max, d);
}

// 64-bit mix of an arc (the splitmix64 finaliser of Steele, Lea and Flood)
__device__ __forceinline__ unsigned long long arc_hash(uint32_t a, uint32_t b, uint32_t wt) {
    unsigned long long x = ((unsigned long long)a << 32 | b) ^ ((unsigned long long)wt * 0x9E3779B97F4A7C15ull);
    x ^= x >> 30;
    x *= 0xBF58476D1CE4E5B9ull;
    x ^= x >> 27;
    x *= 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// The passes over the arcs give every warp an equal, contiguous piece of them,
// whatever the rows: with a warp per row, one warp walked the longest row
// (25,000 arcs of R-MAT scale 18) long after the others were done (builds with a warp
// per row and so: scale 18 38.5 and 37.2 ms, scale 16 7.43 and 7.08 ms, 50,000
// Barabasi-Albert vertices 9.75 and 9.55 ms; the rows are found with one search per
// piece and 32 row ends a step after that).
constexpr int ARC_TPB = 256;
constexpr int ARC_STEP = 128;  // arcs of a warp in flight, four per lane
constexpr int ARC_BLOCKS = 6;  // blocks per SM

// the row that holds arc e < row[n]
__device__ __forceinline__ uint32_t row_of(uint32_t n, const uint64_t *row, uint64_t e) {
    uint32_t lo = 0, hi = n;  // row[lo] <= e < row[hi]
    while (hi - lo > 1) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (row[mid] <= e) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The row of arc e0 + min(lane, last) on each lane of a warp. v: a row at or
// before that of e0, with no whole row of arcs between; on return the row of the
// last of these arcs. 32 row ends a turn, looked up by shuffles; a run of
// EMPTY_TURNS turns over rows without arcs ends in a search for the row of the
// next arc, so that no warp walks a long run of isolated vertices alone (10^7 of
// them between the arcs: a build 390 ms, now 200, as with them at the end).
constexpr int EMPTY_TURNS = 8;
__device__ __forceinline__ uint32_t rows_of_step(uint32_t n, const uint64_t *row, uint64_t e0, uint32_t last,
                                                 uint32_t &v) {
    const uint32_t lane = threadIdx.x & 31, at = min(lane, last);
    uint32_t r = 0, next = 0;  // arcs before `next` have their row
    int empty = 0;
    bool found = false;
    for (;;) {
        const uint64_t i = uint64_t(v) + 1 + lane;
        const uint32_t end = i <= n ? uint32_t(min(row[i] - e0, uint64_t(ARC_STEP))) : uint32_t(ARC_STEP);
        uint32_t c = 0;  // row ends at or before the arc
#pragma unroll
        for (uint32_t o = 16; o; o >>= 1)
            if (__shfl_sync(0xffffffffu, end, c + o - 1) <= at) c += o;
        const uint32_t top = __shfl_sync(0xffffffffu, end, 31);
        if (c == 31 && top <= at) c = 32;
        if (!found && c < 32) {
            r = v + c;
            found = true;
        }
        if (top > last) break;
        v += 32;
        empty = top == next ? empty + 1 : 0;
        next = top;
        if (empty == EMPTY_TURNS) {
            v = row_of(n, row, e0 + next);
            empty = 0;
        }
    }
    v = __shfl_sync(0xffffffffu, r, 31);
    return r;
}

// Ids, weights, strictly increasing rows, no self-loop, in one streaming pass.
// Symmetry by fingerprint: the arcs (v, u, w) form
// the same multiset as their reverses (u, v, w) iff the graph is undirected
// with equal weights both ways, so the sum of h(v, u, w) - h(u, v, w) is 0
// for every undirected graph; any other sum proves an arc without its
// reverse, which check_symm_kernel then locates.
// Weight statistics come from the same pass. Rows or ranks found bad by the
// kernels before end it at once (its rows could lead anywhere), so that one
// wait of the host sees every check. One set of atomics per block (per warp, at
// 39,000 warps, they queued up at their addresses).
__global__ void __launch_bounds__(ARC_TPB, ARC_BLOCKS)
    check_arcs_kernel(uint32_t n, uint64_t m2, uint64_t per_warp, const uint64_t *row, const uint32_t *col,
                      const uint32_t *w, Check *c) {
    if (*(volatile uint32_t *)&c->bits & (BAD_ROWPTR | BAD_RANK)) return;
    __shared__ unsigned long long part[3][ARC_TPB / 32];
    __shared__ float part_sq[ARC_TPB / 32];
    __shared__ uint32_t most[ARC_TPB / 32], least[ARC_TPB / 32];
    uint32_t wmax = 0, wmin = 0xFFFFFFFFu;
    unsigned long long wsum = 0;
    float wsq = 0.0f;  // (for a launch rule: rounding does not matter)
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long fp = 0, gap = 0;
    const uint64_t lo = (uint64_t(blockIdx.x) * (ARC_TPB / 32) + warp) * per_warp, hi = min(lo + per_warp, m2);
    uint32_t row0 = lo < hi ? row_of(n, row, lo) : 0;
    for (uint64_t e0 = lo; e0 < hi; e0 += ARC_STEP) {
        uint32_t nb[ARC_STEP / 32], we[ARC_STEP / 32];
#pragma unroll
        for (int k = 0; k < ARC_STEP / 32; ++k) {
            const uint64_t e = e0 + 32 * k + lane;
            nb[k] = e < hi ? col[e] : 0;
            we[k] = e < hi ? w[e] : 0;
        }
#pragma unroll
        for (int k = 0; k < ARC_STEP / 32; ++k) {
            const uint64_t b = e0 + 32 * k, e = b + lane;
            if (b >= hi) break;
            const uint32_t v = rows_of_step(n, row, b, uint32_t(min(hi - b, uint64_t(32))) - 1, row0);
            if (e >= hi) continue;
            const uint32_t u = nb[k], wt = we[k];
            if (u >= n) { fail(c, BAD_COL, v); continue; }
            if (wt == 0) fail(c, BAD_WEIGHT, v);
            if (u == v) fail(c, BAD_SELF, v);
            if (e > row[v] && col[e - 1] >= u) fail(c, BAD_ORDER, v);
            gap += u > v ? u - v : v - u;
            wmax = max(wmax, wt);
            wmin = min(wmin, wt);
            wsum += wt;
            wsq += float(wt) * float(wt);
            fp += arc_hash(v, u, wt) - arc_hash(u, v, wt);
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        fp += __shfl_xor_sync(0xffffffffu, fp, o);
        gap += __shfl_xor_sync(0xffffffffu, gap, o);
        wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
        wsq += __shfl_xor_sync(0xffffffffu, wsq, o);
    }
    wmax = __reduce_max_sync(0xffffffffu, wmax);
    wmin = __reduce_min_sync(0xffffffffu, wmin);
    if (lane == 0) {
        part[0][warp] = fp;
        part[1][warp] = gap;
        part[2][warp] = wsum;
        part_sq[warp] = wsq;
        most[warp] = wmax;
        least[warp] = wmin;
    }
    __syncthreads();
    if (threadIdx.x) return;
    for (int k = 1; k < ARC_TPB / 32; ++k) {
        fp += part[0][k];
        gap += part[1][k];
        wsum += part[2][k];
        wsq += part_sq[k];
        wmax = max(wmax, most[k]);
        wmin = min(wmin, least[k]);
    }
    if (fp) atomicAdd(&c->fp, fp);
    if (wsum) {
        atomicAdd(&c->gap, gap);
        atomicAdd(&c->wsum, wsum);
        atomicAdd(&c->wsq, double(wsq));
        atomicMax(&c->wmax, wmax);
        atomicMin(&c->wmin, wmin);
    }
}

// exact symmetry check, run only when the fingerprint is not 0: the reverse
// arc with the same weight by binary search in the target row
__global__ void check_symm_kernel(uint32_t n, const uint64_t *row, const uint32_t *col,
                                  const uint32_t *w, Check *c) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t v = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint64_t a = row[v], b = row[v + 1];
        for (uint64_t e = a + lane; e < b; e += 32) {
            const uint32_t u = col[e], wt = w[e];
            if (u >= n) continue;
            uint64_t lo = row[u], hi = row[u + 1];
            bool found = false;
            while (lo < hi) {
                const uint64_t mid = lo + (hi - lo) / 2;
                const uint32_t x = col[mid];
                if (x == v) { found = (w[mid] == wt); break; }
                if (x < v) lo = mid + 1; else hi = mid;
            }
            if (!found) fail(c, BAD_SYMM, uint32_t(v));
        }
    }
}

__global__ void rank_count_kernel(uint32_t n, const uint32_t *rank, uint32_t *cnt, Check *c) {
    for (uint64_t v = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n;
         v += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t r = rank[v];
        if (r >= n) fail(c, BAD_RANK, uint32_t(v));
        else atomicAdd(&cnt[r], 1u);
    }
}

__global__ void rank_perm_kernel(uint32_t n, const uint32_t *rank, const uint32_t *cnt,
                                 uint32_t *pos_of, uint32_t *vert_at, Check *c) {
    for (uint64_t v = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n;
         v += uint64_t(gridDim.x) * blockDim.x) {
        if (cnt[v] != 1) fail(c, BAD_RANK, uint32_t(v));
        const uint32_t r = rank[v];
        if (r < n) {
            const uint32_t p = n - 1 - r;
            pos_of[v] = p;
            vert_at[p] = uint32_t(v);
        }
    }
}

// degrees in rank order
__global__ void rank_degree_kernel(uint32_t n, const uint64_t *row, const uint32_t *vert_at,
                                   uint64_t *deg) {
    for (uint64_t p = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < n;
         p += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t v = vert_at[p];
        deg[p] = row[v + 1] - row[v];
    }
}

// the arcs in rank order, neighbours renumbered: arc i of the new order belongs
// to the vertex of the position whose new row holds i
__global__ void __launch_bounds__(ARC_TPB, ARC_BLOCKS)
    rank_arcs_kernel(uint32_t n, uint64_t m2, uint64_t per_warp, const uint64_t *row, const uint32_t *col,
                     const uint32_t *w, const uint32_t *vert_at, const uint32_t *pos_of, const uint64_t *nrow,
                     uint2 *arc) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t lo = (uint64_t(blockIdx.x) * (ARC_TPB / 32) + (threadIdx.x >> 5)) * per_warp;
    const uint64_t hi = min(lo + per_warp, m2);
    uint32_t row0 = lo < hi ? row_of(n, nrow, lo) : 0;
    for (uint64_t e0 = lo; e0 < hi; e0 += ARC_STEP) {
        uint64_t src[ARC_STEP / 32];
#pragma unroll
        for (int k = 0; k < ARC_STEP / 32; ++k) {
            const uint64_t b = e0 + 32 * k;
            if (b >= hi) break;
            const uint32_t last = uint32_t(min(hi - b, uint64_t(32))) - 1;
            const uint32_t p = rows_of_step(n, nrow, b, last, row0);
            src[k] = row[vert_at[p]] + (b + min(lane, last) - nrow[p]);
        }
        uint32_t u[ARC_STEP / 32], wt[ARC_STEP / 32];
#pragma unroll
        for (int k = 0; k < ARC_STEP / 32; ++k)
            if (e0 + 32 * k + lane < hi) {
                u[k] = col[src[k]];
                wt[k] = w[src[k]];
            }
#pragma unroll
        for (int k = 0; k < ARC_STEP / 32; ++k)
            if (e0 + 32 * k + lane < hi) arc[e0 + 32 * k + lane] = make_uint2(pos_of[u[k]], wt[k]);
        __syncwarp();
    }
}

// the arcs as they are (the caller's numbering kept)
__global__ void pack_arcs_kernel(uint64_t m2, const uint32_t *col, const uint32_t *w, uint2 *arc) {
    for (uint64_t e = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < m2; e += uint64_t(gridDim.x) * blockDim.x)
        arc[e] = make_uint2(col[e], w[e]);
}

int grid_for(uint64_t work, int tpb) {
    uint64_t b = (work + tpb - 1) / tpb;
    if (b > uint64_t(device_sms()) * 32) b = uint64_t(device_sms()) * 32;
    if (b < 1) b = 1;
    return int(b);
}

}  // namespace

#define CK(x)                                                                   \
    do {                                                                        \
        cudaError_t e__ = (x);                                                  \
        if (e__ != cudaSuccess) {                                               \
            st = cuda_status(e__, #x);                                          \
            goto done;                                                          \
        }                                                                       \
    } while (0)

// A graph with short rows keeps the caller's numbering where neighbours are this
// close in it, as a share of the vertices, on average (a grid by rows: 0.001;
// by rank, or at random: a third): the vertices that a tree reaches then lie
// together, and the slots' keys stay in the last level cache (grids of 262,000
// vertices: 143 ms by rank, 127 ms so; 90,000: 33.5 and 32.1; 49,000 and fewer:
// within 1%, the rank order stays). Scale-free graphs gain more from the rank
// order, which puts the hubs together, and so do random bands twice as wide as the
// bound (100,000 vertices: 880 ms kept at 256 threads, 667 by rank at 1024).
// Light-tailed weights only: the block sizes of the other graphs with short rows
// (choose_params) have no kernels for the caller's numbering.
static constexpr double LOCAL_GAP = 1.0 / 128;
static constexpr uint32_t LOCAL_N = 65536;

chl_status prepare_graph(uint32_t n, uint64_t m2, const uint64_t *row, const uint32_t *col,
                         const uint32_t *w, const uint32_t *rank, bool keep_ids, RankGraph &g, cudaStream_t s,
                         int *launches) {
    chl_status st = CHL_OK;
    Check *chk = nullptr;
    Check hchk{};
    uint32_t *cnt = nullptr;
    uint64_t *deg = nullptr;
    // an equal piece of the arcs for each warp, in whole steps
    const uint64_t arc_steps = (m2 + ARC_STEP - 1) / ARC_STEP;
    const uint64_t arc_warps = std::min<uint64_t>(std::max<uint64_t>(arc_steps, 1),
                                                  uint64_t(device_sms()) * ARC_BLOCKS * (ARC_TPB / 32));
    const uint64_t per_warp = std::max<uint64_t>((arc_steps + arc_warps - 1) / arc_warps, 1) * ARC_STEP;
    const unsigned arc_blocks = unsigned((arc_warps + ARC_TPB / 32 - 1) / (ARC_TPB / 32));
    g = RankGraph{};
    g.n = n;
    g.m2 = m2;
    CK(dmalloc(&chk, sizeof(Check), s));
    hchk.wmin = 0xFFFFFFFFu;
    CK(cudaMemcpyAsync(chk, &hchk, sizeof(Check), cudaMemcpyHostToDevice, s));
    CK(dmalloc(&cnt, size_t(n) * sizeof(uint32_t), s));
    CK(cudaMemsetAsync(cnt, 0, size_t(n) * sizeof(uint32_t), s));
    CK(dmalloc(&g.pos_of, size_t(n) * sizeof(uint32_t), s));
    CK(dmalloc(&g.vert_at, size_t(n) * sizeof(uint32_t), s));
    check_rows_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, m2, row, chk);
    rank_count_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, rank, cnt, chk);
    rank_perm_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, rank, cnt, g.pos_of, g.vert_at, chk);
    check_arcs_kernel<<<arc_blocks, ARC_TPB, 0, s>>>(n, m2, per_warp, row, col, w, chk);
    *launches += 4;
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(&hchk, chk, sizeof(Check), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hchk.bits & BAD_ROWPTR) {
        uint64_t last = 0;
        CK(cudaMemcpyAsync(&last, row + n, sizeof(last), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        if (last != m2) {
            st = set_error(CHL_EINVAL, "row_ptr[n] = %llu differs from num_arcs = %llu", (unsigned long long)last,
                           (unsigned long long)m2);
            goto done;
        }
        st = set_error(CHL_EINVAL, "row_ptr is not a valid CSR offset array (vertex %u)", hchk.where);
        goto done;
    }
    if (hchk.bits & BAD_RANK) {
        st = set_error(CHL_EINVAL, "rank is not a permutation of [0,n) (vertex %u)", hchk.where);
        goto done;
    }
    if (!(hchk.bits & BAD_COL) && hchk.fp) {
        // some arc has no reverse of equal weight: find a vertex that shows it
        check_symm_kernel<<<grid_for(uint64_t(n) * 32, 256), 256, 0, s>>>(n, row, col, w, chk);
        *launches += 1;
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(&hchk, chk, sizeof(Check), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        if (!hchk.bits) hchk.bits = BAD_SYMM;  // (a non-zero sum always has a cause)
    }
    if (hchk.bits) {
        const char *what = (hchk.bits & BAD_COL)      ? "a neighbour id is >= n"
                           : (hchk.bits & BAD_WEIGHT) ? "a weight is 0 (weights must be positive)"
                           : (hchk.bits & BAD_SELF)   ? "a self-loop is present"
                           : (hchk.bits & BAD_ORDER)  ? "a row is not strictly increasing (unsorted or duplicate arcs)"
                                                      : "an arc has no reverse arc of equal weight (graph must be undirected)";
        st = set_error(CHL_EINVAL, "invalid graph: %s (vertex %u)", what, hchk.where);
        goto done;
    }
    // renumber by rank position
    CK(dmalloc(&deg, (size_t(n) + 1) * sizeof(uint64_t), s));
    CK(dmalloc(&g.row, (size_t(n) + 1) * sizeof(uint64_t), s));
    CK(dmalloc(&g.arc, (m2 ? m2 : 1) * sizeof(uint2), s));
    g.deg_max = hchk.deg_max;
    g.w_mean = m2 ? double(hchk.wsum) / double(m2) : 1.0;
    g.w_spread = m2 ? hchk.wsq / double(m2) / (g.w_mean * g.w_mean) : 1.0;
    g.local = m2 && double(hchk.gap) / double(m2) < double(n) * LOCAL_GAP;
    g.caller_ids = keep_ids && n >= LOCAL_N && g.local && g.deg_max <= DIRECT_DEGREE && g.w_spread <= HEAVY_SPREAD;
    if (g.caller_ids) {
        CK(cudaMemcpyAsync(g.row, row, (size_t(n) + 1) * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    } else {
        rank_degree_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, row, g.vert_at, deg);
        *launches += 1;
        CK(cudaMemsetAsync(deg + n, 0, sizeof(uint64_t), s));
        CK(exclusive_scan_u64(deg, g.row, uint64_t(n) + 1, s, launches));
    }
    if (g.caller_ids)
        pack_arcs_kernel<<<grid_for(m2, 256), 256, 0, s>>>(m2, col, w, g.arc);
    else
        rank_arcs_kernel<<<arc_blocks, ARC_TPB, 0, s>>>(n, m2, per_warp, row, col, w, g.vert_at, g.pos_of, g.row,
                                                       g.arc);
    *launches += 1;
    CK(cudaGetLastError());
    g.w_max = m2 ? hchk.wmax : 1;
    g.w_min = m2 ? hchk.wmin : 1;
done:
    if (chk) cudaFreeAsync(chk, s);
    if (cnt) cudaFreeAsync(cnt, s);
    if (deg) cudaFreeAsync(deg, s);
    if (st != CHL_OK) free_graph(g, s);
    return st;
}

void free_graph(RankGraph &g, cudaStream_t s) {
    if (g.row) cudaFreeAsync(g.row, s);
    if (g.arc) cudaFreeAsync(g.arc, s);
    if (g.vert_at) cudaFreeAsync(g.vert_at, s);
    if (g.pos_of) cudaFreeAsync(g.pos_of, s);
    g.row = nullptr;
    g.arc = nullptr;
    g.vert_at = nullptr;
    g.pos_of = nullptr;
}

}  // namespace chl
