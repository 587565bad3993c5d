// PPSD queries by merge-intersection of rank-sorted label lists.
//
// d(u,v) = min over hubs h in L_u and L_v of d(u,h) + d(v,h) (Sec. 1, cover
// property); the paper's single-node mode merges the two hub-rank-sorted lists
// (Sec. 6 QLSN, footnote of Sec. 7.2 on linear-merge querying).
//
// One warp per query. The lists are taken in blocks of up to 128 entries (hub
// rank position, ascending; coalesced loads, both blocks in flight together).
// A block of L_u is entered into a table in shared memory by the low bits of
// its hub positions, every entry of the block of L_v looks its hub up there,
// and matches contribute d(u,h)+d(v,h). The block whose last entry is smaller
// is consumed entirely and the other advances past every entry not larger than
// that, a merge on blocks: every common hub is met exactly once. Sums saturate
// at UINT32_MAX; a pair without a common hub (different components) answers
// UINT32_MAX.
#include "chl_common.cuh"

namespace chl {
namespace {

constexpr unsigned FULL = 0xffffffffu;

constexpr uint32_t TAB = 1024;        // table slots per warp (a power of two)
constexpr uint32_t TAB_EMPTY = 0xFFFFFFFFu;
constexpr int QUERY_TPB = 256;
constexpr int QUERY_WARPS = QUERY_TPB / 32;
constexpr int QUERY_CTAS = 4;         // resident per SM

__device__ __forceinline__ uint32_t sat_add(uint32_t a, uint32_t b) {
    const uint32_t s = a + b;
    return s < a ? 0xFFFFFFFFu : s;
}

// A warp's table in shared memory. Its words carry the generation of the block
// that wrote them, so that a new block needs no clearing: only when the
// generations are used up is the table emptied. Words of other generations
// match no lookup.
struct Table {
    uint32_t *slot;
    uint32_t gen;
};
constexpr uint32_t GENERATIONS = 15;  // the empty word holds the 16th

__device__ __forceinline__ void table_clear(uint32_t *tab) {
    const uint4 e = make_uint4(TAB_EMPTY, TAB_EMPTY, TAB_EMPTY, TAB_EMPTY);
#pragma unroll
    for (uint32_t i = 0; i < TAB / 128; ++i) reinterpret_cast<uint4 *>(tab)[i * 32 + (threadIdx.x & 31)] = e;
    __syncwarp();
}

// Calls hit(d(u,h), d(v,h), h) on some lane for every common hub h of u and v,
// whose lists are the ra entries from a0 and the rb entries from b0; all 32
// lanes call it with the same lists. tab: the warp's table. The shorter list
// is the one that is entered into the table (the sum is symmetric).
//
// A table word is the block's generation, the entry's hub position above the
// slot bits and its index in the block; a lookup is one shared load that tells
// match and index. Chunks are entered last to first, so entries of the first
// TAB rank positions, the bulk of the labels, always hold their slot. Others
// may find it taken: a chunk with such entries reads its slots back, and those
// that lost are compared with the block of L_v one by one.
//
// Bound by instruction issue and the latency of its loads: at 104 labels per
// vertex one block covers most lists, so a pair costs one round of list loads
// where the search of 32-entry chunks through warp shuffles that it replaces
// took about seven dependent ones.
// intersect_blocks: blocks of 32 * NB entries, ra <= rb.
template <int NB, typename F>
__device__ __forceinline__ void intersect_blocks(const uint32_t *__restrict__ ha, const uint32_t *__restrict__ da,
                                                 int ra, const uint32_t *__restrict__ hb,
                                                 const uint32_t *__restrict__ db, int rb, Table &tab, F hit) {
    constexpr int TAB_BITS = 10, IDX_BITS = 7;
    constexpr int POS_BITS = 31 - TAB_BITS;  // of a hub position above the slot
    constexpr int BLOCK = 32 * NB;
    static_assert(TAB == 1u << TAB_BITS && BLOCK <= 1 << IDX_BITS && POS_BITS + IDX_BITS == 28, "table word layout");
    constexpr uint32_t IDX = (1u << IDX_BITS) - 1;
    const int lane = threadIdx.x & 31;
    // this lane's next entries
    ha += lane;
    hb += lane;
    db += lane;
    uint32_t y[NB];
    auto load_b = [&] {
#pragma unroll
        for (int k = 0; k < NB; ++k) y[k] = lane + 32 * k < rb ? __ldg(&hb[32 * k]) : 0xFFFFFFFFu;
    };
    for (;;) {
        uint32_t x[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) x[k] = lane + 32 * k < ra ? __ldg(&ha[32 * k]) : 0u;
        load_b();
        const uint32_t gen = tab.gen << POS_BITS;  // as it stands above a position's upper bits
        bool check = false;  // some chunk holds an entry past the first TAB positions
#pragma unroll
        for (int k = NB - 1; k >= 0; --k) {
            if (lane + 32 * k < ra)
                tab.slot[x[k] & (TAB - 1)] = (gen | x[k] >> TAB_BITS) << IDX_BITS | uint32_t(lane + 32 * k);
            check |= x[k] >= TAB;
            __syncwarp();  // the chunks' stores in this order
        }
        unsigned lost = 0;  // chunks whose entry of this lane lost its slot
        if (__any_sync(FULL, check)) {
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (lane + 32 * k < ra && (tab.slot[x[k] & (TAB - 1)] & IDX) != uint32_t(lane + 32 * k)) lost |= 1u << k;
        }
        const bool any_lost = __any_sync(FULL, lost != 0);
        uint32_t xm = 0;  // the block's last hub position, once needed
        for (;;) {
            // both distances of every match, all loads of the block in flight
            uint32_t ma[NB], mb[NB];
            unsigned met = 0;
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const uint32_t t = tab.slot[y[k] & (TAB - 1)];
                const bool on = lane + 32 * k < rb && t >> IDX_BITS == (gen | y[k] >> TAB_BITS);
                ma[k] = on ? __ldg(&da[t & IDX]) : 0u;
                mb[k] = on ? __ldg(&db[32 * k]) : 0u;
                if (on) met |= 1u << k;
            }
            if (any_lost) {
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    for (unsigned m = __ballot_sync(FULL, (lost >> k) & 1u); m; m &= m - 1) {
                        const int l = __ffs(m) - 1;
                        const uint32_t h = __shfl_sync(FULL, x[k], l);
#pragma unroll
                        for (int j = 0; j < NB; ++j)
                            if (y[j] == h) hit(__ldg(&da[32 * k + l]), __ldg(&db[32 * j]), h);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if ((met >> k) & 1u) hit(ma[k], mb[k], y[k]);
            if (ra <= BLOCK && rb <= BLOCK) {
                rb = 0;  // the last blocks of both
                break;
            }
            if (!xm) {
#pragma unroll
                for (int k = 0; k < NB; ++k)
                    if (lane + 32 * k < ra) xm = x[k];
                xm = __reduce_max_sync(FULL, xm);
            }
            uint32_t c = 0;  // entries of the L_v block up to xm
#pragma unroll
            for (int k = 0; k < NB; ++k) c += __popc(__ballot_sync(FULL, y[k] <= xm));
            hb += c;
            db += c;
            rb -= int(c);
            if (c < BLOCK || !rb) break;  // the block of L_u is consumed, or L_v is
            load_b();
        }
        __syncwarp();  // every lane has read the table
        if (++tab.gen == GENERATIONS) {
            table_clear(tab.slot);
            tab.gen = 0;
        }
        if (!rb || ra <= BLOCK) return;
        ha += BLOCK;
        da += BLOCK;
        ra -= BLOCK;
    }
}

template <typename F>
__device__ __forceinline__ void intersect(const uint32_t *__restrict__ hp, const uint32_t *__restrict__ dd,
                                          uint64_t a0, int ra, uint64_t b0, int rb, Table &tab, F hit) {
    if (!ra || !rb) return;
    if (ra > rb) {
        const uint64_t t = a0;
        a0 = b0;
        b0 = t;
        const int r = ra;
        ra = rb;
        rb = r;
    }
    // a pair's cost is its instructions: a list of up to 64 entries does not
    // pay for the chunks that it leaves empty
    if (rb <= 64) intersect_blocks<2>(hp + a0, dd + a0, ra, hp + b0, dd + b0, rb, tab, hit);
    else intersect_blocks<4>(hp + a0, dd + a0, ra, hp + b0, dd + b0, rb, tab, hit);
}

// The warp's batch of pairs over one set of lists: lane j holds pair (u, v) when
// bit j of mask is set, and d becomes min(d, d(u, v)). The lanes load the list
// ranges of all pairs at once, so that a pair waits for its lists and its
// distances only.
__device__ __forceinline__ void merge_batch(const uint64_t *__restrict__ off, const uint32_t *__restrict__ hp,
                                            const uint32_t *__restrict__ dd, unsigned mask, uint32_t u,
                                            uint32_t v, Table &tab, uint32_t &d) {
    const int lane = threadIdx.x & 31;
    uint64_t a = 0, b = 0;
    int la = 0, lb = 0;
    if ((mask >> lane) & 1u) {
        a = __ldg(&off[u]);
        b = __ldg(&off[v]);
        la = int(__ldg(&off[u + 1]) - a);
        lb = int(__ldg(&off[v + 1]) - b);
    }
    for (unsigned m = mask; m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        uint32_t best = 0xFFFFFFFFu;
        intersect(hp, dd, __shfl_sync(FULL, a, j), __shfl_sync(FULL, la, j), __shfl_sync(FULL, b, j),
                  __shfl_sync(FULL, lb, j), tab,
                  [&](uint32_t x, uint32_t y, uint32_t) { best = min(best, sat_add(x, y)); });
        best = __reduce_min_sync(FULL, best);
        if (lane == j) d = min(d, best);
    }
}

// pairs per warp and step: 16 of a large batch (32 leave the last wave of a
// million pairs half empty), fewer where q pairs would leave warps idle
__device__ __forceinline__ uint32_t pairs_per_warp(uint64_t q) {
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5, each = (q + warps - 1) / warps;
    return each < 16 ? uint32_t(each) : 16u;
}

__global__ void __launch_bounds__(QUERY_TPB, QUERY_CTAS) query_kernel(uint32_t n, const uint64_t *__restrict__ off,
                             const uint32_t *__restrict__ hp, const uint32_t *__restrict__ dd,
                             const uint32_t *__restrict__ pairs, uint64_t q,
                             uint32_t *__restrict__ out, int *bad) {
    __shared__ __align__(16) uint32_t tabs[QUERY_WARPS][TAB];
    Table tab{tabs[threadIdx.x >> 5], 0};
    table_clear(tab.slot);
    const uint32_t lane = threadIdx.x & 31, each = pairs_per_warp(q);
    const uint64_t warp = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t i0 = warp * each; i0 < q; i0 += warps * each) {
        const uint64_t i = i0 + lane;
        const bool mine = lane < each && i < q;
        uint32_t u = 0, v = 0, d = 0xFFFFFFFFu;
        if (mine) {
            u = __ldg(&pairs[2 * i]);
            v = __ldg(&pairs[2 * i + 1]);
        }
        const bool ok = mine && u < n && v < n;
        if (mine && !ok) atomicExch(bad, 1);
        merge_batch(off, hp, dd, __ballot_sync(FULL, ok), u, v, tab, d);
        if (mine) out[i] = d;
    }
}

// The best common hub of u and v: the smallest (d(u,h) + d(v,h), hub position)
// packed as sum << 31 | position (all ones: no common hub). At equal sums the
// highest-ranked hub wins, the canonical hub of the pair (the max-rank vertex
// on its shortest paths). All 32 lanes call it; every lane gets the result.
__device__ __forceinline__ uint64_t merge_best(const uint64_t *__restrict__ off,
                                               const uint32_t *__restrict__ hp,
                                               const uint32_t *__restrict__ dd, uint32_t u, uint32_t v,
                                               Table &tab) {
    const uint64_t a0 = __ldg(&off[u]), b0 = __ldg(&off[v]);
    const int la = int(__ldg(&off[u + 1]) - a0), lb = int(__ldg(&off[v + 1]) - b0);
    uint64_t best = ~0ull;
    intersect(hp, dd, a0, la, b0, lb, tab, [&](uint32_t a, uint32_t b, uint32_t h) {
        const uint64_t x = ((uint64_t(a) + b) << 31) | h;
        best = x < best ? x : best;
    });
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const uint64_t x = __shfl_xor_sync(FULL, best, o);
        best = x < best ? x : best;
    }
    return best;
}

// Index of hub position hpos in the list [lo, hi) of the calling half-warp
// (ascending positions; the list holds it, else the result is ~0): 16-way
// search, each round one load per lane. Both halves of the warp call it
// together, each with its own list; half = lane / 16, l = lane % 16.
__device__ __forceinline__ uint64_t find_hub16(const uint32_t *__restrict__ hp, uint64_t lo, uint64_t hi,
                                               uint32_t hpos, int half, int l) {
    while (__any_sync(FULL, hi - lo > 16)) {
        const uint64_t step = (hi - lo + 15) / 16, j = lo + step * l;
        const bool le = j < hi && __ldg(&hp[j]) <= hpos;
        const uint32_t c = __popc((__ballot_sync(FULL, le) >> (16 * half)) & 0xFFFFu);
        if (c == 0) {
            hi = lo;  // every entry lies above hpos
        } else {
            lo += step * (c - 1);
            hi = hi - lo < step ? hi : lo + step;
        }
    }
    const bool eq = lo + l < hi && __ldg(&hp[lo + l]) == hpos;
    const uint32_t m = (__ballot_sync(FULL, eq) >> (16 * half)) & 0xFFFFu;
    return m ? lo + (__ffs(m) - 1) : ~0ull;
}

// Shortest paths by following the SPT parents stored with the labels (Sec. 5.4,
// Extensions): from u and from v towards their canonical hub H, each step the
// parent stored with w's label of H. One warp per pair: the merge, then the
// lower half-warp walks from u and the upper one from v at the same time.
//
// Bound by the chain of dependent loads per path vertex (its list's range, the
// search, the parent): the search takes two rounds up to 256 labels, where a
// binary search by one lane took eight, and the two sides overlap. The v side
// is written from the path's end, whose place is known only once both lengths
// are, so up to PATH_KEEP of its vertices wait in shared memory; a longer one
// is walked again.
constexpr uint32_t PATH_KEEP = 512;
constexpr int PATH_TPB = 128;

__global__ void __launch_bounds__(PATH_TPB) paths_kernel(uint32_t n, const uint64_t *__restrict__ off,
                             const uint32_t *__restrict__ hp, const uint32_t *__restrict__ dd,
                             const uint32_t *__restrict__ par, const uint32_t *__restrict__ pairs,
                             uint64_t q, uint32_t max_len,
                             uint32_t *__restrict__ paths, uint32_t *__restrict__ lens, int *bad) {
    // the merge's table; between merges its space keeps the v side
    __shared__ __align__(16) uint32_t tabs[PATH_TPB / 32][TAB];
    static_assert(PATH_KEEP <= TAB, "the v side waits in the table's space");
    uint32_t *tab = tabs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, half = lane >> 4, l = lane & 15;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t i = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < q; i += warps) {
        const uint32_t u = __ldg(&pairs[2 * i]), v = __ldg(&pairs[2 * i + 1]);
        if (u >= n || v >= n) {
            if (lane == 0) {
                lens[i] = 0;
                atomicExch(bad, 1);
            }
            continue;
        }
        __syncwarp();  // the previous pair's v side is written out
        table_clear(tab);
        Table merge_tab{tab, 0};
        const uint64_t best = merge_best(off, hp, dd, u, v, merge_tab);
        if (best == ~0ull) {  // different components
            if (lane == 0) lens[i] = 0;
            continue;
        }
        const uint32_t hpos = uint32_t(best & 0x7FFFFFFFu);
        uint32_t *out = paths + i * uint64_t(max_len);
        // u side: u, parent, ..., H at positions 0 .. lu - 1; v side: v, ..., H counted
        uint32_t w = half ? v : u, len = 0;
        bool walking = true, ok = true;
        for (uint32_t guard = 0; guard <= n; ++guard) {
            uint64_t lo = 0, hi = 0;
            if (walking) {
                if (l == 0) {
                    if (!half && len < max_len) out[len] = w;
                    if (half && len < PATH_KEEP) tab[len] = w;
                }
                ++len;
                lo = __ldg(&off[w]);
                hi = __ldg(&off[w + 1]);
            }
            const uint64_t j = find_hub16(hp, lo, hi, hpos, half, l);
            if (walking) {
                if (j == ~0ull) {
                    ok = walking = false;
                } else {
                    const uint32_t p = __ldg(&par[j]);
                    if (p == w) walking = false;  // H: its own parent
                    w = p;
                }
            }
            if (!__any_sync(FULL, walking)) break;
        }
        if (!__all_sync(FULL, ok && !walking)) {
            if (lane == 0) {
                lens[i] = 0;
                atomicExch(bad, 2);
            }
            continue;
        }
        const uint32_t lu = __shfl_sync(FULL, len, 0), lv = __shfl_sync(FULL, len, 16);
        // v at the end, back to the vertex after H (the v side's last vertex is H)
        const uint32_t total = lu + lv - 1, kept = min(lv - 1, PATH_KEEP);
        __syncwarp();
        for (uint32_t k = lane; k < kept; k += 32)
            if (total - 1 - k < max_len) out[total - 1 - k] = tab[k];
        if (lv - 1 > kept) {
            w = v;
            for (uint32_t k = 0; k < lv - 1; ++k) {
                if (lane == 0 && k >= kept && total - 1 - k < max_len) out[total - 1 - k] = w;
                const uint64_t j = find_hub16(hp, __ldg(&off[w]), __ldg(&off[w + 1]), hpos, half, l);
                w = __ldg(&par[j]);
            }
        }
        if (lane == 0) lens[i] = total;
    }
}

// a batch mixing label sets: pair i asks set set_of[i]
// (the set count is read from device memory, so a captured launch stays valid
// as sets are added; set id 0xFFFF marks padding that is skipped). With perm,
// the j-th pair answered is perm[j] (grouped order); its answer still goes to
// out[perm[j]]. A set held as hub partitions (QFDL-style, Sec. 6: every
// partition holds the labels of a disjoint hub range for all vertices) answers
// with the minimum of the partial merges.
__global__ void __launch_bounds__(QUERY_TPB, QUERY_CTAS) query_sets_kernel(const QuerySet *__restrict__ sets, const uint32_t *nsets_p,
                                  const uint32_t *__restrict__ pairs,
                                  const uint16_t *__restrict__ set_of, const uint32_t *__restrict__ perm,
                                  uint64_t q, uint32_t *__restrict__ out, int *bad) {
    __shared__ __align__(16) uint32_t tabs[QUERY_WARPS][TAB];
    Table tab{tabs[threadIdx.x >> 5], 0};
    table_clear(tab.slot);
    const uint32_t lane = threadIdx.x & 31, each = pairs_per_warp(q);
    const uint64_t warp = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    const uint32_t nsets = *nsets_p;
    for (uint64_t j0 = warp * each; j0 < q; j0 += warps * each) {
        const uint64_t j = j0 + lane;
        bool mine = lane < each && j < q;
        uint64_t i = 0;
        uint32_t k = 0xFFFFu, u = 0, v = 0, d = 0xFFFFFFFFu;
        if (mine) {
            i = perm ? __ldg(&perm[j]) : j;
            k = __ldg(&set_of[i]);
            mine = k != 0xFFFFu;
        }
        bool ok = false;
        if (mine) {
            u = __ldg(&pairs[2 * i]);
            v = __ldg(&pairs[2 * i + 1]);
            ok = k < nsets && u < sets[k].n && v < sets[k].n;
            if (!ok) atomicExch(bad, 1);
        }
        // the pairs of one set at a time
        for (unsigned left = __ballot_sync(FULL, ok); left;) {
            const uint32_t k0 = __shfl_sync(FULL, k, __ffs(left) - 1);
            const unsigned group = __ballot_sync(FULL, ok && k == k0);
            left &= ~group;
            const QuerySet &S = sets[k0];
            const uint32_t nparts = S.nparts;
            for (uint32_t p = 0; p < max(nparts, 1u); ++p) {
                const QuerySet &P = nparts ? S.parts[p] : S;
                merge_batch(P.offsets, P.hubpos, P.dist, group, u, v, tab, d);
            }
        }
        if (mine) out[i] = d;
    }
}

// a batch over one set, which travels as a kernel parameter
__global__ void __launch_bounds__(QUERY_TPB, QUERY_CTAS)
query_parts_kernel(const __grid_constant__ QueryParts sets, const uint32_t *__restrict__ pairs,
                   const uint32_t *__restrict__ perm, uint64_t q, uint32_t *__restrict__ out, int *bad) {
    __shared__ __align__(16) uint32_t tabs[QUERY_WARPS][TAB];
    Table tab{tabs[threadIdx.x >> 5], 0};
    table_clear(tab.slot);
    const uint32_t lane = threadIdx.x & 31, each = pairs_per_warp(q);
    const uint64_t warp = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t j0 = warp * each; j0 < q; j0 += warps * each) {
        const uint64_t j = j0 + lane;
        const bool mine = lane < each && j < q;
        uint64_t i = 0;
        uint32_t u = 0, v = 0, d = 0xFFFFFFFFu;
        if (mine) {
            i = perm ? __ldg(&perm[j]) : j;
            u = __ldg(&pairs[2 * i]);
            v = __ldg(&pairs[2 * i + 1]);
        }
        const bool ok = mine && u < sets.n && v < sets.n;
        if (mine && !ok) atomicExch(bad, 1);
        const unsigned mask = __ballot_sync(FULL, ok);
        for (uint32_t p = 0; p < sets.nparts; ++p)
            merge_batch(sets.lists[p].offsets, sets.lists[p].hubpos, sets.lists[p].dist, mask, u, v, tab, d);
        if (mine) out[i] = d;
    }
}

// ---- grouped order (QDOL-style, Sec. 6: queries sorted and grouped by the
// vertex partitions they touch, answers rearranged back into arrival order).
// On one GPU a partition is a block of vertex ids: a pair's key is the block
// pair (min(u, v), max(u, v)) over GROUP_BLOCKS blocks per label set, so pairs
// that read the lists of the same two blocks run together. The order is a
// counting sort by key: count, one-CTA exclusive scan, scatter of indices.
// Pairs of an unknown set or with an id >= n go to key 0 (the query kernel
// reports them).
constexpr uint32_t GROUP_BLOCKS = 64;
constexpr uint32_t GROUP_KEYS = GROUP_BLOCKS * GROUP_BLOCKS;

__device__ __forceinline__ uint32_t group_key(uint32_t n, uint32_t u, uint32_t v) {
    if (u >= n || v >= n) return 0;
    if (u > v) {
        const uint32_t t = u;
        u = v;
        v = t;
    }
    const uint32_t bu = uint32_t(uint64_t(u) * GROUP_BLOCKS / n), bv = uint32_t(uint64_t(v) * GROUP_BLOCKS / n);
    return bu * GROUP_BLOCKS + bv;
}

// the set sizes of a batch: of its pairs' sets, or of its one set (sets null)
struct GroupSets {
    const QuerySet *sets;
    const uint32_t *nsets;
    const uint16_t *set_of;
    uint32_t n;
    __device__ __forceinline__ uint32_t key(const uint32_t *pairs, uint64_t i) const {
        uint32_t size = n;
        if (sets) {
            const uint32_t k = __ldg(&set_of[i]);
            if (k >= *nsets) return 0;
            size = sets[k].n;
        }
        return group_key(size, __ldg(&pairs[2 * i]), __ldg(&pairs[2 * i + 1]));
    }
};

__global__ void group_count_kernel(GroupSets g, const uint32_t *pairs, uint64_t q, uint32_t *cnt) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < q;
         i += uint64_t(gridDim.x) * blockDim.x)
        atomicAdd(&cnt[g.key(pairs, i)], 1u);
}

// exclusive prefix of the GROUP_KEYS counts, in place (one CTA of 1024 threads)
__global__ void __launch_bounds__(1024) group_scan_kernel(uint32_t *cnt) {
    constexpr uint32_t PER = GROUP_KEYS / 1024;
    __shared__ uint32_t wsum[32];
    const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t x[PER], s = 0;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        x[k] = cnt[t * PER + k];
        s += x[k];
    }
    uint32_t inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, inc, o);
        if (lane >= uint32_t(o)) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = wsum[lane], wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, wi, o);
            if (lane >= uint32_t(o)) wi += y;
        }
        wsum[lane] = wi - w;
    }
    __syncthreads();
    uint32_t run = wsum[warp] + inc - s;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        cnt[t * PER + k] = run;
        run += x[k];
    }
}

__global__ void group_scatter_kernel(GroupSets g, const uint32_t *pairs, uint64_t q, uint32_t *fill,
                                     uint32_t *perm) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < q;
         i += uint64_t(gridDim.x) * blockDim.x)
        perm[atomicAdd(&fill[g.key(pairs, i)], 1u)] = uint32_t(i);
}

cudaError_t group_order(const GroupSets &g, const uint32_t *pairs, uint64_t q, uint32_t *scratch, uint32_t *perm,
                        cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    if (q > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(scratch, 0, GROUP_KEYS * sizeof(uint32_t), s);
    if (e) return e;
    uint64_t blocks = (q + 255) / 256;
    if (blocks > uint64_t(device_sms()) * 8) blocks = uint64_t(device_sms()) * 8;
    group_count_kernel<<<unsigned(blocks), 256, 0, s>>>(g, pairs, q, scratch);
    group_scan_kernel<<<1, 1024, 0, s>>>(scratch);
    group_scatter_kernel<<<unsigned(blocks), 256, 0, s>>>(g, pairs, q, scratch, perm);
    return cudaGetLastError();
}

// a larger batch runs on as many CTAs as are resident at once, so that the
// clearing of a warp's table is spread over many pairs
uint64_t resident_blocks(uint64_t blocks) {
    const uint64_t most = uint64_t(device_sms()) * QUERY_CTAS;
    return blocks < most ? blocks : most;
}

}  // namespace

cudaError_t launch_group_order(const QuerySet *sets, const uint32_t *nsets, const uint32_t *pairs,
                               const uint16_t *set_of, uint64_t q, uint32_t *scratch, uint32_t *perm,
                               cudaStream_t s) {
    return group_order(GroupSets{sets, nsets, set_of, 0}, pairs, q, scratch, perm, s);
}

cudaError_t launch_group_order_one(uint32_t n, const uint32_t *pairs, uint64_t q, uint32_t *scratch,
                                   uint32_t *perm, cudaStream_t s) {
    return group_order(GroupSets{nullptr, nullptr, nullptr, n}, pairs, q, scratch, perm, s);
}

cudaError_t launch_query_parts(const QueryParts &sets, const uint32_t *pairs, const uint32_t *perm, uint64_t q,
                               uint32_t *out, int *bad, cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    const uint64_t blocks = resident_blocks((q * 32 + QUERY_TPB - 1) / QUERY_TPB);
    query_parts_kernel<<<unsigned(blocks), QUERY_TPB, 0, s>>>(sets, pairs, perm, q, out, bad);
    return cudaGetLastError();
}

cudaError_t launch_query_sets(const QuerySet *sets, const uint32_t *nsets, const uint32_t *pairs,
                              const uint16_t *set_of, const uint32_t *perm, uint64_t q, uint32_t *out,
                              int *bad, cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    const uint64_t blocks = resident_blocks((q * 32 + QUERY_TPB - 1) / QUERY_TPB);
    query_sets_kernel<<<unsigned(blocks), QUERY_TPB, 0, s>>>(sets, nsets, pairs, set_of, perm, q, out, bad);
    return cudaGetLastError();
}

cudaError_t launch_paths(uint32_t n, const uint64_t *offsets, const uint32_t *hubpos,
                         const uint32_t *dist, const uint32_t *parent, const uint32_t *pairs,
                         uint64_t q, uint32_t max_len, uint32_t *paths,
                         uint32_t *lens, int *bad, cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    uint64_t blocks = (q * 32 + PATH_TPB - 1) / PATH_TPB;
    if (blocks > uint64_t(device_sms()) * 64) blocks = uint64_t(device_sms()) * 64;
    paths_kernel<<<unsigned(blocks), PATH_TPB, 0, s>>>(n, offsets, hubpos, dist, parent, pairs, q,
                                                   max_len, paths, lens, bad);
    return cudaGetLastError();
}

cudaError_t launch_query(uint32_t n, const uint64_t *offsets, const uint32_t *hubpos,
                         const uint32_t *dist, const uint32_t *pairs, uint64_t q, uint32_t *out,
                         int *bad, cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    const uint64_t blocks = resident_blocks((q * 32 + QUERY_TPB - 1) / QUERY_TPB);
    query_kernel<<<unsigned(blocks), QUERY_TPB, 0, s>>>(n, offsets, hubpos, dist, pairs, q, out, bad);
    return cudaGetLastError();
}

}  // namespace chl
