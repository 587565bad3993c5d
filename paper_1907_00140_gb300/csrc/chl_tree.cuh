// Device code shared by the tree kernels (chl_tree.cu, chl_small.cu): tree keys,
// and the pruning queries over the Common Label Table and the label table.
#pragma once

#include "chl_common.cuh"

namespace chl {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t CLT_MAX = 64;  // largest Common Label Table (hubs)
constexpr uint32_t LTH_SLOTS = 1024;  // hash of the root's labels in the label table
constexpr uint32_t LTH_MAX = 512;     // most root labels the hash holds
constexpr int QSTEPS = 4;             // label-table query from global memory: loads in flight per lane

// ------------------------------------------------------------------ keys
// Vertices are numbered by rank position (pos 0 = most important), so in the
// tree of root h a vertex outranks h iff its pos is below h. Algorithm 3 keeps
// per vertex its distance and the highest-ranked vertex a[v] on its shortest
// paths; the label decision only asks whether a[v] is h itself, and a[v] can
// never rank below h (every path starts at h). So one bit carries it:
//   key = dist << 1 | clean
// clean = 1 iff no vertex before v on the best known paths outranks h. Under
// unsigned min a shorter distance wins and, at equal distance, clean = 0
// wins: a vertex is outranked as soon as one of its shortest paths is (the
// equal-distance branch of Algorithm 3; Sec. 5.2's example, a[v5] = v1).
// v is live (would get the label (h, d)) iff clean and v >= h, and the bit
// it passes on to its out-neighbours is exactly its own liveness.
// Three layouts (K below is one of these traits; K::T is the stored word):
//   KeyN  uint32  dist << 1 | clean            when every tentative distance is
//                                              provably below 2^31 - 1 (the host
//                                              checks w_max * n)
//   KeyW  uint64  dist << 1 | clean            otherwise
//   KeyP  uint64  dist << 32 | clean << 31 | parent, for path recovery (the
//                 SPT parent stored with each label, Sec. 5.4 (Extensions)):
//                 among equal (dist, clean) the smallest parent id wins, so
//                 the parent is the lowest-numbered tight predecessor, a
//                 deterministic choice. A candidate carries its source
//                 vertex in the parent field.
// All ones is "unreached".
// U: arcs a lane relaxes per step of the arc pass (its loads in flight); the
// 8-byte layouts take two, so that a thread's probe state fits its registers
// at 1024 threads per SM.
// IDS: vertices are numbered as by the caller and their rank positions read from
// p.pos (a type of its own, so that the kernels of rank-ordered graphs pay
// nothing for it).
struct KeyN { using T = uint32_t; static constexpr int S = 1; static constexpr int U = 4; static constexpr bool IDS = false; };
struct KeyW { using T = uint64_t; static constexpr int S = 1; static constexpr int U = 2; static constexpr bool IDS = false; };
struct KeyP { using T = uint64_t; static constexpr int S = 32; static constexpr int U = 2; static constexpr bool IDS = false; };
template <typename K>
struct ById : K {
    static constexpr bool IDS = true;
};

template <typename K>
__device__ __forceinline__ typename K::T key_inf() { return ~typename K::T(0); }
template <typename K>
__device__ __forceinline__ typename K::T make_key(uint64_t dist, bool clean, uint32_t parent) {
    using KS = typename K::T;
    return (KS(dist) << K::S) | (KS(clean) << (K::S - 1)) | (K::S > 1 ? KS(parent) : KS(0));
}
template <typename K>
__device__ __forceinline__ uint32_t key_dist(typename K::T k) { return uint32_t(k >> K::S); }
template <typename K>
__device__ __forceinline__ bool key_clean(typename K::T k) { return (k >> (K::S - 1)) & 1; }
template <typename K>
__device__ __forceinline__ uint32_t key_parent(typename K::T k) {
    return K::S > 1 ? uint32_t(k & 0x7FFFFFFFu) : 0u;
}
// largest distance a key holds below key_inf
template <typename K>
__device__ __forceinline__ uint64_t key_dist_limit() {
    return sizeof(typename K::T) == 4 ? 0x7FFFFFFEull : 0xFFFFFFFEull;
}

// rank position of a vertex; caller's id of a vertex; vertex of a root (given by
// its rank position)
template <typename K>
__device__ __forceinline__ uint32_t pos_at(const TreeLaunch &p, uint32_t v) { return K::IDS ? __ldg(&p.pos[v]) : v; }
template <typename K>
__device__ __forceinline__ uint32_t caller_id(const TreeLaunch &p, uint32_t v) { return K::IDS ? v : __ldg(&p.vert_at[v]); }
template <typename K>
__device__ __forceinline__ uint32_t root_vertex(const TreeLaunch &p, uint32_t h) { return K::IDS ? __ldg(&p.vert_at[h]) : h; }

// bucket of a distance: a shift when the width is a power of two
__device__ __forceinline__ uint32_t bucket_of(const TreeLaunch &p, uint32_t d) {
    return p.delta_shift >= 0 ? d >> p.delta_shift : d / p.delta;
}

template <typename K>
__device__ __forceinline__ bool is_live(typename K::T k, uint32_t vpos, uint32_t h) {
    return key_clean<K>(k) && vpos >= h;
}

__device__ __forceinline__ uint32_t atomic_min_key(uint32_t *a, uint32_t v) { return atomicMin(a, v); }
__device__ __forceinline__ uint64_t atomic_min_key(uint64_t *a, uint64_t v) {
    return atomicMin((unsigned long long *)a, (unsigned long long)v);
}
// In the queries below SH is a kernel's shared state: hch[] (the root's table
// row), lth_key[] and lth_val[] (the root's table labels, hashed).

// Common Label Table pruning (Sec. 5.3): does the distance query between the
// root and v over the table hubs, min_c d(h, c) + d(c, v), reach dv; the table
// row of v is read as 16-byte vectors (rows are padded to a multiple of 4 hubs).
// With d(c, v) <= dv the sum is compared without wider arithmetic, and a missing
// label (all ones) on either side never passes: dv is below it.
template <typename SH>
__device__ __forceinline__ bool clt_prunes(const TreeLaunch &p, const SH &S, uint32_t v, uint32_t dv) {
    const uint4 *row = reinterpret_cast<const uint4 *>(p.hc + size_t(v) * p.hc_stride);
    bool hit = false;
    for (uint32_t c4 = 0; c4 < p.hc_stride / 4; ++c4) {
        const uint4 x = __ldg(&row[c4]);
        const uint32_t b[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) hit |= (b[j] <= dv) & (S.hch[c4 * 4 + j] <= dv - b[j]);
    }
    return hit;
}

// Label table of earlier phases (hybrid pruning): every label of every hub of
// rank position below p.lt_hubs, as CSR by vertex rank position (entries of a
// vertex unordered). min over shared hubs c of d(h,c) + d(c,v) <= dv means a
// vertex outranking h lies on a shortest h-v path, as for the Common Label
// Table: the table is complete for a rank-closed set of hubs (Sec. 5.3). The
// query must see every table label of h and of v: a vertex reached only past a
// pruned one is left with a wrong distance and ancestor unless it is pruned
// too, which the complete query guarantees (a partial one would not). The
// root's table labels are hashed in shared memory, or, when more than the hash
// holds, written into the slot's dense array p.lt_root by hub position.
__device__ __forceinline__ uint32_t lth_slot(uint32_t hp) { return (hp * 2654435761u) >> 22; }

// entry j of the label table: {hub position, distance}
__device__ __forceinline__ uint2 lt_entry(const TreeLaunch &p, uint64_t j) {
    if (!p.lt_db) return __ldg(&p.lt_e[j]);
    const uint32_t x = __ldg(&p.lt_w[j]);
    return make_uint2(x >> p.lt_db, x & ((1u << p.lt_db) - 1));
}

// the root's distance to hub position c by the hash, or NONE
template <typename SH>
__device__ __forceinline__ uint32_t lth_find(const SH &S, uint32_t c) {
    for (uint32_t sx = lth_slot(c);; sx = (sx + 1) & (LTH_SLOTS - 1)) {
        const uint32_t key = S.lth_key[sx];
        if (key == 0) return NONE;  // the hash holds at most half its slots
        if (key == c + 1) return S.lth_val[sx];
    }
}

}  // namespace
}  // namespace chl
