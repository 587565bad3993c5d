// Small trees: shortest-path trees whose whole state lives in shared memory.
//
// The trees of the last phases reach from a handful to a few thousand vertices,
// in rounds of tens of expansions. With the dense per-slot state of
// chl_tree.cu every round is a chain of dependent loads and atomics in global
// memory (list, key, target keys, list appends) over regions far larger than
// the caches, and its time is that chain's latency. Here a CTA keeps the
// vertices its tree has reached in a hash table in shared memory (vertex, key),
// so that only rows, arcs and the pruning tables are read from global memory,
// which all trees share.
//
// The search is the same bucketed label-correcting Dijkstra over the same keys
// (chl_tree.cuh), with one list of pending vertices instead of bucket lists:
//   scan    every pending vertex whose key lies in the current bucket moves to
//           the round's list, the others stay; the scan also tells whether any
//           pending vertex is live
//   expand  the round's vertices are pruned or relax their arcs; an improved
//           vertex that is not pending becomes pending
// and the smallest bucket among the keys that stayed and those that were set
// is the next round's. When it lies above the current bucket, the bucket is
// settled, and the tree stops if no pending vertex is live (the early
// termination of Sec. 5.2, exact at bucket granularity as in chl_tree.cu).
//
// A tree that outgrows the table, its lists or the hash of its root's table
// labels is given up, its root goes to the spill list, and the general kernel
// builds it; so the class of table (threads, slots) is only a matter of speed.
//
// Bound by instruction issue of the few warps that the tables leave room for
// (9 or 12 CTAs of 64 threads per SM; a quarter of the issue slots, 1.5 of 15 cycles
// per instruction on global loads), where the general kernel waits on global
// memory. So it wins where trees are tiny and many: R-MAT scale 18 roots
// [38912, 155648) 0.79 -> 0.35 ms, [9728, 38912) 1.70 -> 1.32 ms, a 50,000-vertex
// Barabasi-Albert graph's [9728, 38912) 1.94 -> 1.11 ms, the last 184,000 roots of
// a 512x512 grid 15.6 -> 10.5 ms. Tables of 4,096 and 8,192 slots for trees of
// about a thousand vertices lost to it on that Barabasi-Albert graph (1.9 ms against
// 4.3 and 5.8); they were not tried on grids.
#include "chl_tree.cuh"

namespace chl {
namespace {

constexpr uint32_t PENDING = 0x80000000u;  // in a slot's id: the vertex is in the pending list
constexpr uint32_t ID_MASK = 0x7FFFFFFFu;
constexpr uint32_t EMPTY = 0xFFFFFFFFu;    // free slot (no vertex: ids are below 2^31 - 1)
constexpr uint32_t ROOT_BITS = 8192;       // filter in front of the hash of the root's table labels
constexpr uint32_t GROUP_DEGREE = 8;       // rows up to this length are relaxed by four lanes, longer ones by a warp

struct Counters {
    uint32_t n_cur, n_next, minb;
};

template <int TPB, int SLOTS, typename K>
struct Tree {
    static constexpr uint32_t CAP = small_capacity(SLOTS);  // vertices a tree may reach
    static constexpr uint32_t FRONT = CAP / 2;      // vertices pending or in a round
    // a thread inserts at most one vertex past CAP before it sees `over`
    static_assert(SLOTS - CAP >= TPB, "probes always meet a free slot");
    typename K::T key[SLOTS];
    uint32_t id[SLOTS];
    uint16_t touch[CAP];      // slots in use
    uint16_t cur[FRONT];      // the round's vertices
    uint16_t pend[2][FRONT];  // pending vertices
    // a chunk of the round's vertices: row start and length (0: pruned), key
    uint64_t rs[TPB];
    uint32_t deg[TPB];
    typename K::T kv[TPB];
    uint32_t hch[CLT_MAX];    // the root's Common Label Table row
    Counters c[2];            // of this round and the next
    uint32_t root, n_touch;
    int over;                 // the tree does not fit
    int stop;                 // error: give up
    int ok;
    uint32_t n_out, n_put;
    uint32_t max_d;           // largest label distance (all trees)
    unsigned long long base;
    unsigned long long n_exp[TPB / 32], n_arcs[TPB / 32], n_pruned[TPB / 32];  // statistics of this tree per warp
    // label-pruned phases only (the launch leaves the rest out otherwise)
    uint32_t lth_key[LTH_SLOTS], lth_val[LTH_SLOTS];
    uint32_t lth_bit[ROOT_BITS / 32];  // by hub position modulo ROOT_BITS
    // the chunk's table queries: list start and length (0: none), distance;
    // the answer replaces the length
    uint64_t la[TPB];
    uint32_t len[TPB], dv[TPB];
};

template <typename T>
__device__ __forceinline__ T peek(const T &x) { return *const_cast<const volatile T *>(&x); }

// relax one arc (u, w) of a vertex of key kv (see make_key): find or insert u,
// lower its key, make it pending in list x
template <int TPB, int SLOTS, typename K>
__device__ __forceinline__ void relax(const TreeLaunch &p, Tree<TPB, SLOTS, K> &S, Counters &c, int x,
                                      typename K::T kv, uint2 a) {
    using KS = typename K::T;
    using TR = Tree<TPB, SLOTS, K>;
    constexpr int BITS = 31 - __builtin_clz(SLOTS);
    const uint32_t u = a.x;
    if (sizeof(KS) == 8 && uint64_t(key_dist<K>(kv)) + a.y > key_dist_limit<K>()) {
        atomicExch(&p.flags[0], ERR_DIST_OVERFLOW);
        S.stop = 1;
        return;
    }
    const KS cand = kv + (KS(a.y) << K::S);
    uint32_t s = (u * 2654435761u) >> (32 - BITS);
    for (uint32_t tries = 0;; ++tries) {
        uint32_t w = peek(S.id[s]);
        if (w == EMPTY) {
            if (peek(S.over)) return;
            w = atomicCAS(&S.id[s], EMPTY, u);
            if (w == EMPTY) {
                const uint32_t t = atomicAdd(&S.n_touch, 1u);
                if (t >= TR::CAP) {
                    S.over = 1;
                    return;
                }
                S.touch[t] = uint16_t(s);
                break;
            }
        }
        if ((w & ID_MASK) == u) break;
        s = (s + 1) & (SLOTS - 1);
        if (tries >= SLOTS) {  // (cannot happen: free slots remain)
            S.over = 1;
            return;
        }
    }
    if (cand >= peek(S.key[s])) return;
    if (cand >= atomic_min_key(&S.key[s], cand)) return;
    atomicMin(&c.minb, bucket_of(p, key_dist<K>(cand)));
    if (!(atomicOr(&S.id[s], PENDING) & PENDING)) {
        const uint32_t at = atomicAdd(&c.n_next, 1u);
        if (at < TR::FRONT) S.pend[x][at] = uint16_t(s);
        else S.over = 1;
    }
}

// append val where on, in warp order, to a list counted in shared memory
__device__ __forceinline__ void append16(bool on, uint32_t val, uint16_t *list, uint32_t *counter, uint32_t most) {
    const unsigned m = __ballot_sync(FULL, on);
    if (!m) return;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    uint32_t b = 0;
    if (lane == leader) b = atomicAdd(counter, uint32_t(__popc(m)));
    b = __shfl_sync(FULL, b, leader) + __popc(m & ((1u << lane) - 1));
    if (on && b < most) list[b] = uint16_t(val);
}

// Answers the chunk's m table queries, eight lanes each: every lane takes every
// eighth entry of the list, eight loads in flight, and the group stops after a
// step with a witness (the general kernel's lt_scan runs a whole warp for one of
// the longer lists of the larger trees).
template <typename TR>
__device__ __forceinline__ void answer_queries(const TreeLaunch &p, TR &S, uint32_t m) {
    constexpr int LANES = 8, STEPS = 8;
    const int lane = threadIdx.x & 31, l = lane % LANES, group = lane / LANES;
    for (uint32_t q0 = (threadIdx.x - lane) / LANES; q0 < m; q0 += blockDim.x / LANES) {
        const uint32_t q = q0 + group;
        uint32_t len = 0, dv = 0;
        uint64_t a = 0;
        if (q < m) {
            len = S.len[q];
            a = S.la[q];
            dv = S.dv[q];
        }
        bool found = false;
        for (uint32_t j0 = 0; __any_sync(FULL, !found && j0 < len); j0 += LANES * STEPS) {
            uint2 e[STEPS];
#pragma unroll
            for (int t = 0; t < STEPS; ++t) {
                const uint32_t j = j0 + t * LANES + l;
                e[t] = !found && j < len ? lt_entry(p, a + j) : make_uint2(0, NONE);
            }
            bool hit = false;
#pragma unroll
            for (int t = 0; t < STEPS; ++t) {
                // most entries are no hub of the root: one load tells
                const bool on = e[t].y <= dv && (S.lth_bit[(e[t].x & (ROOT_BITS - 1)) >> 5] >> (e[t].x & 31) & 1u);
                if (on) hit |= lth_find(S, e[t].x) <= dv - e[t].y;  // (never for NONE: dv is below it)
            }
            const unsigned h = __ballot_sync(FULL, hit);
            found |= ((h >> (group * LANES)) & ((1u << LANES) - 1)) != 0;
        }
        if (q < m && l == 0) S.len[q] = found;
    }
}

template <int TPB, int SLOTS, typename K>
__global__ void __launch_bounds__(TPB) plant_small_kernel(TreeLaunch p, uint32_t *spill, unsigned int *spill_n) {
    using KS = typename K::T;
    using TR = Tree<TPB, SLOTS, K>;
    extern __shared__ __align__(16) unsigned char raw[];
    TR &S = *reinterpret_cast<TR *>(raw);
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < SLOTS; i += TPB) {
        S.id[i] = EMPTY;
        S.key[i] = key_inf<K>();
    }
    if (tid == 0) S.max_d = 0;
    // launch statistics, of the trees built here: a spilled tree's work is counted
    // by the kernel that builds it (the first three on lane 0, of its warp)
    unsigned long long n_exp = 0, n_arcs = 0, n_pruned = 0, n_rounds = 0, n_buckets = 0, n_trees = 0;

    for (;;) {
        __syncthreads();  // the previous tree's table is clean, S.root is read
        if (tid == 0) {
            uint32_t r = NONE;
            if (!p.flags[1] && !p.flags[0]) {
                const uint32_t cnt = p.count_dev ? *(volatile const uint32_t *)p.count_dev : p.root_count;
                const uint32_t i = atomicAdd(p.next_root, 1u);
                if (i < cnt) r = p.root_list ? p.root_list[i] : p.root_begin + i;
            }
            S.root = r;
            S.over = S.stop = 0;
            S.n_out = S.n_put = 0;
            S.n_touch = 0;
            S.c[0] = Counters{0, 0, NONE};
        }
        __syncthreads();
        const uint32_t h = S.root;
        if (h == NONE) break;
        const uint32_t hv = root_vertex<K>(p, h);
        uint32_t rounds = 0, buckets = 0;
        if (lane == 0) S.n_exp[tid >> 5] = S.n_arcs[tid >> 5] = S.n_pruned[tid >> 5] = 0;
        // the pruning tables of the root (see chl_tree.cu)
        const bool prune = p.hc && h >= p.hc_hubs;
        if (prune)
            for (uint32_t k = tid; k < p.hc_stride; k += TPB) S.hch[k] = __ldg(&p.hc[size_t(hv) * p.hc_stride + k]);
        const bool lt = p.lt_off && h >= p.lt_hubs;
        bool fits = true;
        if (lt) {
            const uint64_t a = __ldg(&p.lt_off[hv]);
            const uint32_t cnt = uint32_t(__ldg(&p.lt_off[hv + 1]) - a);
            fits = cnt <= LTH_MAX;
            if (fits) {
                for (uint32_t i = tid; i < LTH_SLOTS; i += TPB) S.lth_key[i] = 0;
                for (uint32_t i = tid; i < ROOT_BITS / 32; i += TPB) S.lth_bit[i] = 0;
                __syncthreads();
                for (uint32_t i = tid; i < cnt; i += TPB) {
                    const uint2 e = lt_entry(p, a + i);
                    atomicOr(&S.lth_bit[(e.x & (ROOT_BITS - 1)) >> 5], 1u << (e.x & 31));
                    for (uint32_t sx = lth_slot(e.x);; sx = (sx + 1) & (LTH_SLOTS - 1)) {
                        if (atomicCAS(&S.lth_key[sx], 0u, e.x + 1) == 0u) {
                            S.lth_val[sx] = e.y;
                            break;
                        }
                    }
                }
            }
        }
        if (fits) {
            if (tid == 0) {
                constexpr int BITS = 31 - __builtin_clz(SLOTS);
                const uint32_t s = (hv * 2654435761u) >> (32 - BITS);
                S.id[s] = hv | PENDING;
                S.key[s] = make_key<K>(0, true, h);
                S.touch[0] = uint16_t(s);
                S.n_touch = 1;
                S.pend[0][0] = uint16_t(s);
            }
            __syncthreads();
            uint32_t n_pend = 1, b = 0;
            int x = 0, r = 0;
            bool entered = true;  // the current bucket was entered by this round
            for (;;) {
                // ---- scan the pending vertices
                Counters &c = S.c[r];
                const uint64_t t_hi = uint64_t(b + 1) * p.delta;
                uint32_t mb = NONE;
                bool live = false;
                for (uint32_t i0 = 0; i0 < n_pend; i0 += TPB) {
                    const uint32_t i = i0 + tid;
                    bool in = false, keep = false;
                    uint32_t s = 0;
                    if (i < n_pend) {
                        s = S.pend[x][i];
                        const KS k = S.key[s];
                        const uint32_t v = S.id[s] & ID_MASK, d = key_dist<K>(k);
                        live |= is_live<K>(k, pos_at<K>(p, v), h);
                        in = d < t_hi;
                        keep = !in;
                        if (in) S.id[s] = v;  // no longer pending
                        else mb = min(mb, bucket_of(p, d));
                    }
                    append16(in, s, S.cur, &c.n_cur, TR::FRONT);
                    append16(keep, s, S.pend[x ^ 1], &c.n_next, TR::FRONT);
                }
                mb = __reduce_min_sync(FULL, mb);
                if (lane == 0 && mb != NONE) atomicMin(&c.minb, mb);
                const bool any_live = __syncthreads_or(live);
                if (tid == 0) S.c[r ^ 1] = Counters{0, 0, NONE};  // the last round's, read by all
                if (entered && !any_live) break;  // no pending vertex can still receive the root as hub
                // ---- expand the round's vertices
                const uint32_t n_cur = c.n_cur;
                for (uint32_t i0 = 0; i0 < n_cur; i0 += TPB) {
                    const uint32_t m = min(n_cur - i0, uint32_t(TPB));
                    const bool ex = uint32_t(tid) < m;
                    uint32_t s = 0, v = 0, dv = 0, deg = 0, len = 0;
                    KS k = 0;
                    bool cut = false;
                    if (ex) {
                        s = S.cur[i0 + tid];
                        v = peek(S.id[s]) & ID_MASK;
                        k = peek(S.key[s]);
                        dv = key_dist<K>(k);
                        const uint64_t rs = __ldg(&p.row[v]);
                        deg = uint32_t(__ldg(&p.row[v + 1]) - rs);
                        S.rs[tid] = rs;
                        const uint32_t vpos = pos_at<K>(p, v);
                        S.kv[tid] = make_key<K>(dv, is_live<K>(k, vpos, h), vpos);
                        if (lt) {
                            const uint64_t a = __ldg(&p.lt_off[v]);
                            len = uint32_t(__ldg(&p.lt_off[v + 1]) - a);
                            S.la[tid] = a;
                            S.dv[tid] = dv;
                        }
                        cut = prune && clt_prunes(p, S, v, dv);
                        if (lt) {
                            cut |= vpos < p.lt_hubs;  // a table hub: the complete query would prune it
                            if (cut) len = 0;
                            S.len[tid] = len;
                        }
                    }
                    if (lt) {
                        __syncthreads();
                        answer_queries(p, S, m);
                        __syncthreads();
                        if (ex && len) cut = S.len[tid] != 0;
                    }
                    if (cut) {
                        deg = 0;
                        if (key_clean<K>(k)) atomic_min_key(&S.key[s], make_key<K>(dv, false, 0));
                    }
                    if (ex) S.deg[tid] = deg;
                    {
                        const unsigned em = __ballot_sync(FULL, ex), pm = __ballot_sync(FULL, cut);
                        const uint32_t arcs = __reduce_add_sync(FULL, deg);
                        if (lane == 0) {
                            S.n_exp[tid >> 5] += __popc(em);
                            S.n_pruned[tid >> 5] += __popc(pm);
                            S.n_arcs[tid >> 5] += arcs;
                        }
                    }
                    __syncthreads();
                    // short rows: four lanes each
                    for (uint32_t j = tid; j < 4 * m; j += TPB) {
                        const uint32_t i = j >> 2, d = S.deg[i];
                        if (d > GROUP_DEGREE) continue;
                        for (uint32_t e = j & 3; e < d; e += 4) relax(p, S, c, x ^ 1, S.kv[i], __ldg(&p.arc[S.rs[i] + e]));
                    }
                    __syncwarp();
                    // long rows: a warp each
                    for (uint32_t i = tid >> 5; i < m; i += TPB / 32) {
                        const uint32_t d = S.deg[i];
                        if (d <= GROUP_DEGREE) continue;
                        for (uint32_t e = lane; e < d && !peek(S.over); e += 32)
                            relax(p, S, c, x ^ 1, S.kv[i], __ldg(&p.arc[S.rs[i] + e]));
                    }
                    __syncthreads();
                }
                if (S.over || S.stop) break;
                if (++rounds > p.round_limit) {
                    if (tid == 0) atomicExch(&p.flags[0], ERR_ROUND_LIMIT);
                    break;
                }
                n_pend = c.n_next;
                if (!n_pend) break;
                entered = c.minb > b;
                buckets += entered;
                b = c.minb;
                x ^= 1;
                r ^= 1;
            }
        } else if (tid == 0) {
            S.over = 1;
        }
        __syncthreads();
        if (S.over || S.stop) {
            for (int i = tid; i < SLOTS; i += TPB) {
                S.id[i] = EMPTY;
                S.key[i] = key_inf<K>();
            }
            if (S.stop) break;
            if (tid == 0) spill[atomicAdd(spill_n, 1u)] = h;
            continue;
        }
        ++n_trees;
        n_rounds += rounds;
        n_buckets += buckets;
        if (lane == 0) {
            n_exp += S.n_exp[tid >> 5];
            n_arcs += S.n_arcs[tid >> 5];
            n_pruned += S.n_pruned[tid >> 5];
        }
        // ---- emission: count, reserve the tree's output range, write, reset
        const uint32_t nt = S.n_touch;
        uint32_t mine = 0, far = 0;
        for (uint32_t i = tid; i < nt; i += TPB) {
            const uint32_t s = S.touch[i];
            const KS k = S.key[s];
            const bool on = is_live<K>(k, pos_at<K>(p, S.id[s] & ID_MASK), h);
            mine += on;
            if (on) far = max(far, key_dist<K>(k));
        }
        mine = __reduce_add_sync(FULL, mine);
        far = __reduce_max_sync(FULL, far);
        if (lane == 0 && mine) {
            atomicAdd(&S.n_out, mine);
            atomicMax(&S.max_d, far);
        }
        __syncthreads();
        if (tid == 0) {
            const uint32_t nlab = S.n_out;
            const unsigned long long old = atomicAdd(p.out_count, (unsigned long long)nlab);
            S.ok = old + nlab <= p.out_cap;
            S.base = old;
            if (!S.ok) {
                // nlab >= 1 (the root), so only the first range past the end starts within it
                if (old <= p.out_cap) *p.out_valid = old;
                p.failed[atomicAdd(p.failed_count, 1u)] = h;
                atomicExch(&p.flags[1], 1);
            }
        }
        __syncthreads();
        const bool ok = S.ok;
        const unsigned long long base = S.base;
        for (uint32_t i0 = tid - lane; i0 < nt; i0 += TPB) {
            const uint32_t i = i0 + lane;
            bool on = false;
            uint32_t v = 0;
            KS k = 0;
            if (i < nt) {
                const uint32_t s = S.touch[i];
                v = S.id[s] & ID_MASK;
                k = S.key[s];
                on = ok && is_live<K>(k, pos_at<K>(p, v), h);
                S.id[s] = EMPTY;
                S.key[s] = key_inf<K>();
            }
            const unsigned m = __ballot_sync(FULL, on);
            if (!m) continue;
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(&S.n_put, uint32_t(__popc(m)));
            at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1));
            if (on) {
                p.out_v[base + at] = caller_id<K>(p, v);
                p.out_h[base + at] = h;
                p.out_d[base + at] = key_dist<K>(k);
                if (p.out_p) p.out_p[base + at] = __ldg(&p.vert_at[key_parent<K>(k)]);
            }
        }
    }
    if (lane == 0) {
        if (n_exp) atomicAdd(&p.stats[0], n_exp);
        if (n_arcs) atomicAdd(&p.stats[1], n_arcs);
        if (n_pruned) atomicAdd(&p.stats[6], n_pruned);
    }
    if (tid == 0) {
        atomicAdd(&p.stats[3], n_trees);
        atomicAdd(&p.stats[4], n_rounds);
        atomicAdd(&p.stats[5], n_buckets);
        atomicMax(&p.stats[7], (unsigned long long)S.max_d);
    }
}

// The classes: threads and slots. Few slots put more trees on an SM.
template <int TPB, int SLOTS, typename K>
cudaError_t launch_class(const TreeLaunch &p, uint32_t max_trees, uint32_t *spill, unsigned int *spill_n,
                         cudaStream_t s) {
    using TR = Tree<TPB, SLOTS, K>;
    const size_t bytes = p.lt_off ? sizeof(TR) : offsetof(TR, lth_key);
    cudaError_t e = cudaFuncSetAttribute(plant_small_kernel<TPB, SLOTS, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(sizeof(TR)));
    if (e) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, plant_small_kernel<TPB, SLOTS, K>, TPB, bytes);
    if (e) return e;
    const uint32_t most = uint32_t(device_sms()) * uint32_t(per_sm > 0 ? per_sm : 1);
    const uint32_t ctas = max_trees < most ? max_trees : most;
    plant_small_kernel<TPB, SLOTS, K><<<ctas, TPB, bytes, s>>>(p, spill, spill_n);
    return cudaGetLastError();
}

template <int TPB, int SLOTS>
cudaError_t launch_key(const TreeLaunch &p, uint32_t max_trees, uint32_t *spill, unsigned int *spill_n,
                       cudaStream_t s) {
    if (p.pos)
        return p.out_p            ? launch_class<TPB, SLOTS, ById<KeyP>>(p, max_trees, spill, spill_n, s)
               : p.key_bytes == 4 ? launch_class<TPB, SLOTS, ById<KeyN>>(p, max_trees, spill, spill_n, s)
                                  : launch_class<TPB, SLOTS, ById<KeyW>>(p, max_trees, spill, spill_n, s);
    if (p.out_p) return launch_class<TPB, SLOTS, KeyP>(p, max_trees, spill, spill_n, s);
    if (p.key_bytes == 4) return launch_class<TPB, SLOTS, KeyN>(p, max_trees, spill, spill_n, s);
    return launch_class<TPB, SLOTS, KeyW>(p, max_trees, spill, spill_n, s);
}

}  // namespace

cudaError_t launch_plant_small(const TreeLaunch &p, int cls, uint32_t max_trees, uint32_t *spill,
                               unsigned int *spill_n, cudaStream_t s) {
    if (!max_trees) return cudaSuccess;
    switch (cls) {
        case 0: return launch_key<SMALL_THREADS[0], SMALL_SLOTS[0]>(p, max_trees, spill, spill_n, s);
        case 1: return launch_key<SMALL_THREADS[1], SMALL_SLOTS[1]>(p, max_trees, spill, spill_n, s);
        case 2: return launch_key<SMALL_THREADS[2], SMALL_SLOTS[2]>(p, max_trees, spill, spill_n, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace chl
