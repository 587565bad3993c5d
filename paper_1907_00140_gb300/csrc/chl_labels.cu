// Label assembly: from the (vertex, hub, dist) records the trees emit, in
// whatever order the trees finished, to per-vertex lists sorted by hub rank
// (Algorithm 2, "sort labels in L_v using hub rank"; the lists are stored
// per vertex only, as in the footnote of Sec. 7.2).
//
//   1. count labels per vertex (atomic histogram)
//   2. exclusive scan -> offsets
//   3. scatter (hubpos << 32 | dist) into each vertex's segment
//   4. sort every segment by hubpos (= descending R of the hub) and write it to
//      the hub (caller id), hubpos and dist arrays: one warp per segment up to
//      1024 labels (bitonic networks in registers), one CTA per segment up to
//      MAX_SEGMENT labels (in shared memory); a longer segment (one CTA each) is
//      sorted in chunks in shared memory, then the sorted runs are merged
//      pairwise in global memory
#include "chl_common.cuh"

namespace chl {

cudaError_t exclusive_scan_u64(const uint64_t *in, uint64_t *out, uint64_t n, cudaStream_t s,
                               int *launches);

namespace {

constexpr uint32_t MAX_SEGMENT = 16384;  // longest segment sorted in shared memory at once
constexpr uint32_t LONG_CHUNK = 4096;    // chunk of a longer segment sorted in shared memory

__global__ void count_kernel(uint64_t T, const uint32_t *v, uint64_t *cnt) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x)
        atomicAdd((unsigned long long *)&cnt[v[i]], 1ull);
}

// unsorted table by rank position: (hubpos, dist) straight into each
// vertex's segment; records of hubs below min_hub are left out (the dense
// Common Label Table answers for those hubs)
__global__ void count_table_kernel(uint64_t T, const uint32_t *v, const uint32_t *h,
                                   const uint32_t *index_of, uint32_t min_hub, uint64_t *cnt) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x)
        if (h[i] >= min_hub) atomicAdd((unsigned long long *)&cnt[index_of ? index_of[v[i]] : v[i]], 1ull);
}

// the entries of a label table in either form
struct TableEntries {
    uint2 *e;
    uint32_t *w;
    int db;
    explicit TableEntries(const LabelTable &t) : e(t.e), w(t.w), db(t.db) {}
    __device__ __forceinline__ void put(uint64_t k, uint32_t hub, uint32_t dist) const {
        if (db) w[k] = hub << db | dist;
        else e[k] = make_uint2(hub, dist);
    }
    __device__ __forceinline__ uint2 get(uint64_t k) const {
        if (!db) return e[k];
        const uint32_t x = w[k];
        return make_uint2(x >> db, x & ((1u << db) - 1));
    }
};

__global__ void scatter_table_kernel(uint64_t T, const uint32_t *v, const uint32_t *h,
                                     const uint32_t *d, const uint32_t *index_of, uint32_t min_hub,
                                     const uint64_t *off, uint64_t *fill, TableEntries e) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x) {
        if (h[i] < min_hub) continue;
        const uint32_t x = index_of ? index_of[v[i]] : v[i];
        const uint64_t k = off[x] + atomicAdd((unsigned long long *)&fill[x], 1ull);
        e.put(k, h[i], d[i]);
    }
}

// entries per vertex of the grown table: its old entries plus the new ones
__global__ void grown_count_kernel(uint32_t n, const uint64_t *old_off, uint64_t *cnt) {
    for (uint64_t v = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < n;
         v += uint64_t(gridDim.x) * blockDim.x)
        cnt[v] += old_off[v + 1] - old_off[v];
}

// one warp per vertex: its old entries to the front of its new segment
__global__ void copy_segments_kernel(uint32_t n, const uint64_t *old_off, TableEntries old_e,
                                     const uint64_t *new_off, TableEntries e) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t v = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint64_t a = old_off[v], len = old_off[v + 1] - a, o = new_off[v];
        for (uint64_t i = lane; i < len; i += 32) {
            const uint2 x = old_e.get(a + i);
            e.put(o + i, x.x, x.y);
        }
    }
}

// new records after each vertex's old entries
__global__ void scatter_new_kernel(uint64_t T0, uint64_t T, const uint32_t *v, const uint32_t *h,
                                   const uint32_t *d, const uint32_t *index_of, uint32_t min_hub,
                                   const uint64_t *old_off, const uint64_t *off, uint64_t *fill,
                                   TableEntries e) {
    for (uint64_t i = T0 + uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x) {
        if (h[i] < min_hub) continue;
        const uint32_t x = index_of ? index_of[v[i]] : v[i];
        const uint64_t k = off[x] + (old_off[x + 1] - old_off[x]) +
                           atomicAdd((unsigned long long *)&fill[x], 1ull);
        e.put(k, h[i], d[i]);
    }
}

__global__ void scatter_kernel(uint64_t T, const uint32_t *v, const uint32_t *h, const uint32_t *d,
                               const uint64_t *off, uint64_t *fill, uint64_t *tmp) {
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t x = v[i];
        const uint64_t k = off[x] + atomicAdd((unsigned long long *)&fill[x], 1ull);
        tmp[k] = (uint64_t(h[i]) << 32) | d[i];
    }
}

// Segments by length: warp classes of up to 32, 128, 256, 512 and 1024 labels,
// then one CTA's shared memory, then longer ones
constexpr int CLASSES = 7, BIG = 5, LONG = 6;
struct SortLists {
    uint32_t *list;    // CLASSES lists of n vertices
    uint32_t *counts;  // CLASSES counters
    uint32_t n;
    __device__ __forceinline__ const uint32_t *of(int c) const { return list + size_t(c) * n; }
};

// work lists of the segments that hold labels; records the longest
__global__ void classify_kernel(SortLists w, const uint64_t *off, unsigned long long *max_len) {
    const int lane = threadIdx.x & 31;
    unsigned long long most = 0;
    for (uint64_t v0 = uint64_t(blockIdx.x) * blockDim.x + (threadIdx.x - lane); v0 < w.n;
         v0 += uint64_t(gridDim.x) * blockDim.x) {
        const uint64_t v = v0 + lane;
        const uint64_t len = v < w.n ? off[v + 1] - off[v] : 0;
        most = len > most ? len : most;
        const int c = len == 0 ? -1 : len <= 32 ? 0 : len <= 128 ? 1 : len <= 256 ? 2 : len <= 512 ? 3
                      : len <= 1024 ? 4 : len <= MAX_SEGMENT ? BIG : LONG;
        const unsigned m = __match_any_sync(0xffffffffu, c);
        const int leader = __ffs(m) - 1;
        uint32_t b = 0;
        if (c >= 0 && lane == leader) b = atomicAdd(&w.counts[c], uint32_t(__popc(m)));
        b = __shfl_sync(0xffffffffu, b, leader);
        if (c >= 0) w.list[size_t(c) * w.n + b + __popc(m & ((1u << lane) - 1))] = uint32_t(v);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, most, o);
        most = x > most ? x : most;
    }
    if (lane == 0 && most) atomicMax(max_len, most);
}

// the label arrays a sorted segment is written to
struct SortOut {
    const uint32_t *vert_at;
    uint32_t *hub, *hubpos, *dist;
    __device__ __forceinline__ void put(uint64_t i, uint64_t k) const {
        const uint32_t hp = uint32_t(k >> 32);
        hubpos[i] = hp;
        dist[i] = uint32_t(k);
        hub[i] = __ldg(&vert_at[hp]);
    }
};

// One warp sorts a segment of at most 32 * E keys (hubpos, dist) in registers:
// lane l holds elements l * E .. l * E + E - 1 of the bitonic network, so only
// the strides of E and more cross lanes (15 of 45 stages at 512 keys). The
// sorted elements pass through shared memory, padded by one per lane, so that
// they are written coalesced. buf: 32 * (E + 1) words of 8 bytes.
//
// Bound by instruction issue (about 3,000 warp instructions per 512 keys); the
// network in shared memory with one CTA per segment that it replaces ran 45
// stages with a barrier each.
template <int E>
__device__ __forceinline__ void sort_warp(uint32_t v, const uint64_t *off, const uint64_t *tmp, const SortOut &out,
                                          uint64_t *buf) {
    const int lane = threadIdx.x & 31;
    const uint64_t a = off[v];
    const uint32_t len = uint32_t(off[v + 1] - a);
    uint32_t h[E], d[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const uint32_t i = uint32_t(j) * 32 + lane;  // any order: the keys are unsorted
        const uint64_t k = i < len ? __ldg(&tmp[a + i]) : ~0ull;
        h[j] = uint32_t(k >> 32);
        d[j] = uint32_t(k);
    }
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
        for (int s = k >> 1; s > 0; s >>= 1) {
            if (s < E) {
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const int q = j ^ s;
                    if (q < j) continue;
                    const bool up = k < E ? (j & k) == 0 : (lane & (k / E)) == 0;
                    const bool swap = (h[j] > h[q]) == up;  // (equal only among fillers)
                    const uint32_t hj = swap ? h[q] : h[j], hq = swap ? h[j] : h[q];
                    const uint32_t dj = swap ? d[q] : d[j], dq = swap ? d[j] : d[q];
                    h[j] = hj;
                    h[q] = hq;
                    d[j] = dj;
                    d[q] = dq;
                }
            } else {
                const int m = s / E;
                const bool low = ((lane & m) == 0) == ((lane & (k / E)) == 0);  // keeps the smaller
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const uint32_t oh = __shfl_xor_sync(0xffffffffu, h[j], m);
                    const uint32_t od = __shfl_xor_sync(0xffffffffu, d[j], m);
                    if ((oh < h[j]) == low) {
                        h[j] = oh;
                        d[j] = od;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < E; ++j) buf[lane * (E + 1) + j] = uint64_t(h[j]) << 32 | d[j];
    __syncwarp();
    for (uint32_t i = lane; i < len; i += 32) out.put(a + i, buf[i + i / E]);
    __syncwarp();  // the next segment reuses the buffer
}

constexpr int SORT_TPB = 128;

// segments of up to 256 labels (classes 0 to 2), the longest class first
__global__ void __launch_bounds__(SORT_TPB) sort_short_kernel(SortLists w, const uint64_t *off, const uint64_t *tmp,
                                                              SortOut out) {
    __shared__ uint64_t buf[SORT_TPB / 32][32 * 9];
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5, me = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t c2 = w.counts[2], c1 = c2 + w.counts[1], c0 = c1 + w.counts[0];
    uint64_t *b = buf[threadIdx.x >> 5];
    for (uint32_t i = me; i < c0; i += warps) {
        if (i < c2) sort_warp<8>(w.of(2)[i], off, tmp, out, b);
        else if (i < c1) sort_warp<4>(w.of(1)[i - c2], off, tmp, out, b);
        else sort_warp<1>(w.of(0)[i - c1], off, tmp, out, b);
    }
}

// segments of 257 to 1024 labels (classes 3 and 4), the longest class first
__global__ void __launch_bounds__(SORT_TPB) sort_mid_kernel(SortLists w, const uint64_t *off, const uint64_t *tmp,
                                                            SortOut out) {
    __shared__ uint64_t buf[SORT_TPB / 32][32 * 33];
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5, me = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t c4 = w.counts[4], c3 = c4 + w.counts[3];
    uint64_t *b = buf[threadIdx.x >> 5];
    for (uint32_t i = me; i < c3; i += warps) {
        if (i < c4) sort_warp<32>(w.of(4)[i], off, tmp, out, b);
        else sort_warp<16>(w.of(3)[i - c4], off, tmp, out, b);
    }
}

// One CTA per segment longer than MAX_SEGMENT: its chunks of LONG_CHUNK keys
// are sorted in shared memory (bitonic), then runs of width w, 2w, 4w, ...
// are merged pairwise between tmp and tmp2 (each thread writes an equal share
// of a merged pair, starting where the merge path of its first output crosses
// the two runs); the sorted segment goes to the label arrays. Keys (hubpos << 32 | dist)
// are distinct within a segment (one label per hub), so the order is unique.
__global__ void __launch_bounds__(1024) sort_long_kernel(const uint32_t *list, const uint32_t *count,
                                                         const uint64_t *off, uint64_t *tmp,
                                                         uint64_t *tmp2, SortOut out) {
    __shared__ uint64_t sm[LONG_CHUNK];
    const uint32_t tid = threadIdx.x, nt = blockDim.x;
    for (uint32_t sidx = blockIdx.x; sidx < *count; sidx += gridDim.x) {
        const uint32_t v = list[sidx];
        const uint64_t a = off[v], len = off[v + 1] - a;
        for (uint64_t c0 = 0; c0 < len; c0 += LONG_CHUNK) {
            const uint32_t cl = uint32_t(len - c0 < LONG_CHUNK ? len - c0 : LONG_CHUNK);
            for (uint32_t i = tid; i < LONG_CHUNK; i += nt) sm[i] = i < cl ? tmp[a + c0 + i] : ~0ull;
            __syncthreads();
            for (uint32_t k = 2; k <= LONG_CHUNK; k <<= 1) {
                for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                    for (uint32_t i = tid; i < LONG_CHUNK; i += nt) {
                        const uint32_t ix = i ^ j;
                        if (ix > i) {
                            const uint64_t x = sm[i], y = sm[ix];
                            if ((x > y) == ((i & k) == 0)) {
                                sm[i] = y;
                                sm[ix] = x;
                            }
                        }
                    }
                    __syncthreads();
                }
            }
            for (uint32_t i = tid; i < cl; i += nt) tmp[a + c0 + i] = sm[i];
            __syncthreads();
        }
        uint64_t *src = tmp + a, *dst = tmp2 + a;
        for (uint64_t w = LONG_CHUNK; w < len; w *= 2) {
            for (uint64_t p0 = 0; p0 < len; p0 += 2 * w) {
                const uint64_t na = len - p0 < w ? len - p0 : w;
                const uint64_t nb = len - p0 > w ? (len - p0 - w < w ? len - p0 - w : w) : 0;
                const uint64_t m = na + nb;
                const uint64_t *A = src + p0, *B = A + na;
                const uint64_t k0 = m * tid / nt, k1 = m * (tid + 1) / nt;
                if (k0 >= k1) continue;
                // i = keys of A among the first k0 outputs (smallest i with A[i] > B[k0 - i - 1])
                uint64_t lo = k0 > nb ? k0 - nb : 0, hi = k0 < na ? k0 : na;
                while (lo < hi) {
                    const uint64_t mid = (lo + hi) >> 1;
                    if (A[mid] <= B[k0 - mid - 1]) lo = mid + 1; else hi = mid;
                }
                uint64_t i = lo, j = k0 - lo;
                for (uint64_t k = k0; k < k1; ++k) {
                    const bool take_a = j >= nb || (i < na && A[i] <= B[j]);
                    dst[p0 + k] = take_a ? A[i++] : B[j++];
                }
            }
            __syncthreads();
            uint64_t *t = src;
            src = dst;
            dst = t;
        }
        for (uint64_t i = tid; i < len; i += nt) out.put(a + i, src[i]);
        __syncthreads();
    }
}

// one CTA per segment: bitonic sort in shared memory (size rounded up to a power of two)
constexpr int BLOCK_TPB = 1024;
__global__ void __launch_bounds__(BLOCK_TPB) sort_block_kernel(const uint32_t *list, const uint32_t *count,
                                                               const uint64_t *off, const uint64_t *tmp,
                                                               SortOut out) {
    constexpr int TPB = BLOCK_TPB;
    extern __shared__ uint64_t sm[];
    for (uint32_t s = blockIdx.x; s < *count; s += gridDim.x) {
        const uint32_t v = list[s];
        const uint64_t a = off[v];
        const uint32_t len = uint32_t(off[v + 1] - a);
        uint32_t P = 1;
        while (P < len) P <<= 1;
        for (uint32_t i = threadIdx.x; i < P; i += TPB) sm[i] = i < len ? tmp[a + i] : ~0ull;
        __syncthreads();
        for (uint32_t k = 2; k <= P; k <<= 1) {
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t i = threadIdx.x; i < P; i += TPB) {
                    const uint32_t ix = i ^ j;
                    if (ix > i) {
                        const uint64_t x = sm[i], y = sm[ix];
                        const bool up = ((i & k) == 0);
                        if ((x > y) == up) {
                            sm[i] = y;
                            sm[ix] = x;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (uint32_t i = threadIdx.x; i < len; i += TPB) out.put(a + i, sm[i]);
        __syncthreads();
    }
}

int grid_for(uint64_t work, int tpb) {
    uint64_t b = (work + tpb - 1) / tpb;
    const uint64_t cap = uint64_t(device_sms()) * 32;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return int(b);
}

}  // namespace

#define CKE(x)                                   \
    do {                                         \
        e = (x);                                 \
        if (e != cudaSuccess) goto done;         \
    } while (0)

cudaError_t assemble_labels(uint32_t n, uint64_t T, const uint32_t *in_v, const uint32_t *in_h,
                            const uint32_t *in_d, const uint32_t *vert_at, LabelCSR &out,
                            int *too_long, cudaStream_t s, int *launches) {
    cudaError_t e = cudaSuccess;
    uint64_t *cnt = nullptr, *tmp = nullptr, *tmp2 = nullptr;
    uint32_t *lists = nullptr, *counts = nullptr;
    unsigned long long *maxlen = nullptr;
    unsigned long long hmax = 0;
    const int sms = device_sms();
    *too_long = 0;
    out = LabelCSR{};
    const size_t Tb = (T ? T : 1);
    CKE(dmalloc(&out.offsets, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(dmalloc(&out.hub, Tb * sizeof(uint32_t), s));
    CKE(dmalloc(&out.hubpos, Tb * sizeof(uint32_t), s));
    CKE(dmalloc(&out.dist, Tb * sizeof(uint32_t), s));
    CKE(dmalloc(&cnt, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(dmalloc(&tmp, Tb * sizeof(uint64_t), s));
    CKE(dmalloc(&lists, CLASSES * size_t(n) * sizeof(uint32_t), s));
    CKE(dmalloc(&counts, CLASSES * sizeof(uint32_t), s));
    CKE(dmalloc(&maxlen, sizeof(unsigned long long), s));
    CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(cudaMemsetAsync(counts, 0, CLASSES * sizeof(uint32_t), s));
    CKE(cudaMemsetAsync(maxlen, 0, sizeof(unsigned long long), s));
    count_kernel<<<grid_for(T, 256), 256, 0, s>>>(T, in_v, cnt);
    *launches += 1;
    CKE(cudaGetLastError());
    CKE(exclusive_scan_u64(cnt, out.offsets, uint64_t(n) + 1, s, launches));
    CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
    scatter_kernel<<<grid_for(T, 256), 256, 0, s>>>(T, in_v, in_h, in_d, out.offsets, cnt, tmp);
    {
        const SortLists w{lists, counts, n};
        const SortOut so{vert_at, out.hub, out.hubpos, out.dist};
        classify_kernel<<<grid_for(n, 256), 256, 0, s>>>(w, out.offsets, maxlen);
        *launches += 2;
        CKE(cudaGetLastError());
        sort_short_kernel<<<sms * 8, SORT_TPB, 0, s>>>(w, out.offsets, tmp, so);
        *launches += 1;
        if (n > 256) {  // (a list holds at most n labels)
            sort_mid_kernel<<<sms * 4, SORT_TPB, 0, s>>>(w, out.offsets, tmp, so);
            *launches += 1;
        }
        CKE(cudaGetLastError());
        if (n > 1024) {
            CKE(cudaMemcpyAsync(&hmax, maxlen, sizeof(hmax), cudaMemcpyDeviceToHost, s));
            CKE(cudaStreamSynchronize(s));
        }
        if (hmax > 1024) {
            // the attribute belongs to the current device: set on every call
            CKE(cudaFuncSetAttribute(sort_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     int(MAX_SEGMENT * sizeof(uint64_t))));
            sort_block_kernel<<<sms, BLOCK_TPB, MAX_SEGMENT * sizeof(uint64_t), s>>>(
                lists + BIG * size_t(n), counts + BIG, out.offsets, tmp, so);
            *launches += 1;
        }
        if (hmax > MAX_SEGMENT) {
            CKE(dmalloc(&tmp2, Tb * sizeof(uint64_t), s));
            sort_long_kernel<<<sms, 1024, 0, s>>>(lists + LONG * size_t(n), counts + LONG, out.offsets, tmp, tmp2, so);
            *launches += 1;
        }
        CKE(cudaGetLastError());
    }
done:
    if (cnt) cudaFreeAsync(cnt, s);
    if (tmp) cudaFreeAsync(tmp, s);
    if (tmp2) cudaFreeAsync(tmp2, s);
    if (lists) cudaFreeAsync(lists, s);
    if (counts) cudaFreeAsync(counts, s);
    if (maxlen) cudaFreeAsync(maxlen, s);
    if (e != cudaSuccess || *too_long) {
        if (out.offsets) cudaFreeAsync(out.offsets, s);
        if (out.hub) cudaFreeAsync(out.hub, s);
        if (out.hubpos) cudaFreeAsync(out.hubpos, s);
        if (out.dist) cudaFreeAsync(out.dist, s);
        out = LabelCSR{};
    }
    return e;
}

static cudaError_t alloc_entries(LabelTable &t, uint64_t T, int db, cudaStream_t s) {
    t.db = db;
    return db ? dmalloc(&t.w, (size_t(T) + 2) * sizeof(uint32_t), s) : dmalloc(&t.e, (size_t(T) + 2) * sizeof(uint2), s);
}

// Entries are allocated with two spare ones past the last, so that a read
// widened to 16-byte boundaries (two entries) stays inside the array.
cudaError_t assemble_table(uint32_t n, uint64_t T, const uint32_t *in_v, const uint32_t *in_h,
                           const uint32_t *in_d, const uint32_t *index_of, uint32_t min_hub,
                           int db, LabelTable &out, cudaStream_t s, int *launches) {
    cudaError_t e = cudaSuccess;
    uint64_t *cnt = nullptr;
    out = LabelTable{};
    CKE(dmalloc(&out.offsets, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(alloc_entries(out, T, db, s));
    CKE(dmalloc(&cnt, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
    count_table_kernel<<<grid_for(T, 256), 256, 0, s>>>(T, in_v, in_h, index_of, min_hub, cnt);
    *launches += 1;
    CKE(cudaGetLastError());
    CKE(exclusive_scan_u64(cnt, out.offsets, uint64_t(n) + 1, s, launches));
    CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
    scatter_table_kernel<<<grid_for(T, 256), 256, 0, s>>>(T, in_v, in_h, in_d, index_of, min_hub,
                                                          out.offsets, cnt, TableEntries(out));
    *launches += 1;
    CKE(cudaGetLastError());
done:
    if (cnt) cudaFreeAsync(cnt, s);
    if (e != cudaSuccess) {
        free_table(out, s);
    }
    return e;
}

cudaError_t grow_table(uint32_t n, LabelTable &lt, uint64_t T0, uint64_t T, const uint32_t *in_v,
                       const uint32_t *in_h, const uint32_t *in_d, const uint32_t *index_of,
                       uint32_t min_hub, int db, cudaStream_t s, int *launches, LabelTable *keep_old) {
    cudaError_t e = cudaSuccess;
    uint64_t *cnt = nullptr;
    LabelTable out;
    const uint64_t dT = T - T0;
    CKE(dmalloc(&out.offsets, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(alloc_entries(out, T, db, s));
    CKE(dmalloc(&cnt, (size_t(n) + 1) * sizeof(uint64_t), s));
    CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
    if (dT) {
        count_table_kernel<<<grid_for(dT, 256), 256, 0, s>>>(dT, in_v + T0, in_h + T0, index_of, min_hub,
                                                             cnt);
        *launches += 1;
    }
    grown_count_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, lt.offsets, cnt);
    *launches += 1;
    CKE(cudaGetLastError());
    CKE(exclusive_scan_u64(cnt, out.offsets, uint64_t(n) + 1, s, launches));
    copy_segments_kernel<<<grid_for(uint64_t(n) * 32, 256), 256, 0, s>>>(n, lt.offsets, TableEntries(lt),
                                                                         out.offsets, TableEntries(out));
    *launches += 1;
    CKE(cudaGetLastError());
    if (dT) {
        CKE(cudaMemsetAsync(cnt, 0, (size_t(n) + 1) * sizeof(uint64_t), s));
        scatter_new_kernel<<<grid_for(dT, 256), 256, 0, s>>>(T0, T, in_v, in_h, in_d, index_of, min_hub,
                                                             lt.offsets, out.offsets, cnt, TableEntries(out));
        *launches += 1;
        CKE(cudaGetLastError());
    }
done:
    if (cnt) cudaFreeAsync(cnt, s);
    if (e != cudaSuccess) {
        free_table(out, s);
        return e;
    }
    if (keep_old) {
        *keep_old = lt;  // still read by trees on another stream: the caller frees it after them
    } else {
        free_table(lt, s);
    }
    lt = out;
    return e;
}

void free_table(LabelTable &t, cudaStream_t s) {
    if (t.offsets) cudaFreeAsync(t.offsets, s);
    if (t.e) cudaFreeAsync(t.e, s);
    if (t.w) cudaFreeAsync(t.w, s);
    t = LabelTable{};
}

namespace {

// record i's parent goes to the slot of its hub in its vertex's sorted list
// (hub positions are unique within a list)
__global__ void place_parents_kernel(uint64_t T, const uint32_t *in_v, const uint32_t *in_h,
                                     const uint32_t *in_p, const uint64_t *off,
                                     const uint32_t *hubpos, uint32_t *parent) {
    for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < T;
         i += uint64_t(gridDim.x) * blockDim.x) {
        const uint32_t v = in_v[i], hp = in_h[i];
        uint64_t lo = off[v], hi = off[v + 1];  // hubpos[lo..hi) ascending, contains hp
        while (hi - lo > 1) {
            const uint64_t mid = (lo + hi) >> 1;
            if (hubpos[mid] <= hp) lo = mid; else hi = mid;
        }
        parent[lo] = in_p[i];
    }
}

}  // namespace

cudaError_t place_parents(uint64_t T, const uint32_t *in_v, const uint32_t *in_h, const uint32_t *in_p,
                          const LabelCSR &csr, uint32_t *parent, cudaStream_t s, int *launches) {
    if (!T) return cudaSuccess;
    place_parents_kernel<<<grid_for(T, 256), 256, 0, s>>>(T, in_v, in_h, in_p, csr.offsets,
                                                           csr.hubpos, parent);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace chl
