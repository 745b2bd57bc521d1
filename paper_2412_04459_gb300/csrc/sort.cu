// Render work order and the sort of each tile's pairs by (key, value).
//
// The tile id is the most significant part of a key and is sorted by
// counting: the scan of the per-tile counts gives every tile its range and
// k_emit writes each pair into its tile's range (order within a tile
// arbitrary).  Each tile's list is then sorted by the Morton bits that can
// differ:
//   k_order        the render work order: one entry per tile, or per
//                  1024-entry segment of a longer list, longest first; and
//                  the lists of each length class for the sort
//   k_sort_lists   every list of up to kSortCap pairs, and every
//                  kSortCap-pair chunk of a longer one, by a merge sort in
//                  shared memory, each by a group of threads of its size
//   k_merge_long   the sorted chunks of longer lists, merged in rounds of
//                  pairwise merges, one thread-block cluster per list
//
// Where the parts of a pair fit 64 bits (Morton bits that can differ, sign
// pattern, voxel id: every scene up to level 12 of fewer than 2^25 voxels, or
// level 14 of fewer than 2^19) pairs are emitted, sorted and merged as one word each and become
// (key, value) on the last write; otherwise the sort moves (Morton bits,
// index in the list) words and the merge whole pairs.
#include "svr_internal.cuh"

namespace svr {

// ------------------------------------------------------------------- order

// Chunks of a list and merge rounds over them.
__device__ __forceinline__ int list_chunks(int L) { return (L + kSortCap - 1) / kSortCap; }
__device__ __forceinline__ int merge_rounds(int chunks) { return chunks > 1 ? 32 - __clz(chunks - 1) : 0; }

constexpr int kOrderThreads = 256;

// Places every tile's entries in the work order (k_scan_down counted them
// per group; the order within a group is arbitrary and results do not depend
// on it): each CTA counts its tiles' entries per group in shared memory and
// reserves them with one atomic per group.  One CTA alone took 9 us for the
// 4,240 tiles of a 1280 x 840 view and 118 us for 115,200 tiles.  CTA 0 also
// writes the queue's counts and the sort classes.
__global__ void __launch_bounds__(kOrderThreads) k_order(FrameDev f) {
    begin_kernel();
    constexpr int G = 2 * kOrderGroups;
    __shared__ unsigned cnt[G], start[G], mine[G];
    const int t = threadIdx.x, i = blockIdx.x * kOrderThreads + t;
    if (t < G) {
        cnt[t] = f.plan->cnt[t];
        mine[t] = 0u;
    }
    __syncthreads();
    if (t < G) {   // groups from the last to the first
        unsigned acc = 0;
        for (int b = G - 1; b > t; --b) acc += cnt[b];
        start[t] = acc;
    }
    const bool valid = i < f.total_tiles;
    const uint2 rg = valid ? f.ranges[i] : make_uint2(0u, 0u);
    const uint2 ts = valid ? f.tile_seg[i] : make_uint2(0u, 0u);
    const int L = (int)(rg.y - rg.x);
    const int bk = order_bucket((unsigned)L, ts.x);
    unsigned p0 = 0, p1 = 0;   // places among this CTA's entries of the tile's groups
    if (valid) {
        p0 = atomicAdd(&mine[ts.x > 1 ? kFirstSeg + bk : bk], 1u);
        if (ts.x > 1) p1 = atomicAdd(&mine[bk], ts.x - 1);
    }
    __syncthreads();
    if (t < G && mine[t]) mine[t] = start[t] + atomicAdd(&f.plan->pos[t], mine[t]);
    __syncthreads();
    if (valid) {
        f.order[mine[ts.x > 1 ? kFirstSeg + bk : bk] + p0] = make_uint2((unsigned)i, 0u);
        for (unsigned sg = 1; sg < ts.x; ++sg) f.order[mine[bk] + p1 + sg - 1] = make_uint2((unsigned)i, sg);
        if (ts.x > 1 && L >= kSortCap) {
            const int nc = list_chunks(L);
            const unsigned c0 = atomicAdd(&f.plan->n_chunks, (unsigned)nc);
            for (int c = 0; c < nc; ++c)
                if ((int64_t)c0 + c < sort_chunk_capacity(f.capacity)) f.chunks[c0 + c] = make_uint2((unsigned)i, (unsigned)c);
        }
    }
    if (blockIdx.x == 0 && t == 0) {
        f.status->n_queue = start[0] + cnt[0];
        f.status->n_listed = start[0];   // group 0 (the empty lists) is last
        f.status->fwd_done = 0;          // the segment sums belong to the last sort
        SortPlan *p = f.plan;
        p->n_huge = start[kFirstSeg + 14];   // first segments of lists of 2^13 pairs and more
        for (int c = 3; c < kSortClasses; ++c) {
            p->first[c] = start[kFirstSeg + c + 9];
            p->count[c] = cnt[kFirstSeg + c + 9];
        }
        p->first[2] = start[11];             // unsplit lists of 512 to 1024 pairs
        p->count[2] = cnt[11] + cnt[10];
        p->first[1] = start[9];
        p->count[1] = cnt[9];
        p->first[0] = start[8];
        p->count[0] = start[0] - start[8];
    }
}

// -------------------------------------------------------- per-tile merge sort
//
// A group of GT threads (32 .. 512, a power of two) sorts up to 16 GT words:
// 16 words per thread by a sorting network in registers, then rounds of
// pairwise merges through shared memory, each thread writing 16 consecutive
// outputs after a binary search for where they start (merge path).  About 230
// thread instructions per word for 8192 words; the LSD radix passes of 8-bit
// digits this replaces took 170 per pass and word (warp match, digit tables
// and six barriers a pass), four or five passes, on chunks of 1024 that were
// then merged serially.  The shared array leaves one word free after every 16
// (pad), so that threads at the same place of their 16 words fall in distinct
// banks.  What bounds it now: shared-memory latency of the serial merge steps.

constexpr int kSortThreads = 512;
constexpr int kSortVT = 16;
constexpr uint64_t kWordMax = ~0ull;
constexpr int kIdxBits = 16;   // low bits of an index word: the pair's place in its list or chunk
constexpr size_t kSortSmemBytes = (size_t)kSortCap / 16 * 17 * sizeof(uint64_t);

__device__ __forceinline__ int pad(int p) { return p + (p >> 4); }

// How pairs are sorted: whole words; or (Morton bits, index) words, equal
// Morton bits by value.  Two pairs of a tile have equal Morton bits at max level
// 16 (the rays of two sign patterns), and at any level where voxels overlap
// (one given twice, or with its first child), which no call refuses.  The order
// must then be by value too: the merges of long lists take their runs as sorted
// by (key, value), and from runs that are not they would place two pairs in one
// slot and leave another one unwritten.  Emission and sort of 1M voxels over
// 4,240 tiles: 114 us as words, 158 us as index words (declared as level 15).
constexpr int kWords = 0, kIndex = 1;

template <int MODE>
struct Less {
    const uint32_t *v;   // the list's values
    __device__ __forceinline__ bool operator()(uint64_t a, uint64_t b) const {
        if (MODE == kWords || ((a ^ b) >> kIdxBits) != 0 || a == kWordMax || b == kWordMax) return a < b;
        return v[a & 0xFFFFu] < v[b & 0xFFFFu];
    }
};

// Batcher's odd-even merge sort of VT words in registers: stages (P, K), in
// each the words K apart within blocks of 2 P (recursive, so that every index
// is a constant).
template <int VT, int P, int K, class L>
__device__ __forceinline__ void sort_stage(uint64_t (&x)[VT], const L &less) {
#pragma unroll
    for (int i = 0; i < VT - K; ++i)
        if (i >= K % P && (i - K % P) % (2 * K) < K && i / (2 * P) == (i + K) / (2 * P)) {
            const uint64_t a = x[i], b = x[i + K];
            const bool swap = less(b, a);
            x[i] = swap ? b : a;
            x[i + K] = swap ? a : b;
        }
    if constexpr (K > 1) sort_stage<VT, P, K / 2>(x, less);
    else if constexpr (2 * P < VT) sort_stage<VT, 2 * P, 2 * P>(x, less);
}

template <int VT, class L>
__device__ __forceinline__ void sort_network(uint64_t (&x)[VT], const L &less) {
    if constexpr (VT > 1) sort_stage<VT, 1, 1>(x, less);
}

// Barrier of the calling group: gt threads, group g of its CTA.
__device__ __forceinline__ void group_sync(int gt, int g) {
    if (gt == 32) __syncwarp();
    else if (gt == kSortThreads) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(gt) : "memory");
}

// VT outputs of the merge of sorted s[pad(a0..a1)) and s[pad(b0..b1)) from
// output k on; fewer are left if the runs end (then kWordMax).
template <int VT, class L>
__device__ __forceinline__ void merge_out(const uint64_t *s, int a0, int a1, int b0, int b1, int k, uint64_t (&x)[VT],
                                          const L &less) {
    int lo = max(0, k - (b1 - b0)), hi = min(k, a1 - a0);
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        // A[m] goes before B[k - 1 - m] unless B's is smaller
        if (less(s[pad(b0 + k - 1 - m)], s[pad(a0 + m)])) hi = m;
        else lo = m + 1;
    }
    int ia = a0 + lo, ib = b0 + k - lo;
    uint64_t a = ia < a1 ? s[pad(ia)] : kWordMax, b = ib < b1 ? s[pad(ib)] : kWordMax;
#pragma unroll
    for (int i = 0; i < VT; ++i) {
        const bool tb = less(b, a);
        x[i] = tb ? b : a;
        const int p = tb ? ++ib : ++ia;
        const uint64_t n = p < (tb ? b1 : a1) ? s[pad(p)] : kWordMax;
        if (tb) b = n;
        else a = n;
    }
}

// Sorts the group's VT gt words (thread t's x[i], in any order; kWordMax
// where there is none): on return s[pad(p)] holds the p-th smallest, visible
// to the group.
template <int VT, class L>
__device__ __forceinline__ void group_sort(uint64_t (&x)[VT], uint64_t *s, int t, int gt, int g, const L &less) {
    sort_network<VT>(x, less);
    const int o = t * VT;
    bool wide = false;   // whether the last merge read other warps' words
    for (int m = 1;; m *= 2) {   // runs of m threads' words
        const bool next_wide = m > 16;
        if (wide) group_sync(gt, g);
        else __syncwarp();
#pragma unroll
        for (int i = 0; i < VT; ++i) s[pad(o + i)] = x[i];
        const bool last = m >= gt;
        if (next_wide || last) group_sync(gt, g);
        else __syncwarp();
        if (last) return;
        const int p0 = (t & ~(2 * m - 1)) * VT, w = m * VT;
        merge_out<VT>(s, p0, p0 + w, p0 + w, p0 + 2 * w, o - p0, x, less);
        wide = next_wide;
    }
}

// One list (chunk < 0) or one chunk of a list: the n pairs from c0 of tile
// tile's range, sorted by a group and written as keys and values, or, for a
// chunk that will be merged (dst >= 0), into buffer dst in the merge's form.
template <int MODE, int VT>
__device__ __forceinline__ void sort_list(const FrameDev &f, uint64_t *s, int t, int gt, int g, int tile, uint32_t c0,
                                          int n, int dst) {
    uint64_t *gk = f.keys[0] + c0;
    uint32_t *gv = f.vals[0] + c0;
    const Less<MODE> less = {gv};
    const int lo_bit = f.key_shift - f.sort_bits;
    const uint64_t mask = (1ull << f.sort_bits) - 1ull;
    uint64_t x[VT];
#pragma unroll
    for (int i = 0; i < VT; ++i) {
        const int p = i * gt + t;
        uint64_t k = p < n ? gk[p] : kWordMax;
        if (MODE != kWords && p < n) k = (((k >> lo_bit) & mask) << kIdxBits) | (uint64_t)p;
        x[i] = k;
    }
    group_sort<VT>(x, s, t, gt, g, less);
    if (MODE == kWords) {
        if (dst >= 0) {
            for (int p = t; p < n; p += gt) f.keys[dst][c0 + p] = s[pad(p)];
        } else {
            for (int p = t; p < n; p += gt) {
                uint64_t k;
                uint32_t v;
                word_pair(f, tile, s[pad(p)], k, v);
                gk[p] = k;
                gv[p] = v;
            }
        }
    } else {
        uint32_t v[VT];
#pragma unroll
        for (int i = 0; i < VT; ++i) {
            const int p = i * gt + t;
            v[i] = p < n ? gv[s[pad(p)] & 0xFFFFu] : 0u;
        }
        group_sync(gt, g);   // every value is read before any is overwritten
        const int d = dst >= 0 ? dst : 0;
#pragma unroll
        for (int i = 0; i < VT; ++i) {
            const int p = i * gt + t;
            if (p >= n) continue;
            f.keys[d][c0 + p] = pair_key(f, tile, s[pad(p)] >> kIdxBits, v[i] >> 29);
            f.vals[d][c0 + p] = v[i];
        }
    }
    group_sync(gt, g);   // s is reused by the group's next list
}

// A persistent grid takes units from a counter, the longest first: a chunk of
// a long list or a list of class 5 (512 threads), 2 lists of class 4 (256
// threads each), 4 of class 3, 8 of class 2, 16 of class 1 or 0 (a warp each).
// So every list is sorted by about a sixteenth of its length in threads, and
// the short ones fill the tail.
template <int MODE>
__global__ void __launch_bounds__(kSortThreads, 2) k_sort_lists(FrameDev f) {
    begin_kernel();
    extern __shared__ __align__(16) unsigned char dyn[];
    uint64_t *smem = reinterpret_cast<uint64_t *>(dyn);
    __shared__ unsigned unit;
    const SortPlan *plan = f.plan;
    const unsigned n_chunks = min(plan->n_chunks, (unsigned)sort_chunk_capacity(f.capacity));
    for (;;) {
        if (threadIdx.x == 0) unit = atomicAdd(&f.plan->next, 1u);
        __syncthreads();
        unsigned u = unit;
        __syncthreads();
        // the group's list or chunk: n pairs from c0
        int gt = kSortThreads, n, dst = -1;
        unsigned tile;
        uint32_t c0;
        if (u < n_chunks) {
            const uint2 q = f.chunks[u];
            const uint2 rg = f.ranges[q.x];
            if (!SVR_IN_BOUNDS(f.debug, kDbgRange, rg.y, f.capacity + 1)) continue;
            const int L = (int)(rg.y - rg.x), first = (int)q.y * kSortCap;
            const int r = merge_rounds(list_chunks(L));
            if (r) dst = r & 1;   // the merge rounds alternate between the buffers and end in the first
            tile = q.x;
            c0 = rg.x + first;
            n = min(kSortCap, L - first);
        } else {
            u -= n_chunks;
            int c = kSortClasses - 1;
            for (; c >= 0; --c) {
                const int per = 16 >> (c > 0 ? c - 1 : 0);
                const unsigned units = (plan->count[c] + per - 1) / per;
                if (u < units) break;
                u -= units;
            }
            if (c < 0) return;
            gt = 32 << (c > 0 ? c - 1 : 0);
            const unsigned e = u * (kSortThreads / gt) + threadIdx.x / gt;
            if (e >= plan->count[c]) continue;
            tile = f.order[plan->first[c] + e].x;
            const uint2 rg = f.ranges[tile];
            if (!SVR_IN_BOUNDS(f.debug, kDbgRange, rg.y, f.capacity + 1)) continue;
            c0 = rg.x;
            n = (int)(rg.y - rg.x);
            // the class's longest list fits; one that did not would stay unsorted
            if (!SVR_IN_BOUNDS(f.debug, kDbgSortList, n, gt * kSortVT + 1) || n > gt * kSortVT) continue;
        }
        const int g = threadIdx.x / gt, t = threadIdx.x & (gt - 1);
        uint64_t *s = smem + (size_t)g * (gt / 16 * 17 * kSortVT);
        // as few words per thread as hold the list: a class's lists are half
        // to wholly as long as its longest, a long list's last chunk may be
        // short
        if (n <= gt) {
            if (n > 1 || MODE == kWords || dst >= 0) sort_list<MODE, 1>(f, s, t, gt, g, (int)tile, c0, n, dst);
        } else if (n <= 4 * gt) {
            sort_list<MODE, 4>(f, s, t, gt, g, (int)tile, c0, n, dst);
        } else if (n <= 8 * gt) {
            sort_list<MODE, 8>(f, s, t, gt, g, (int)tile, c0, n, dst);
        } else if (n <= 12 * gt) {
            sort_list<MODE, 12>(f, s, t, gt, g, (int)tile, c0, n, dst);
        } else {
            sort_list<MODE, kSortVT>(f, s, t, gt, g, (int)tile, c0, n, dst);
        }
    }
}

// ------------------------------------------------------------ long lists

constexpr int kMergeThreads = 512;
constexpr int kMergeVT = 8;
constexpr int kPiece = kMergeThreads * kMergeVT;   // outputs merged at a time by a CTA
static_assert(kSortCap % kPiece == 0, "a piece lies in one pair of runs");

__device__ __forceinline__ bool pair_less(uint64_t ka, uint32_t va, uint64_t kb, uint32_t vb) {
    return ka < kb || (ka == kb && va < vb);
}

// Outputs taken from run A among the first k of the merge of A (na) and B
// (nb), found by the whole warp: 32 probes per round (a run of 64K words
// costs four dependent loads).  Buffers are read through L2: other CTAs of
// the cluster wrote them in the round before.
template <bool WORDS>
__device__ __forceinline__ int merge_split(const uint64_t *ak, const uint32_t *av, int na, const uint64_t *bk,
                                           const uint32_t *bv, int nb, int k) {
    const int lane = threadIdx.x & 31;
    int lo = max(0, k - nb), hi = min(k, na);
    while (lo < hi) {
        const int s = (hi - lo + 31) >> 5;
        const int m = lo + (lane + 1) * s - 1;
        bool below = false;   // A[m] goes before B[k - 1 - m]
        if (m < hi) {
            const uint64_t a = __ldcg(ak + m), b = __ldcg(bk + k - 1 - m);
            below = WORDS ? !(b < a) : !pair_less(b, __ldcg(bv + k - 1 - m), a, __ldcg(av + m));
        }
        const int c = __popc(__ballot_sync(0xffffffffu, below));
        lo += s * c;
        hi = min(hi, lo + s - 1);
    }
    return lo;
}

// Lists of more than kSortCap pairs: their sorted chunks are merged pairwise
// in rounds between the two buffers, the last round into the first.  A
// cluster takes one list at a time; a round's outputs are cut
// into pieces of 4096, each merged in shared memory by one CTA (two searches
// for its ends, coalesced loads and stores), and the cluster barrier
// separates the rounds.  One CTA per list, merging in global memory by
// itself, took 48 us for a single list of 8,714 pairs and 3.1 ms for 46
// lists of up to 90,564.
template <bool WORDS, int CLUSTER>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(kMergeThreads, 2) k_merge_long(FrameDev f) {
    begin_kernel();
    __shared__ uint64_t sk[kPiece / 16 * 17];
    __shared__ uint32_t sv[WORDS ? 1 : kPiece];
    __shared__ int split[2];
    const int t = threadIdx.x, warp = t >> 5;
    const int rank = (int)(blockIdx.x % CLUSTER);
    const unsigned n_huge = f.plan->n_huge;
    const Less<kWords> less = {nullptr};
    for (unsigned e = blockIdx.x / CLUSTER; e < n_huge; e += gridDim.x / CLUSTER) {
        const unsigned tile = f.order[e].x;
        const uint2 rg = f.ranges[tile];
        if (!SVR_IN_BOUNDS(f.debug, kDbgRange, rg.y, f.capacity + 1)) continue;   // the whole cluster alike
        const int L = (int)(rg.y - rg.x);
        const int rounds = merge_rounds(list_chunks(L));
        for (int r = 0; r < rounds; ++r) {
            const int src = (rounds - r) & 1, dst = src ^ 1;
            const bool last = r == rounds - 1;
            const uint64_t *k0 = f.keys[src] + rg.x;
            const uint32_t *v0 = f.vals[src] + rg.x;
            const int64_t w = (int64_t)kSortCap << r;
            for (int64_t o = (int64_t)rank * kPiece; o < L; o += (int64_t)CLUSTER * kPiece) {
                const int64_t p0 = o / (2 * w) * (2 * w);
                const int64_t mid = tmin<int64_t>(L, p0 + w), end = tmin<int64_t>(L, p0 + 2 * w);
                const int na = (int)(mid - p0), nb = (int)(end - mid);
                const int d0 = (int)(o - p0), d1 = (int)(tmin<int64_t>(o + kPiece, end) - p0);
                if (warp < 2) {
                    const int c = merge_split<WORDS>(k0 + p0, v0 + p0, na, k0 + mid, v0 + mid, nb, warp ? d1 : d0);
                    if ((t & 31) == 0) split[warp] = c;
                }
                __syncthreads();
                const int a0 = split[0], a1 = split[1], b0 = d0 - a0;
                const int ca = a1 - a0, n = d1 - d0;
                for (int i = t; i < n; i += kMergeThreads) {
                    const int64_t from = i < ca ? p0 + a0 + i : mid + b0 + (i - ca);
                    sk[pad(i)] = __ldcg(k0 + from);
                    if (!WORDS) sv[i] = __ldcg(v0 + from);
                }
                __syncthreads();
                if constexpr (WORDS) {
                    uint64_t x[kMergeVT];
                    merge_out<kMergeVT>(sk, 0, ca, ca, n, min(t * kMergeVT, n), x, less);
                    __syncthreads();
#pragma unroll
                    for (int i = 0; i < kMergeVT; ++i)
                        if (t * kMergeVT + i < n) sk[pad(t * kMergeVT + i)] = x[i];
                    __syncthreads();
                    for (int i = t; i < n; i += kMergeThreads) {
                        if (last) {
                            uint64_t k;
                            uint32_t v;
                            word_pair(f, (int)tile, sk[pad(i)], k, v);
                            f.keys[dst][rg.x + o + i] = k;
                            f.vals[dst][rg.x + o + i] = v;
                        } else {
                            f.keys[dst][rg.x + o + i] = sk[pad(i)];
                        }
                    }
                } else {
                    // each pair's place: its own among its run plus the other
                    // run's pairs before it
                    for (int i = t; i < n; i += kMergeThreads) {
                        const uint64_t k = sk[pad(i)];
                        const uint32_t v = sv[i];
                        const bool in_a = i < ca;
                        int lo = in_a ? ca : 0, hi = in_a ? n : ca;
                        const int q0 = lo;
                        while (lo < hi) {
                            const int m = (lo + hi) >> 1;
                            if (pair_less(sk[pad(m)], sv[m], k, v)) lo = m + 1;
                            else hi = m;
                        }
                        const int at = (in_a ? i : i - ca) + lo - q0;
                        f.keys[dst][rg.x + o + at] = k;
                        f.vals[dst][rg.x + o + at] = v;
                    }
                }
                __syncthreads();   // shared memory is reused by the next piece
            }
            // the round's outputs are visible to the whole cluster
            asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
}

// ---------------------------------------------------------------- launchers

static unsigned sm_count() {
    static DeviceCache cache;
    return device_cached(cache, [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return (unsigned)(n > 0 ? n : 1);
    });
}

cudaError_t launch_order(const FrameDev &f, cudaStream_t s) {
    return launch(k_order, dim3((unsigned)((f.total_tiles + kOrderThreads - 1) / kOrderThreads)), kOrderThreads, 0, s, f);
}

// Clusters: one per possible long list, at most two CTAs per SM.  Few tiles
// make few and longer lists, which take eight CTAs each (a preview of 280
// tiles: 71 us, 133 with four); many tiles make many lists of two or three
// chunks, whose rounds have work for fewer (8 x 2560x1440 views: 555 us with
// eight CTAs, 292 with four, 189 with two; 16 mixed views: 113, 61 and 56).
// Between, it is the number of long lists that decides, which the host does not
// know.  svr_bin_sort with eight / two, us: 177 of them over 1,080 tiles 744 / 985, 458
// over 4,240 651 / 581, 432 over 8,030 622 / 534, 181 over 14,400 540 / 530; none over
// 8,030 106 / 122, 9,760 106 / 123, 14,400 114 / 125, one over 9,600 188 / 202.
constexpr int kFewTiles = 8192;

template <bool WORDS, int CLUSTER>
static cudaError_t merge_long(const FrameDev &f, cudaStream_t s) {
    const int64_t lists = tmin<int64_t>(f.capacity / kSortCap, f.total_tiles);
    const unsigned clusters = (unsigned)tmin<int64_t>(lists > 0 ? lists : 1, 2 * sm_count() / CLUSTER);
    return launch(k_merge_long<WORDS, CLUSTER>, dim3(clusters * CLUSTER), kMergeThreads, 0, s, f);
}

template <int MODE>
static cudaError_t sort_lists(const FrameDev &f, cudaStream_t s) {
    // at most one CTA per possible unit, at most as many as are resident at
    // once; they take units from the device-side counts
    const int64_t units = (int64_t)f.total_tiles + sort_chunk_capacity(f.capacity);
    static DeviceCache attr_set, cache;
    cudaError_t e = cudaSuccess;
    // the shared-memory opt-in is a per-device function attribute
    device_cached(attr_set, [&e] {
        e = cudaFuncSetAttribute(k_sort_lists<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortSmemBytes);
        return e == cudaSuccess ? 1u : 0u;
    });
    if (e != cudaSuccess) return e;
    const unsigned resident = device_cached(cache, [] {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sort_lists<MODE>, kSortThreads, kSortSmemBytes);
        return sm_count() * (unsigned)(per_sm > 0 ? per_sm : 1);
    });
    e = launch(k_sort_lists<MODE>, dim3((unsigned)tmin<int64_t>(units, resident)), kSortThreads, kSortSmemBytes, s, f);
    // no list can be longer than every voxel with every sign pattern
    if (e != cudaSuccess || f.capacity <= kSortCap || 8 * f.n_vox <= kSortCap) return e;
    return f.total_tiles <= kFewTiles ? merge_long<MODE == kWords, 8>(f, s) : merge_long<MODE == kWords, 2>(f, s);
}

cudaError_t launch_tile_sort(const FrameDev &f, cudaStream_t s) {
    if (f.capacity == 0) return cudaSuccess;
    return f.vid_bits > 0 ? sort_lists<kWords>(f, s) : sort_lists<kIndex>(f, s);
}

}  // namespace svr
