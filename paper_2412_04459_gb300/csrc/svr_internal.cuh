// Internal declarations of the sparse-voxel rasterizer (sm_103a).
// Shared by the kernel translation units and the C ABI; not installed.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/svr.h"

namespace svr {

template <class T>
__host__ __device__ __forceinline__ T tmin(T a, T b) {
    return a < b ? a : b;
}

constexpr int kMaxLevel = 16;
constexpr int kMaxViews = SVR_MAX_VIEWS;
constexpr float kNear = 1e-3f;             // corners at camera depth <= kNear are "behind"
constexpr uint64_t kTripleOnes = 0x249249249249ull;  // bit 0 of each of the 16 triples
constexpr int kScanTile = 256;             // entries per block of the count scan
// Tile lists longer than kSegLen entries are rendered as segments of kSegLen
// consecutive entries (the last one shorter), each by its own warps, and
// merged afterwards; kSegFields floats per pixel and segment carry the
// partial sums between the warps and on to the backward: colour (0..2),
// depth (3), transmittance after and before (4, 5; 5 holds the stopping
// index until the merge), work counts (6, 7), normal (8..10), distortion
// loss sums (11..13).
constexpr int kSegLen = 1024;
constexpr int kSegFields = 14;
// A tile's pairs are counted and emitted through sub-buckets (by voxel id), so
// that the atomics on a busy tile spread over separate cache lines; the
// sub-buckets of a tile are adjacent in its range.  Fewer tiles are busier,
// and the scan's cost grows with all of them: 32 up to 8192 tiles, 16 up to
// 131,072, else 8.  Preprocess and binning, us with 8 / 16 / 32:
//   1,080 tiles (8M voxels)   1504 / 1465 / 1401    57,600 (4 x 4M)  1836 / 1800 / 1820
//   4,240                     1344 / 1335 / 1304    115,200 (2 x 1M)  471 /  480 /  526
//   8,030                     1288 / 1284 / 1287    230,400 (4 x 1M)  800 /  828 /  914
//   14,400 (1M voxels)         241 /  239 /  246    460,800 (8 x 2M) 2413 / 2479 / 2682
// so 32 and 16 meet at the first line, and 16 and 8 between 57,600 and 115,200.
__host__ __device__ __forceinline__ int tile_sub_log2(int64_t ntiles) {
    return ntiles <= 8192 ? 5 : ntiles <= 131072 ? 4 : 3;
}

// Blocks of the scan over n sub-buckets, at most kScanBlocks: every block sums
// the sums of all, so without a bound the loads grow with the square of the
// tiles (svr_bin_sort of a few pairs over 115,200 tiles 301 us without the bound,
// 281 with it; 460,800: 906 and 841; 4.2 M: 7.7 and 3.7 ms).  Beyond 2^18
// sub-buckets a block then takes several rounds of kScanTile.
constexpr int kScanBlocks = 1024;
__host__ __device__ __forceinline__ int scan_rounds(int64_t n) {
    const int64_t most = (int64_t)kScanTile * kScanBlocks;
    return (int)((n + most - 1) / most);
}
__host__ __device__ __forceinline__ int scan_blocks(int64_t n) {
    const int64_t per = (int64_t)kScanTile * scan_rounds(n);
    return (int)((n + per - 1) / per);
}

// A tile list up to kSortCap pairs is sorted by one group of threads in shared
// memory; a longer one as chunks of at most kSortCap pairs, merged afterwards.
constexpr int kSortCap = 8192;

// Chunks a workspace holds for pair_capacity pairs: a list of L >= kSortCap
// pairs takes ceil(L / kSortCap) <= 2 L / kSortCap chunks.
__host__ __device__ __forceinline__ int64_t sort_chunk_capacity(int64_t capacity) {
    return 2 * capacity / kSortCap + 1;
}

// Words of one bit per voxel.
__host__ __device__ __forceinline__ size_t hit_words(int64_t n_vox) { return (size_t)((n_vox + 31) / 32); }

// Segment slots a workspace holds for pair_capacity pairs: a split tile of
// L > kSegLen entries takes ceil(L / kSegLen) < 2 L / kSegLen slots.
__host__ __device__ __forceinline__ int64_t seg_slot_capacity(int64_t capacity) {
    return 2 * capacity / kSegLen + 1;
}

// Camera of one view as the kernels see it: intrinsics, [R | t], the ray
// origin -R^T t (computed in double on the host) and the view's tile grid.
struct DevCam {
    float fx, fy, cx, cy;
    float R[9];
    float t[3];
    float ro[3];
    int W, H;
    int ntx, nty;
    int tile;
    int tile_base;     // first global tile id of the view
    int64_t pix_base;  // first pixel of the view in the contiguous outputs
};

// Device status block at the start of the workspace (64 bytes).
struct Status {
    unsigned flags;       // SVR_FLAG_*
    unsigned n_pairs_lo;  // total pair count (64-bit, split)
    unsigned n_pairs_hi;
    int bad_voxel;        // smallest invalid voxel id (all bits set: none)
    unsigned fwd_next;    // next work item of the forward render (the last warp of a launch resets it)
    unsigned bwd_next;    // next work item of the backward render (k_grid_bwd resets it)
    unsigned n_queue;     // (tile, segment) entries of the render work order
    unsigned slots_used;  // segment slots taken by the split tiles
    unsigned fwd_done;    // bit 0: a forward filled the segment sums of the current sort; bit 1: with
                          // the normal image; bit 2: with the distortion loss
    unsigned unused0;
    unsigned fwd_exit;    // warps of the running forward launch that ran out of work
    unsigned maxw_next;   // next work item of the maximum-weight pass over split lists (reset before it)
    unsigned unused1;
    unsigned n_listed;    // work-order entries of non-empty lists (the empty tiles' entries come last)
    unsigned pad[2];
};

// A work item of the render kernels: the 8x4 block `blk` of a tile and its
// block list, or the part of it in one segment of a split tile's list.
// k_block_lists writes those of every work-order entry e with a non-empty list
// at e B + blk, so a warp has all it needs about its work one load after it
// was given its number (the order, ranges, segments and lengths were four
// dependent loads).
struct __align__(16) RenderItem {
    uint32_t tile;     // global tile
    uint32_t blkseg;   // block | segment << 8
    uint32_t n;        // entries of the block list (in this segment)
    uint32_t beg, end; // the tile's range in the sorted pairs
    uint32_t slot;     // segment slot of a split tile, else kNoSlot
    uint32_t walked;   // entries the forward's first walk took (written by it)
    uint32_t pad;
};
constexpr uint32_t kNoSlot = 0xFFFFFFFFu;

// Groups of the render work order: floor(log2(length)) + 1 of a tile's list,
// one more for a split list, so that every split list (longer than kSegLen)
// precedes every unsplit one; a split list's first segment goes to group
// kFirstSeg + its group, ahead of all others.  Group 0: the empty lists.
constexpr int kOrderGroups = 34;
constexpr int kFirstSeg = kOrderGroups;

__device__ __forceinline__ int order_bucket(unsigned len, unsigned nseg) {
    return len ? 32 - __clz(len) + (nseg > 1 ? 1 : 0) : 0;
}

// Sort classes by list length: threads per list.  A list of 2^(c+7) to
// 2^(c+8) - 1 pairs goes to class c = 1 .. 5 (32 2^(c-1) threads of 16 pairs
// each: 2^(c+8)), a shorter one to class 0, whose lists take a warp each as
// well.  A list of exactly 1024 pairs, unsplit, goes to class 2, which it fills.
constexpr int kSortClasses = 6;

// Counters of the work order and the sort (cleared by k_scan_reduce, counted
// by k_scan_down, the rest filled by k_order).
struct SortPlan {
    unsigned cnt[2 * kOrderGroups];   // work-order entries of each group
    unsigned pos[2 * kOrderGroups];   // entries of each group already placed
    unsigned n_chunks;                // chunks of the lists of at least kSortCap pairs
    unsigned n_huge;                  // such lists: the first n_huge work-order entries
    unsigned next;                    // next unit of k_sort_lists
    unsigned first[kSortClasses];     // first work-order entry of each class's lists
    unsigned count[kSortClasses];     // and their number
};

// Index checks of the SVR_DEBUG build (compiled out otherwise).  A failed
// check counts itself in the device's DebugBlock, keeps the first failure's
// site, index and bound, and the access is skipped (a read takes index 0 or a
// neutral value); nothing traps.  svr_debug_report() reads and clears it.
struct DebugBlock {
    unsigned long long count;
    unsigned site, pad;
    long long index, bound;
};

enum DebugSite : unsigned {
    kDbgTile = 1,        // tile id >= total_tiles (emission)
    kDbgRange = 2,       // tile range end > pair capacity (sort, render)
    kDbgVoxel = 3,       // voxel id of a list entry >= n_vox (block lists, render staging)
    kDbgGradPoint = 4,   // corner index >= n_pts (render backward atomics)
    kDbgRecSlot = 5,     // gradient record slot >= kRecCap (render backward)
    kDbgSegSlot = 6,     // segment slot >= seg_slots (render)
    kDbgBlockList = 7,   // block list longer than its tile list or segment (render)
    kDbgSortList = 8,    // tile list longer than its sort class takes (sort)
};

#ifdef SVR_DEBUG
__device__ __forceinline__ bool in_bounds(DebugBlock *d, unsigned site, long long i, long long n) {
    if (i >= 0 && i < n) return true;
    if (d != nullptr && atomicAdd(&d->count, 1ull) == 0ull) {
        d->site = site;
        d->index = i;
        d->bound = n;
    }
    return false;
}
#define SVR_IN_BOUNDS(dbg, site, i, n) ::svr::in_bounds((dbg), (site), (long long)(i), (long long)(n))
#else
#define SVR_IN_BOUNDS(dbg, site, i, n) true
#endif

// Index i if SVR_IN_BOUNDS(i < n) holds, else 0 (the access reads element 0).
template <class I>
__device__ __forceinline__ I checked(DebugBlock *dbg, unsigned site, I i, long long n) {
    return SVR_IN_BOUNDS(dbg, site, i, n) ? i : I(0);
}

// The current device's DebugBlock (allocated on first use; nullptr in
// builds without SVR_DEBUG).
DebugBlock *debug_block();

// Per-voxel record of one view (64 bytes):
//   r0 = (lo - r_o).xyz, size      lo = centre - size / 2, the min corner
//   r1, r2 = the raw density as a polynomial about the voxel's centre, from
//            the 8 gathered corner densities: coefficients of 1, z, y, yz and
//            x, xz, xy, xyz (see density_coeffs)
//   r3 = colour rgb, bit c of the w word set if channel c was > 0 before the clamp
struct Record {
    float4 r0, r1, r2, r3;
};

// Asynchronous 16-byte global -> shared copy (cp.async, L2 only), its
// commit and the wait for all but the N most recent groups.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Ray direction of pixel (x, y): R^T ((x + .5 - cx) / fx, (y + .5 - cy) / fy, 1),
// written with explicit roundings so every kernel derives the same bits.
__device__ __forceinline__ float3 pixel_dir(const DevCam &c, int x, int y) {
    float dx = __fdiv_rn(__fsub_rn(__fadd_rn((float)x, 0.5f), c.cx), c.fx);
    float dy = __fdiv_rn(__fsub_rn(__fadd_rn((float)y, 0.5f), c.cy), c.fy);
    float3 d;
    d.x = __fadd_rn(__fadd_rn(__fmul_rn(c.R[0], dx), __fmul_rn(c.R[3], dy)), c.R[6]);
    d.y = __fadd_rn(__fadd_rn(__fmul_rn(c.R[1], dx), __fmul_rn(c.R[4], dy)), c.R[7]);
    d.z = __fadd_rn(__fadd_rn(__fmul_rn(c.R[2], dx), __fmul_rn(c.R[5], dy)), c.R[8]);
    return d;
}

// 4 (rd.x < 0) + 2 (rd.y < 0) + (rd.z < 0).
__device__ __forceinline__ int sign_bits(float3 d) {
    return (d.x < 0.f ? 4 : 0) | (d.y < 0.f ? 2 : 0) | (d.z < 0.f ? 1 : 0);
}

// Trilinear interpolation of Eq. interp written about the voxel's centre: with
// x, y, z in [-1/2, 1/2] the raw density is sum_m a_m x^i y^j z^k over m = 4 i
// + 2 j + k, whose coefficients follow from the corners g (corner bit order
// as m's) by taking mean and difference along each axis in turn.  Seven
// multiply-adds evaluate it, against four differences, seven multiply-adds
// and three more differences per sample from the corners.
// The linear ones, whose direction is the voxel's normal, are taken as far
// face minus near face, so that a nearly constant voxel's normal does not
// depend on the order of the axes.
__device__ __forceinline__ void density_coeffs(float g[8]) {
    const float gx = 0.25f * ((g[4] + g[5] + g[6] + g[7]) - (g[0] + g[1] + g[2] + g[3]));
    const float gy = 0.25f * ((g[2] + g[3] + g[6] + g[7]) - (g[0] + g[1] + g[4] + g[5]));
    const float gz = 0.25f * ((g[1] + g[3] + g[5] + g[7]) - (g[0] + g[2] + g[4] + g[6]));
#pragma unroll
    for (int bit = 1; bit < 8; bit *= 2)
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if (!(m & bit)) {
                const float lo = g[m], hi = g[m + bit];
                g[m] = 0.5f * (lo + hi);
                g[m + bit] = hi - lo;
            }
    g[1] = gz;
    g[2] = gy;
    g[4] = gx;
}

// 2^x, results below 2^-126 included: a raw density of -100 has a weight, an
// optical depth of 95 a transmittance.  That takes three instructions more than
// the form that flushes them (3 % of the 1M-voxel step; flushing first and taking
// the samples again where it could show cost as much).
__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
constexpr float kLog2e = 1.44269504f, kLn2 = 0.693147181f;

// 1 / x to 1 ulp, the hardware instruction on its own.
__device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// explin (Eq. explin): x above 1.1, else exp(x / 1.1 - 1 + ln 1.1).  log2(e) is
// a factor of its own: folded into the two constants, whose roundings no longer
// offset that of ex2, alpha was 0.6 to 1 % further from 64 bits.
__device__ __forceinline__ float explin(float x) {
    return x > 1.1f ? x : ex2(fmaf(x, 0.909090909f, -0.904689820f) * kLog2e);
}

// Real SH basis, degree 0..3, index l*l + l + m, no Condon-Shortley phase,
// as polynomials of the unit direction (x, y, z).  Constants are
// sqrt((2l+1)/(4 pi) (l-|m|)!/(l+|m|)!) times the factors of the
// corresponding Legendre / trigonometric polynomial.
__device__ __forceinline__ void sh_basis(float x, float y, float z, float Y[16]) {
    const float xx = x * x, yy = y * y, zz = z * z;
    Y[0] = 0.28209479177387814f;
    Y[1] = 0.4886025119029199f * y;
    Y[2] = 0.4886025119029199f * z;
    Y[3] = 0.4886025119029199f * x;
    Y[4] = 1.0925484305920792f * x * y;
    Y[5] = 1.0925484305920792f * y * z;
    Y[6] = 0.31539156525252005f * (3.f * zz - 1.f);
    Y[7] = 1.0925484305920792f * x * z;
    Y[8] = 0.5462742152960396f * (xx - yy);
    Y[9] = 0.5900435899266435f * y * (3.f * xx - yy);
    Y[10] = 2.890611442640554f * x * y * z;
    Y[11] = 0.4570457994644658f * y * (5.f * zz - 1.f);
    Y[12] = 0.3731763325901154f * z * (5.f * zz - 3.f);
    Y[13] = 0.4570457994644658f * x * (5.f * zz - 1.f);
    Y[14] = 1.445305721320277f * z * (xx - yy);
    Y[15] = 0.5900435899266435f * x * (xx - 3.f * yy);
}

// Everything the kernels need about a frame: the view table, the scene
// arrays and the workspace buffers.  Passed by value as a kernel parameter,
// so launches need no host-to-device copies (CUDA-graph capturable).
// Per-(view, voxel) arrays are indexed view * n_vox + voxel.
struct FrameDev {
    DevCam views[kMaxViews];
    int n_views;
    int total_tiles;         // sum of the views' tile counts
    int sub_log2;            // log2 of a tile's sub-buckets
    int key_shift;           // Morton bits kept in the key; the tile id sits above them
    Status *status;
    uint8_t *tile_mask;      // [total_tiles]
    uint8_t *block_sign;     // [total_tiles][B]: sign-bit mask of each 8x4 block's in-image pixels
    uint64_t *octpath;       // [N]
    short4 *rect;            // [V * N] tile rectangle tx0, tx1, ty0, ty1
    uint32_t *count;         // [V * N] pairs of each (view, voxel)
    uint32_t *tile_cnt;      // [2^sub_log2][total_tiles] pairs of each tile's sub-buckets (k_preprocess)
    uint32_t *cursor;        // [2^sub_log2][total_tiles] next free slot of each sub-bucket
    Record *rec;             // [V * N]
    ushort4 *box;            // [V * N] inclusive pixel range x0, x1, y0, y1 a hit can fall in
    uint32_t *may_hit;       // single view: [hit_words(N)] bit v mod 32 of word v / 32: voxel v has a pair and
                             // a box that is not empty
    unsigned long long *scan_blocks;   // [scan_blocks(2^sub_log2 total_tiles)] their sums
    uint64_t *keys[2];
    uint32_t *vals[2];
    SortPlan *plan;
    uint2 *chunks;           // [sort_chunk_capacity] (tile, chunk) of the long lists
    int sort_bits;           // Morton bits that can differ between two pairs of a tile
    int vid_bits;            // > 0: a pair is emitted and sorted as one 64-bit word (see pair_word),
                             // with this many low bits for the voxel id; 0: as its key and value
    uint2 *ranges;           // [total_tiles]
    uint2 *order;            // [total_tiles + seg slots] (tile, segment), longest segments first
    uint2 *tile_seg;         // [total_tiles] segments of the tile's list, first segment slot
    uint32_t *merge_cnt;     // [total_tiles * B] segments of a (tile, block) finished by the forward
    uint32_t *seg_len;       // [slots * B] block-list entries of each (segment, block)
    float *seg_part;         // [slots * B][kSegFields][32] per-pixel segment sums
    int64_t seg_slots;       // slots the workspace holds
    uint2 *blist;            // per (tile, 8x4 block) lists of (value, sorted index): block b of a tile
                             // whose list is [beg, end) owns [B beg + b (end - beg), ...)
    RenderItem *items;       // [(total_tiles + seg slots) * B]
    uint32_t *hmask;         // the forward's hit masks: block b of tile g (list [beg, end)) owns the
                             // words from B beg + b (end - beg) + 32 (g B + b); word p of it is, for
                             // p in batch [32 k, 32 k + 32) of the block's walk, the mask of the
                             // batch's entries (bit i: position 32 k + i) that pixel p mod 32 hit
    int blocks_per_tile;     // B = tile * tile / 32
    float4 *dcol;            // [V * N] colour gradient and priority accumulators
    float4 *dgrid;           // [N][2] corner-density gradient accumulators (after dcol)
    int64_t n_vox;
    int64_t n_pts;
    int64_t capacity;
    float world_size;
    float world_min[3];      // w_c - w_s / 2
    int max_level;
    int K;
    float t_stop;
    float bg[3];
    const float *centre;
    const uint8_t *level;
    const int32_t *corner_idx;
    const float *grid;
    const float *sh;
    DebugBlock *debug;       // index-check report of the SVR_DEBUG build (else nullptr)
};

// The word of a pair where its parts fit 64 bits: the Morton bits that can
// differ, then (max level 16 only) the sign pattern, then the voxel id.
// Words of one tile order like its (key, value) pairs: below max level 16 the
// lowest Morton triple is the sign pattern itself (a padded triple).
__host__ __device__ __forceinline__ int word_sign_bits(int max_level) { return max_level >= kMaxLevel ? 3 : 0; }

__device__ __forceinline__ uint64_t pair_word(const FrameDev &f, uint64_t code, unsigned s, uint32_t vid) {
    const uint64_t m = (code ^ ((uint64_t)s * kTripleOnes)) >> (48 - f.sort_bits);
    const uint64_t hi = f.max_level >= kMaxLevel ? (m << 3) | s : m;
    return (hi << f.vid_bits) | vid;
}

// Key and value of tile g's pair from its Morton bits, sign pattern and voxel id.
__device__ __forceinline__ uint64_t pair_key(const FrameDev &f, int g, uint64_t morton, unsigned s) {
    const int lo = f.key_shift - f.sort_bits;   // low bits of the order: padded triples, all s
    return ((uint64_t)g << f.key_shift) | (morton << lo) | (((uint64_t)s * kTripleOnes) & ((1ull << lo) - 1ull));
}

__device__ __forceinline__ void word_pair(const FrameDev &f, int g, uint64_t word, uint64_t &key, uint32_t &val) {
    const uint32_t vid = (uint32_t)(word & ((1ull << f.vid_bits) - 1ull));
    const uint64_t hi = word >> f.vid_bits;
    const unsigned s = (unsigned)hi & 7u;
    key = pair_key(f, g, f.max_level >= kMaxLevel ? hi >> 3 : hi, s);
    val = (s << 29) | vid;
}

// View that owns global tile g.
__device__ __forceinline__ int view_of_tile(const FrameDev &f, int g) {
    int v = 0;
#pragma unroll
    for (int step = kMaxViews / 2; step > 0; step /= 2)
        if (v + step < f.n_views && g >= f.views[v + step].tile_base) v += step;
    return v;
}

// A launch constant (a persistent grid size, an SM count) kept per device,
// so that a process driving several GPUs in turn launches each with its
// own; 0 means not computed yet.  Concurrent first calls may both compute
// it and store the same value.
constexpr int kMaxDevices = 64;
struct DeviceCache {
    std::atomic<unsigned> v[kMaxDevices];
};

template <class F>
unsigned device_cached(DeviceCache &c, F compute) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return compute();
    unsigned x = c.v[dev].load(std::memory_order_relaxed);
    if (x == 0) {
        x = compute();
        c.v[dev].store(x, std::memory_order_relaxed);
    }
    return x;
}

// Programmatic dependent launch: a kernel launched with launch() may start
// while the stream's kernel before it still runs; it first lets the next one
// do the same and then waits for all of the kernel before (and so, that one
// having waited too, for everything before it), before it reads or writes
// memory.  So the ten kernels from the tile masks to the forward do not wait
// for one another's launch: 742 -> 718 us for the 1M-voxel step, 183 -> 174 us
// for the smallest view.  The backward's kernels are launched plainly: with
// them the step took 773 us.  Large frames do not gain.  Preprocess to forward,
// us without and with: 1M voxels over 8,030 tiles 417 and 396, 14,400 562 and 553,
// 16,060 (two views) 696 and 683, 16,960 (four) 985 and 986, 28,800 (8M voxels, two)
// 3147 and 3176; 8M voxels over 1,080 to 16,000 tiles lose up to 1 %.
// Such a kernel is resident while the ones before it still write, so what it
// reads is not constant for its lifetime: it loads with ordinary or L2 loads
// only, which the wait orders, never through __ldg or const __restrict__
// pointers (ld.global.nc).
constexpr int kOverlapTiles = 16384;

__device__ __forceinline__ void begin_kernel() {
    asm volatile("griddepcontrol.launch_dependents;\ngriddepcontrol.wait;" ::: "memory");
}

template <class... Params, class... Args>
cudaError_t launch(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                   const FrameDev &f, Args... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = f.total_tiles <= kOverlapTiles ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, f, args...);
}

// Records a printf-style message for svr_last_error() and returns code.
int set_error(int code, const char *fmt, ...);

// svr_preprocess for a frame that no backward will follow: its workspace holds
// neither gradient accumulators nor hit masks.
int preprocess_forward_only(svr_frame *frame, const svr_scene *scene, const svr_camera *cam,
                            const svr_params *params, void *ws, size_t ws_bytes, int64_t pair_capacity,
                            void *stream);

cudaError_t launch_tile_mask(const FrameDev &f, cudaStream_t s);
cudaError_t launch_preprocess(const FrameDev &f, cudaStream_t s);
cudaError_t launch_scan(const FrameDev &f, cudaStream_t s);
cudaError_t launch_order(const FrameDev &f, cudaStream_t s);
cudaError_t launch_emit(const FrameDev &f, cudaStream_t s);
cudaError_t launch_tile_sort(const FrameDev &f, cudaStream_t s);
cudaError_t launch_block_lists(const FrameDev &f, int sorted_alt, cudaStream_t s);
cudaError_t launch_render_fwd(const FrameDev &f, float *rgb, float *depth,
                              float *alpha, float *T_final, int32_t *last, int2 *stats, float *normal,
                              float *max_weight, float *dist, cudaStream_t s);
cudaError_t launch_render_bwd(const FrameDev &f, const float *d_rgb,
                              const float *d_depth, const float *d_alpha, const float *T_final,
                              const int32_t *last, float *d_grid, float *d_sh, const float *d_normal,
                              float *priority, const float *d_dist, const float *dist, float *max_weight,
                              cudaStream_t s);

}  // namespace svr
