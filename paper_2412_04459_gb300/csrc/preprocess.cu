// Per-view preprocessing, count scan and pair emission (sm_103a).
//
//   k_tile_mask   per 8x4 pixel block and per tile: OR of 1 << signbits(r_d)
//                 over the in-image pixels
//                 (ray sign bits of Sec. B.2; duplication per sign pattern,
//                 Sec. B.1)
//   k_preprocess  per (view, voxel): lattice index, Morton code (Sec. A.1),
//                 tile rectangle of the projected corners (Sec. 3.1.2), pair
//                 count, conservative pixel box, view-dependent colour
//                 (Eq. vox_color), gathered densities
//                 and, per tile, the pairs it will hold (atomics);
//                 k_preprocess_views does the same for a batch of views with
//                 one thread per voxel, reading its densities and SH once
//   k_scan_*      exclusive scan of the tiles' pair counts (block sums, then
//                 each block scans its part after summing the earlier blocks;
//                 the sub-buckets of a tile are adjacent): each sub-bucket's
//                 start, each tile's range and segments, the work order's
//                 group counts, the total, the capacity check
//   k_emit        writes each (voxel, tile, sign pattern s) pair into its
//                 tile's range (an atomic cursor per sub-bucket; the order
//                 within a tile is left to the per-tile sort):
//                 key = tile << S | top S bits of (octpath ^ s replicated),
//                 value = s << 29 | voxel id, written as one word that the
//                 sort turns into them where it fits 64 bits (pair_word; one
//                 8-byte store instead of 12 bytes in two) (Sec. B.1; the per-triple
//                 permutation of Sec. B.2 is b ^ s, applied to all 16
//                 triples at once).  S = 48 for one view (the paper's layout:
//                 16-bit tile id over the 48-bit order); a batch of views uses
//                 the global tile id over the 3 (max_level + 1) Morton bits
//                 that can differ, so more than 2^16 tiles fit in 64 bits.
#include <climits>

#include "svr_internal.cuh"

namespace svr {

// --------------------------------------------------------------- tile masks

// A ray component is a rounded affine function of the pixel, monotonic along
// each image axis, so where the four corner pixels of a tile agree in its sign
// every pixel between does, and the tile and its blocks hold that one pattern.
// Four lanes take a tile's corners.  The few tiles whose corners differ (or
// whose rays overflow) are walked by the whole warp, 8x4 pixel block by block
// (the render's warp blocks, tile / 8 per block row): each block's sign-bit
// mask goes to block_sign, their OR to tile_mask.  A warp takes up to eight
// tiles at a time, which lie far apart, so that a row of tiles along an axis of
// the image is walked by many warps.
// Every tile walked, at two divisions per pixel, was 100 us of the 8 x
// 2560x1440 batch; a warp's tiles side by side, 74 us.
constexpr int kMaskThreads = 128;
constexpr int kMaskWarps = 4096;

__global__ void __launch_bounds__(kMaskThreads) k_tile_mask(FrameDev f) {
    begin_kernel();
    // also starts the frame: status cleared (no smallest invalid voxel yet)
    // and the tiles' pair counters zeroed, before k_preprocess counts
    if (blockIdx.x == 0 && threadIdx.x < sizeof(Status) / 4)
        reinterpret_cast<unsigned *>(f.status)[threadIdx.x] =
            threadIdx.x == offsetof(Status, bad_voxel) / 4 ? 0xFFFFFFFFu : 0u;
    const int lane = threadIdx.x & 31;
    const int n_threads = gridDim.x * kMaskThreads, n_warps = n_threads / 32;
    const int warp = blockIdx.x * (kMaskThreads / 32) + (threadIdx.x >> 5);
    for (int64_t i = blockIdx.x * kMaskThreads + threadIdx.x; i < ((int64_t)f.total_tiles << f.sub_log2); i += n_threads)
        f.tile_cnt[i] = 0u;
    const int B = f.blocks_per_tile;
    for (int base = 0; base + warp < f.total_tiles; base += 8 * n_warps) {
        const int g = base + (lane >> 2) * n_warps + warp, c = lane & 3;
        const bool valid = g < f.total_tiles;
        const DevCam &cam = f.views[view_of_tile(f, valid ? g : base + warp)];
        const int T = cam.tile, bpr = T >> 3, tile = (valid ? g : base + warp) - cam.tile_base;
        const int x0 = (tile % cam.ntx) * T, y0 = (tile / cam.ntx) * T;
        const int x1 = min(x0 + T, cam.W) - 1, y1 = min(y0 + T, cam.H) - 1;
        const float3 d = pixel_dir(cam, (c & 1) ? x1 : x0, (c & 2) ? y1 : y0);
        const int s = isfinite(d.x) && isfinite(d.y) && isfinite(d.z) ? sign_bits(d) : 8;
        const int s0 = __shfl_sync(0xffffffffu, s, lane & ~3);
        const unsigned differ = __ballot_sync(0xffffffffu, s != s0 || s == 8);
        const bool walk = valid && ((differ >> (lane & ~3)) & 0xFu) != 0u;
        if (valid && !walk) {
            for (int b = c; b < B; b += 4)
                f.block_sign[(size_t)g * B + b] =
                    x0 + (b % bpr) * 8 <= x1 && y0 + (b / bpr) * 4 <= y1 ? (uint8_t)(1u << s) : (uint8_t)0;
            if (c == 0) f.tile_mask[g] = (uint8_t)(1u << s);
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, walk && c == 0); todo; todo &= todo - 1u) {
            const int h = __shfl_sync(0xffffffffu, g, __ffs(todo) - 1);
            const DevCam &hc = f.views[view_of_tile(f, h)];
            const int ht = h - hc.tile_base;
            const int hx = (ht % hc.ntx) * T, hy = (ht / hc.ntx) * T;
            unsigned m = 0;
            for (int b = 0; b < B; ++b) {
                const int x = hx + (b % bpr) * 8 + (lane & 7), y = hy + (b / bpr) * 4 + (lane >> 3);
                const unsigned bit = (x < hc.W && y < hc.H) ? 1u << sign_bits(pixel_dir(hc, x, y)) : 0u;
                const unsigned bm = __reduce_or_sync(0xffffffffu, bit);
                if (lane == b) f.block_sign[(size_t)h * B + b] = (uint8_t)bm;
                m |= bm;
            }
            if (lane == 0) f.tile_mask[h] = (uint8_t)m;
        }
    }
}

// --------------------------------------------------------------- preprocess

// Spread the low 16 bits of x to bit positions 0, 3, 6, ..., 45.
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0xFFFFu;
    x = (x | (x << 16)) & 0x0000FF0000FFull;
    x = (x | (x << 8)) & 0x00F00F00F00Full;
    x = (x | (x << 4)) & 0x0C30C30C30C3ull;
    x = (x | (x << 2)) & 0x249249249249ull;
    return x;
}

__device__ __forceinline__ void mark_invalid(Status *st, int64_t v) {
    atomicOr(&st->flags, SVR_FLAG_INVALID_VOXEL);
    atomicMin(reinterpret_cast<unsigned *>(&st->bad_voxel), (unsigned)v);
}

// Lattice index of voxel v (centre = w_min + v_s (ijk + 1/2)) and the
// validity of its level, centre and corner indices.
__device__ __forceinline__ bool voxel_valid(const FrameDev &f, int64_t v, float c0, float c1, float c2, int l,
                                            float &vs, int ijk[3], int4 &i0, int4 &i1) {
    bool ok = l >= 1 && l <= f.max_level;
    vs = ldexpf(f.world_size, -l);
    ijk[0] = ijk[1] = ijk[2] = 0;
    if (ok) {
        const float cc[3] = {c0, c1, c2};
        const int n = 1 << l;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float fi = (cc[a] - f.world_min[a]) / vs - 0.5f;
            float r = rintf(fi);
            ok = ok && fabsf(fi - r) <= 0.25f && r >= 0.f && r < (float)n;
            ijk[a] = (int)r;
        }
    }
    // corner indices must name grid points
    const int4 *ci = reinterpret_cast<const int4 *>(f.corner_idx + 8 * v);
    i0 = ci[0];
    i1 = ci[1];
    const int64_t np = f.n_pts;
    const int lo = min(min(min(i0.x, i0.y), min(i0.z, i0.w)), min(min(i1.x, i1.y), min(i1.z, i1.w)));
    const int hi = max(max(max(i0.x, i0.y), max(i0.z, i0.w)), max(max(i1.x, i1.y), max(i1.z, i1.w)));
    return ok && lo >= 0 && (int64_t)hi < np;
}

// Pixel box of a voxel across the camera plane (some corners at depth <=
// kNear): its rectangle is the whole image, but a ray meets only the part in
// front, whose points have X / Z beyond the nearest X over the largest Z where
// the voxel lies to one side of the axis (the same for Y).  Widened by a margin
// far above the rounding of the projection and of the ray test; empty
// (x0 > x1) where no pixel is left, which is usual: most such voxels lie far
// to the side.
__device__ __noinline__ ushort4 straddle_box(const DevCam &cam, float c0, float c1, float c2, float h) {
    float X0 = INFINITY, X1 = -INFINITY, Y0 = INFINITY, Y1 = -INFINITY, Z1 = -INFINITY;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float px = (c & 4) ? c0 + h : c0 - h;
        const float py = (c & 2) ? c1 + h : c1 - h;
        const float pz = (c & 1) ? c2 + h : c2 - h;
        const float X = fmaf(cam.R[0], px, fmaf(cam.R[1], py, fmaf(cam.R[2], pz, cam.t[0])));
        const float Y = fmaf(cam.R[3], px, fmaf(cam.R[4], py, fmaf(cam.R[5], pz, cam.t[1])));
        const float Z = fmaf(cam.R[6], px, fmaf(cam.R[7], py, fmaf(cam.R[8], pz, cam.t[2])));
        X0 = fminf(X0, X);
        X1 = fmaxf(X1, X);
        Y0 = fminf(Y0, Y);
        Y1 = fmaxf(Y1, Y);
        Z1 = fmaxf(Z1, Z);
    }
    const float m = 2e-5f * (fmaxf(fabsf(X0), fabsf(X1)) + fmaxf(fabsf(Y0), fabsf(Y1)) + Z1 + h) +
                    4e-6f * (fabsf(cam.t[0]) + fabsf(cam.t[1]) + fabsf(cam.t[2]) + fabsf(c0) + fabsf(c1) + fabsf(c2));
    const float iz = 1.0f / (Z1 + m);
    const float u0 = X0 - m > 0.f ? fmaf(cam.fx, (X0 - m) * iz, cam.cx) : -INFINITY;
    const float u1 = X1 + m < 0.f ? fmaf(cam.fx, (X1 + m) * iz, cam.cx) : INFINITY;
    const float v0 = Y0 - m > 0.f ? fmaf(cam.fy, (Y0 - m) * iz, cam.cy) : -INFINITY;
    const float v1 = Y1 + m < 0.f ? fmaf(cam.fy, (Y1 + m) * iz, cam.cy) : INFINITY;
    const float fx0 = fmaxf(floorf(u0 - 1.f - 1e-4f * fabsf(u0)), 0.f);
    const float fx1 = fminf(floorf(u1 + 1.f + 1e-4f * fabsf(u1)), (float)(cam.W - 1));
    const float fy0 = fmaxf(floorf(v0 - 1.f - 1e-4f * fabsf(v0)), 0.f);
    const float fy1 = fminf(floorf(v1 + 1.f + 1e-4f * fabsf(v1)), (float)(cam.H - 1));
    if (!(fx0 <= fx1 && fy0 <= fy1)) return make_ushort4(1, 0, 1, 0);
    return make_ushort4((unsigned short)fx0, (unsigned short)fx1, (unsigned short)fy0, (unsigned short)fy1);
}

// Projection of a voxel in one view: tile rectangle and conservative pixel box.
__device__ __forceinline__ short4 project_voxel(const DevCam &cam, float c0, float c1, float c2, float h,
                                                ushort4 &box) {
    float umin = INFINITY, umax = -INFINITY, vmin = INFINITY, vmax = -INFINITY, zmin = INFINITY;
    int behind = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float px = (c & 4) ? c0 + h : c0 - h;
        const float py = (c & 2) ? c1 + h : c1 - h;
        const float pz = (c & 1) ? c2 + h : c2 - h;
        const float X = fmaf(cam.R[0], px, fmaf(cam.R[1], py, fmaf(cam.R[2], pz, cam.t[0])));
        const float Y = fmaf(cam.R[3], px, fmaf(cam.R[4], py, fmaf(cam.R[5], pz, cam.t[1])));
        const float Z = fmaf(cam.R[6], px, fmaf(cam.R[7], py, fmaf(cam.R[8], pz, cam.t[2])));
        if (Z <= kNear) {
            ++behind;
        } else {
            const float u = fmaf(cam.fx, X / Z, cam.cx);
            const float w = fmaf(cam.fy, Y / Z, cam.cy);
            zmin = fminf(zmin, Z);
            umin = fminf(umin, u);
            umax = fmaxf(umax, u);
            vmin = fminf(vmin, w);
            vmax = fmaxf(vmax, w);
        }
    }
    short4 rc = make_short4(0, -1, 0, -1);
    box = make_ushort4(0, (unsigned short)(cam.W - 1), 0, (unsigned short)(cam.H - 1));
    if (behind == 8) {
        // culled
    } else if (behind > 0) {
        rc = make_short4(0, (short)(cam.ntx - 1), 0, (short)(cam.nty - 1));
        box = straddle_box(cam, c0, c1, c2, h);
    } else if (!(umax < 0.f || umin >= (float)cam.W || vmax < 0.f || vmin >= (float)cam.H)) {
        // pixels whose centre (x + 1/2, y + 1/2) can lie in the projected box,
        // widened by a rounding margin: a conservative filter for the render.
        // Empty (x0 > x1) for a voxel that falls between the pixel centres, as
        // most of the finest ones do.
        // The margin's last term is the rounding of coordinates far from the
        // world's origin, in pixels.
        const float e = 5e-7f / zmin *
                        (fabsf(cam.t[0]) + fabsf(cam.t[1]) + fabsf(cam.t[2]) + fabsf(c0) + fabsf(c1) + fabsf(c2));
        const float mu = 0.01f + 1e-5f * fmaxf(fabsf(umin), fabsf(umax)) + cam.fx * e;
        const float mv = 0.01f + 1e-5f * fmaxf(fabsf(vmin), fabsf(vmax)) + cam.fy * e;
        const float fx0 = fmaxf(ceilf(umin - 0.5f - mu), 0.f), fx1 = fminf(floorf(umax - 0.5f + mu), (float)(cam.W - 1));
        const float fy0 = fmaxf(ceilf(vmin - 0.5f - mv), 0.f), fy1 = fminf(floorf(vmax - 0.5f + mv), (float)(cam.H - 1));
        box = fx0 <= fx1 && fy0 <= fy1 ? make_ushort4((unsigned short)fx0, (unsigned short)fx1, (unsigned short)fy0,
                                                      (unsigned short)fy1)
                                       : make_ushort4(1, 0, 1, 0);
        // a power of two, so its inverse is exact (four divisions were 2 % of
        // the kernel: 8 views of 8M voxels 2671 -> 2618 us)
        const float inv_T = 1.0f / (float)cam.tile;
        const int tx0 = umin < 0.f ? 0 : min(cam.ntx - 1, (int)floorf(umin * inv_T));
        const int tx1 = umax >= (float)cam.W ? cam.ntx - 1 : min(cam.ntx - 1, (int)floorf(umax * inv_T));
        const int ty0 = vmin < 0.f ? 0 : min(cam.nty - 1, (int)floorf(vmin * inv_T));
        const int ty1 = vmax >= (float)cam.H ? cam.nty - 1 : min(cam.nty - 1, (int)floorf(vmax * inv_T));
        rc = make_short4((short)tx0, (short)tx1, (short)ty0, (short)ty1);
    }
    return rc;
}

// Voxels over more tiles than this are counted and emitted by their whole
// warp: those near the camera or across its plane cover up to every tile of
// the image, and one thread at a time over them was 142 + 334 us of a 1.3 ms
// view from inside a scene (1,200 tiles, 2,400 such voxels).
constexpr int kCoopTiles = 16;

__device__ __forceinline__ int rect_tiles(const short4 &rc) {
    return max((int)rc.y - rc.x + 1, 0) * max((int)rc.w - rc.z + 1, 0);
}

__device__ __forceinline__ short4 shfl_rect(const short4 &rc, int src) {
    const int lo = __shfl_sync(0xffffffffu, ((int)(unsigned short)rc.x) | ((int)rc.y << 16), src);
    const int hi = __shfl_sync(0xffffffffu, ((int)(unsigned short)rc.z) | ((int)rc.w << 16), src);
    return make_short4((short)(lo & 0xFFFF), (short)(lo >> 16), (short)(hi & 0xFFFF), (short)(hi >> 16));
}

// Pair count of voxel v with tile rectangle rc (the tiles' counts raised by
// atomics).  Called by all lanes of the warp; an empty rc counts nothing.
__device__ __forceinline__ uint32_t count_pairs(const FrameDev &f, const DevCam &cam, int64_t v, const short4 &rc) {
    const int lane = threadIdx.x & 31;
    const uint8_t *mask = f.tile_mask + cam.tile_base;
    uint32_t *cnt = f.tile_cnt + cam.tile_base;
    const int sub = (int)(v & ((1 << f.sub_log2) - 1));
    const bool coop = rect_tiles(rc) > kCoopTiles;
    uint32_t n = 0;
    if (!coop) {
        for (int ty = rc.z; ty <= rc.w; ++ty) {
            for (int tx = rc.x; tx <= rc.y; ++tx) {
                const int tile = ty * cam.ntx + tx;
                const uint32_t c = __popc(mask[tile]);
                if (c) atomicAdd(cnt + (size_t)sub * f.total_tiles + tile, c);
                n += c;
            }
        }
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, coop); todo; todo &= todo - 1u) {
        const int src = __ffs(todo) - 1;
        const short4 q = shfl_rect(rc, src);
        const int w = q.y - q.x + 1, area = rect_tiles(q);
        uint32_t *to = cnt + (size_t)__shfl_sync(0xffffffffu, sub, src) * f.total_tiles;
        uint32_t all = 0;
        for (int i = lane; i < area; i += 32) {
            const int tile = (q.z + i / w) * cam.ntx + q.x + i % w;
            const uint32_t c = __popc(mask[tile]);
            if (c) atomicAdd(to + tile, c);
            all += c;
        }
        all = __reduce_add_sync(0xffffffffu, all);
        if (lane == src) n = all;
    }
    return n;
}

// Colour of the voxel in one view (Eq. vox_color): degree-3 SH at the
// direction from the view's ray origin to the centre, clamped at 0; bit c of
// the w word set if channel c was > 0 before the clamp.
__device__ __forceinline__ void view_basis(const DevCam &cam, float c0, float c1, float c2, float Y[16]) {
    float dx = c0 - cam.ro[0], dy = c1 - cam.ro[1], dz = c2 - cam.ro[2];
    const float inv = 1.0f / sqrtf(dx * dx + dy * dy + dz * dz);
    dx *= inv;
    dy *= inv;
    dz *= inv;
    sh_basis(dx, dy, dz, Y);
}

__device__ __forceinline__ float4 voxel_colour(const float Y[16], const float sh[48]) {
    float col[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        float acc = 0.f;
#pragma unroll
        for (int n = 0; n < 16; ++n) acc = fmaf(Y[n], sh[3 * n + ch], acc);
        col[ch] = acc;
    }
    const unsigned bits = (col[0] > 0.f ? 1u : 0u) | (col[1] > 0.f ? 2u : 0u) | (col[2] > 0.f ? 4u : 0u);
    return make_float4(fmaxf(col[0], 0.f), fmaxf(col[1], 0.f), fmaxf(col[2], 0.f), __uint_as_float(bits));
}

__device__ __forceinline__ void load_sh(const FrameDev &f, int64_t v, float sh[48]) {
    const float4 *shv = reinterpret_cast<const float4 *>(f.sh + 48 * v);
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        const float4 s4 = shv[q];
        sh[4 * q + 0] = s4.x;
        sh[4 * q + 1] = s4.y;
        sh[4 * q + 2] = s4.z;
        sh[4 * q + 3] = s4.w;
    }
}

// Corner densities beyond this are taken as it: their voxels are as empty or as
// opaque, and the differences of the polynomial stay finite.  (The lowest float,
// or minus infinity, as the density of points that are to hold nothing gave
// infinite differences of both signs, and NaN images.)  NaN stays NaN.
constexpr float kDensityMost = 1e36f;

// A voxel's density polynomial from its gathered corner densities.
__device__ __forceinline__ void gather_density(const FrameDev &f, const int4 &i0, const int4 &i1, float4 &r1,
                                               float4 &r2) {
    float g[8] = {f.grid[i0.x], f.grid[i0.y], f.grid[i0.z], f.grid[i0.w],
                  f.grid[i1.x], f.grid[i1.y], f.grid[i1.z], f.grid[i1.w]};
    float most = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) most = fmaxf(most, fabsf(g[c]));
    if (most > kDensityMost) {
#pragma unroll
        for (int c = 0; c < 8; ++c) g[c] = g[c] > kDensityMost ? kDensityMost : g[c] < -kDensityMost ? -kDensityMost : g[c];
    }
    density_coeffs(g);
    r1 = make_float4(g[0], g[1], g[2], g[3]);
    r2 = make_float4(g[4], g[5], g[6], g[7]);
}

__device__ __forceinline__ void write_octpath(const FrameDev &f, int64_t v, int l, const int ijk[3]) {
    f.octpath[v] = ((spread3(ijk[0]) << 2) | (spread3(ijk[1]) << 1) | spread3(ijk[2])) << (3 * (kMaxLevel - l));
}

// One view (grid.y = view): one thread per (view, voxel).  No thread leaves
// before the pair count, which the warp takes together.
__global__ void __launch_bounds__(128, 8) k_preprocess(FrameDev f) {
    begin_kernel();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = v < f.n_vox;
    const int view = blockIdx.y;
    const DevCam &cam = f.views[view];
    const int64_t iv = (int64_t)view * f.n_vox + v;
    const short4 none = make_short4(0, -1, 0, -1);
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, vs = 0.f;
    int4 i0 = make_int4(0, 0, 0, 0), i1 = i0;
    short4 rc = none;
    ushort4 box = make_ushort4(0, 0, 0, 0);
    if (in) {
        c0 = f.centre[3 * v + 0];
        c1 = f.centre[3 * v + 1];
        c2 = f.centre[3 * v + 2];
        const int l = f.level[v];
        int ijk[3];
        if (voxel_valid(f, v, c0, c1, c2, l, vs, ijk, i0, i1)) {
            if (view == 0) write_octpath(f, v, l, ijk);
            rc = project_voxel(cam, c0, c1, c2, 0.5f * vs, box);
        } else if (view == 0) {
            mark_invalid(f.status, v);
        }
    }
    // which of the warp's voxels a pixel can hit: those with a tile rectangle
    // (and so with pairs) and a box that is not empty
    const unsigned hit = __ballot_sync(0xffffffffu, rc.x <= rc.y && box.x <= box.y);
    if (in && (threadIdx.x & 31) == 0) f.may_hit[v >> 5] = hit;
    const uint32_t cnt = count_pairs(f, cam, v, rc);
    if (!in) return;
    f.rect[iv] = rc;
    f.count[iv] = cnt;
    if (cnt == 0) return;
    f.box[iv] = box;
    const float h = 0.5f * vs;
    // record of this view: min corner relative to the ray origin, size,
    // density polynomial, colour
    Record r;
    r.r0 = make_float4((c0 - h) - cam.ro[0], (c1 - h) - cam.ro[1], (c2 - h) - cam.ro[2], vs);
    gather_density(f, i0, i1, r.r1, r.r2);
    float Y[16], sh[48];
    view_basis(cam, c0, c1, c2, Y);
    load_sh(f, v, sh);
    r.r3 = voxel_colour(Y, sh);
    f.rec[iv] = r;
}

// Several views: one thread per voxel.  The voxel's validity, Morton code,
// densities and SH coefficients are read once for all views (the SH only
// while the views' colours are evaluated, which are written first, into the
// records' colour words); then each view's projection, tile counts and the
// rest of its record.
__global__ void __launch_bounds__(128) k_preprocess_views(FrameDev f) {
    begin_kernel();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = v < f.n_vox;
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, vs = 0.f;
    int4 i0 = make_int4(0, 0, 0, 0), i1 = i0;
    bool ok = false;
    float4 g0, g1;
    if (in) {
        c0 = f.centre[3 * v + 0];
        c1 = f.centre[3 * v + 1];
        c2 = f.centre[3 * v + 2];
        const int l = f.level[v];
        int ijk[3];
        ok = voxel_valid(f, v, c0, c1, c2, l, vs, ijk, i0, i1);
        if (!ok) {
            mark_invalid(f.status, v);
        } else {
            write_octpath(f, v, l, ijk);
            float sh[48];
            load_sh(f, v, sh);
            for (int view = 0; view < f.n_views; ++view) {
                float Y[16];
                view_basis(f.views[view], c0, c1, c2, Y);
                f.rec[(int64_t)view * f.n_vox + v].r3 = voxel_colour(Y, sh);
            }
            gather_density(f, i0, i1, g0, g1);
        }
    }
    const float h = 0.5f * vs;
    for (int view = 0; view < f.n_views; ++view) {
        const DevCam &cam = f.views[view];
        const int64_t iv = (int64_t)view * f.n_vox + v;
        ushort4 box = make_ushort4(0, 0, 0, 0);
        const short4 rc = ok ? project_voxel(cam, c0, c1, c2, h, box) : make_short4(0, -1, 0, -1);
        const uint32_t cnt = count_pairs(f, cam, v, rc);
        if (!in) continue;
        f.rect[iv] = rc;
        f.count[iv] = cnt;
        if (cnt == 0) continue;
        f.box[iv] = box;
        Record *r = f.rec + iv;
        r->r0 = make_float4((c0 - h) - cam.ro[0], (c1 - h) - cam.ro[1], (c2 - h) - cam.ro[2], vs);
        r->r1 = g0;
        r->r2 = g1;
    }
}

// --------------------------------------------------------------------- scan

// Block-wide exclusive scan of one value per thread (256 threads).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *warp_sums, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    uint32_t wpre = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint32_t s = warp_sums[w];
        wpre += (w < warp) ? s : 0u;
        tot += s;
    }
    __syncthreads();
    total = tot;
    return wpre + inc - x;
}

// Scan position i is sub-bucket i mod 2^sub_log2 of tile i / 2^sub_log2, stored
// sub-bucket-major (count[sub * ntiles + tile]).
__device__ __forceinline__ int64_t sub_index(const FrameDev &f, int64_t i) {
    return (i & ((1 << f.sub_log2) - 1)) * (int64_t)f.total_tiles + (i >> f.sub_log2);
}

// Sum of one 64-bit value per thread over the CTA (256 threads), in every thread.
__device__ __forceinline__ unsigned long long block_sum(unsigned long long x, unsigned long long *warp_sums) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = x;
    __syncthreads();
    x = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) x += warp_sums[w];
    return x;
}

// Sums of the scan blocks, `rounds` times 256 entries each (scan_rounds).  Also
// clears the counters of the work order and the sort for k_scan_down.
__global__ void __launch_bounds__(256) k_scan_reduce(FrameDev f, int rounds) {
    begin_kernel();
    __shared__ unsigned long long ws[8];
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i < (int)(sizeof(SortPlan) / 4); i += 256) reinterpret_cast<unsigned *>(f.plan)[i] = 0u;
        if (threadIdx.x == 0) f.status->slots_used = 0;
    }
    const int64_t n = (int64_t)f.total_tiles << f.sub_log2;
    unsigned long long acc = 0;
    for (int r = 0; r < rounds; ++r) {
        const int64_t i = ((int64_t)blockIdx.x * rounds + r) * kScanTile + threadIdx.x;
        if (i < n) acc += f.tile_cnt[sub_index(f, i)];
    }
    acc = block_sum(acc, ws);
    if (threadIdx.x == 0) f.scan_blocks[blockIdx.x] = acc;
}

// Sub-bucket starts (the emission cursors) from the counts, and per tile its
// range, its segments (with slots for a split list's) and its work-order
// group's count.  Each CTA first sums the block sums of all earlier CTAs, so no
// separate top-level scan is launched, and of all CTAs, so that every one
// knows whether the pairs exceed the capacity: then all ranges are empty and
// nothing is emitted, so it does not matter that the starts, 32-bit sums, wrap.
__global__ void __launch_bounds__(256) k_scan_down(FrameDev f, int nb, int rounds) {
    begin_kernel();
    __shared__ uint32_t ws[8];
    __shared__ unsigned long long wpre[8], wall[8];
    __shared__ unsigned group_cnt[2 * kOrderGroups], slots, slot0;
    const int t = threadIdx.x, lane = t & 31;
    if (t < 2 * kOrderGroups) group_cnt[t] = 0u;
    if (t == 0) slots = 0u;
    unsigned long long pre = 0, all = 0;
    for (int j = t; j < nb; j += 256) {
        const unsigned long long x = f.scan_blocks[j];
        all += x;
        if (j < (int)blockIdx.x) pre += x;
    }
    pre = block_sum(pre, wpre);
    all = block_sum(all, wall);
    const bool over = all > (unsigned long long)f.capacity;
    const int64_t n = (int64_t)f.total_tiles << f.sub_log2;
    uint32_t carry = (uint32_t)pre;
    for (int r = 0; r < rounds; ++r) {
        const int64_t i = ((int64_t)blockIdx.x * rounds + r) * kScanTile + t;
        const uint32_t x = i < n ? f.tile_cnt[sub_index(f, i)] : 0u;
        uint32_t tot;
        const uint32_t c = carry + block_exclusive_scan(x, ws, tot);
        if (i < n) f.cursor[sub_index(f, i)] = c;
        carry += tot;
        // the lanes of a tile's sub-buckets: the first one takes the tile
        const int last_sub = (1 << f.sub_log2) - 1;
        const uint32_t end = __shfl_sync(0xffffffffu, c + x, lane | last_sub);
        const bool tile = i < n && (i & last_sub) == 0;
        const uint2 rg = over || end == c ? make_uint2(0u, 0u) : make_uint2(c, end);
        const unsigned len = rg.y - rg.x;
        unsigned nseg = len > (unsigned)kSegLen ? (len + kSegLen - 1) / kSegLen : 1u, base = 0;
        if (tile && nseg > 1) base = atomicAdd(&slots, nseg);
        __syncthreads();
        if (t == 0) {
            slot0 = slots ? atomicAdd(&f.status->slots_used, slots) : 0u;
            slots = 0u;
        }
        __syncthreads();
        if (tile) {
            if (nseg > 1) {
                base += slot0;
                if ((int64_t)base + nseg > f.seg_slots) nseg = 1, base = 0;  // only past the pair capacity
            }
            const int bk = order_bucket(len, nseg);
            if (nseg > 1) {
                atomicAdd(&group_cnt[kFirstSeg + bk], 1u);
                atomicAdd(&group_cnt[bk], nseg - 1);
            } else {
                atomicAdd(&group_cnt[bk], 1u);
            }
            f.ranges[i >> f.sub_log2] = rg;
            f.tile_seg[i >> f.sub_log2] = make_uint2(nseg, base);
        }
    }
    __syncthreads();
    if (t < 2 * kOrderGroups && group_cnt[t]) atomicAdd(&f.plan->cnt[t], group_cnt[t]);
    if (blockIdx.x == 0 && t == 0) {
        f.status->n_pairs_lo = (unsigned)(all & 0xFFFFFFFFull);
        f.status->n_pairs_hi = (unsigned)(all >> 32);
        if (over) atomicOr(&f.status->flags, SVR_FLAG_CAPACITY);
    }
}

// --------------------------------------------------------------------- emit

// Bound by the round trips of the counts, rectangles and atomics, so by the
// warps that are resident: batches of four tiles take 48 registers, of eight
// 58.  8 views of 8M voxels 1502 -> 1185 us, 16 mixed views 492 -> 430, one view
// of 1M 45 -> 40 (batches of two: 1199, 438, 42); CTAs of 128 threads instead
// of 256: 1158, 423, 39, and a camera inside the scene 77 -> 73.  32 registers
// by launch bounds spill: 1440, 484, 50.
constexpr int kEmitBatch = 4;
constexpr int kEmitCoop = 4;   // tiles per lane of a cooperative batch (two: 1144 and 417, but 84 inside)
constexpr int kEmitThreads = 128;

// Writes the pairs of voxel v in tile g, whose sign patterns are m, from slot o.
__device__ __forceinline__ void write_pairs(const FrameDev &f, int g, unsigned m, uint32_t o, uint64_t code,
                                            uint32_t v) {
    if ((int64_t)o + __popc(m) > f.capacity) {  // counts and emission disagree: never expected
        atomicOr(&f.status->flags, SVR_FLAG_CAPACITY);
        return;
    }
    while (m) {
        const unsigned s = __ffs(m) - 1;
        m &= m - 1;
        if (f.vid_bits > 0) {
            f.keys[0][o] = pair_word(f, code, s, v);
        } else {
            f.keys[0][o] = ((uint64_t)g << f.key_shift) | ((code ^ ((uint64_t)s * kTripleOnes)) >> (48 - f.key_shift));
            f.vals[0][o] = (s << 29) | v;
        }
        ++o;
    }
}

// grid.y = view.  A voxel over more than kCoopTiles tiles is left to the warp.
__global__ void __launch_bounds__(kEmitThreads) k_emit(FrameDev f) {
    begin_kernel();
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f.status->flags & SVR_FLAG_CAPACITY) return;   // not raised here while the pairs fit
    const int view = blockIdx.y, lane = threadIdx.x & 31;
    const DevCam &cam = f.views[view];
    const int64_t iv = (int64_t)view * f.n_vox + v;
    short4 rc = make_short4(0, -1, 0, -1);
    uint64_t code = 0;
    if (v < f.n_vox && f.count[iv] != 0) {
        rc = f.rect[iv];
        code = f.octpath[v];
    }
    const int sub = (int)(v & ((1 << f.sub_log2) - 1));
    uint32_t *cur = f.cursor + (size_t)sub * f.total_tiles;
    const bool coop = rect_tiles(rc) > kCoopTiles;
    // the rectangle's tiles in row-major batches of kEmitBatch: a batch's
    // cursor atomics are issued together, so a voxel over several tiles waits
    // for one atomic round trip per batch rather than per tile
    int tx = rc.x, ty = rc.z;
    while (!coop && ty <= rc.w) {
        int gb[kEmitBatch];
        unsigned mb[kEmitBatch];
#pragma unroll
        for (int i = 0; i < kEmitBatch; ++i) {
            gb[i] = cam.tile_base + ty * cam.ntx + tx;
            mb[i] = ty <= rc.w && SVR_IN_BOUNDS(f.debug, kDbgTile, gb[i], f.total_tiles) ? (unsigned)f.tile_mask[gb[i]]
                                                                                   : 0u;
            if (++tx > rc.y) {
                tx = rc.x;
                ++ty;
            }
        }
        uint32_t ob[kEmitBatch];
#pragma unroll
        for (int i = 0; i < kEmitBatch; ++i) ob[i] = mb[i] ? atomicAdd(cur + gb[i], (uint32_t)__popc(mb[i])) : 0u;
#pragma unroll
        for (int i = 0; i < kEmitBatch; ++i) write_pairs(f, gb[i], mb[i], ob[i], code, (uint32_t)v);
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, coop); todo; todo &= todo - 1u) {
        const int src = __ffs(todo) - 1;
        const short4 q = shfl_rect(rc, src);
        const int w = q.y - q.x + 1, area = rect_tiles(q);
        const uint64_t qcode = __shfl_sync(0xffffffffu, code, src);
        const uint32_t qv = __shfl_sync(0xffffffffu, (uint32_t)v, src);
        uint32_t *to = f.cursor + (size_t)__shfl_sync(0xffffffffu, sub, src) * f.total_tiles;
        for (int i0 = lane; i0 < area; i0 += 32 * kEmitCoop) {
            int gb[kEmitCoop];
            unsigned mb[kEmitCoop];
            uint32_t ob[kEmitCoop];
#pragma unroll
            for (int j = 0; j < kEmitCoop; ++j) {
                const int i = i0 + 32 * j;
                gb[j] = cam.tile_base + (q.z + i / w) * cam.ntx + q.x + i % w;
                mb[j] = i < area && SVR_IN_BOUNDS(f.debug, kDbgTile, gb[j], f.total_tiles) ? (unsigned)f.tile_mask[gb[j]]
                                                                                         : 0u;
            }
#pragma unroll
            for (int j = 0; j < kEmitCoop; ++j) ob[j] = mb[j] ? atomicAdd(to + gb[j], (uint32_t)__popc(mb[j])) : 0u;
#pragma unroll
            for (int j = 0; j < kEmitCoop; ++j) write_pairs(f, gb[j], mb[j], ob[j], qcode, qv);
        }
    }
}

// ---------------------------------------------------------------- launchers

cudaError_t launch_tile_mask(const FrameDev &f, cudaStream_t s) {
    const int warps = tmin(f.total_tiles, kMaskWarps), per = kMaskThreads / 32;
    return launch(k_tile_mask, dim3((unsigned)((warps + per - 1) / per)), kMaskThreads, 0, s, f);
}

cudaError_t launch_preprocess(const FrameDev &f, cudaStream_t s) {
    if (f.n_vox == 0) return cudaSuccess;
    return launch(f.n_views == 1 ? k_preprocess : k_preprocess_views, dim3((unsigned)((f.n_vox + 127) / 128)), 128, 0, s,
                  f);
}

cudaError_t launch_scan(const FrameDev &f, cudaStream_t s) {
    const int64_t n = (int64_t)f.total_tiles << f.sub_log2;
    const int rounds = scan_rounds(n), nb = scan_blocks(n);
    static_assert(kScanTile == 256, "one entry per thread and round");
    const cudaError_t e = launch(k_scan_reduce, dim3(nb), 256, 0, s, f, rounds);
    return e != cudaSuccess ? e : launch(k_scan_down, dim3(nb), 256, 0, s, f, nb, rounds);
}

cudaError_t launch_emit(const FrameDev &f, cudaStream_t s) {
    if (f.n_vox == 0) return cudaSuccess;
    const dim3 grid((unsigned)((f.n_vox + kEmitThreads - 1) / kEmitThreads), (unsigned)f.n_views);
    return launch(k_emit, grid, kEmitThreads, 0, s, f);
}

}  // namespace svr
