// Volume lifetime, host transfer and projective TSDF fusion.
//
// Fusion follows the KinectFusion rule the paper adopts (Sec. III, "Method
// overview"): each node is transformed into the camera, projected to its
// nearest pixel, and, when that pixel has a usable depth d and the node lies
// no deeper than one truncation behind it, the truncated z-distance
// t = min(1, (d - z_c) / tau) enters a running average with weight 1.
//
// GB300 layout: tiles of 32 x 8 x 8 nodes (x fastest, so a warp touches one
// 128-byte line of each array per slice); a tile is dropped before any memory
// access when its box lies outside the view frustum, beyond depth_max + tau or
// (in grids of many tiles) behind every depth of the pixels it covers.  Node
// loads and stores happen only for nodes that pass every test, so HBM traffic
// is proportional to the nodes actually updated.  The camera-frame depth of a
// node is formed as a double-precision tile base (split into a float pair)
// plus a small float offset, which keeps the signed distance accurate to
// ~1e-7 m at any distance from the grid origin.
#include <stdlib.h>
#include <string.h>

#include <cstring>
#include <vector>

#include <type_traits>

#include "pf_internal.cuh"

namespace pf {
void align_release(const pf_volume* v);  // align.cu
}

namespace {

constexpr int TX = PF_TX, TY = PF_TY, TZ = PF_TZ;

struct IntegArgs {
    void* tsdf;
    void* weight;
    int nx, ny, nz;
    float trunc;
    float max_weight;
    CamK cam;
    const float* depth;
    const double* pose_dev;             // camera-to-world pose in device memory, or null: use pose
    double pose[12];                    // row-major 3x4
    double origin[3];
    double vs;
    float plane[4][3];                  // inward normals of the four side planes of the frustum
    float zfar;                         // nodes deeper than this are never updated
    float margin;                       // added to a tile's half sides in the culls
    int* tile_stamp;                    // tiles with a changed node value get *stamp_dev (null: no cell view)
    const int* stamp_dev;               // fusion counter on the device
    int tiles[3];                       // fusion tiles per axis
    FusionList list;                    // tiles that survive the cull, with their bases
    SurfaceMap surf;
};

// Starts a fusion: empties the tile lists and, with a cell view, advances the
// fusion counter the tile stamps refer to (on the device, so a captured and
// replayed launch sequence still marks each fusion apart).  The launch of a
// fusion with the depth cull also reduces the image to its blocks' largest
// usable depths (0: none), one warp a block; without an image one CTA only
// empties the lists.
constexpr int BEGIN_WARPS = 8;

__global__ void __launch_bounds__(32 * BEGIN_WARPS) fusion_begin_kernel(FusionList list, int* stamp_counter,
                                                                       const float* __restrict__ depth, CamK cam)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        list.count[0] = 0;
        list.count[1] = 0;
        if (stamp_counter) *stamp_counter += 1;
    }
    if (!depth) return;
    const int b = blockIdx.x * BEGIN_WARPS + (threadIdx.x >> 5);
    const int bw = (cam.width + PF_DEPTH_BLOCKS - 1) / PF_DEPTH_BLOCKS;
    const int bh = (cam.height + PF_DEPTH_BLOCKS - 1) / PF_DEPTH_BLOCKS;
    const int u0 = b % PF_DEPTH_BLOCKS * bw, v0 = b / PF_DEPTH_BLOCKS * bh;
    float m = 0.0f;
    for (int p = threadIdx.x & 31; p < bw * bh; p += 32) {
        const int u = u0 + p % bw, v = v0 + p / bw;
        if (u >= cam.width || v >= cam.height) continue;
        const float z = __ldg(depth + (size_t)v * cam.width + u);
        if (pf_depth_usable(z, cam.dmin, cam.dmax)) m = fmaxf(m, z);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) list.depth_max[b] = m;
}

// Whether every pixel that a node of a tile can project to lacks a usable
// depth or has one more than the truncation in front of the whole tile: then
// no node of it is updated.  c, e: centre and half sides of the tile's bounding
// box along the camera's axes.  A tile that reaches the camera plane or covers
// many blocks is kept without a look.
__device__ inline bool tile_occluded(const IntegArgs& a, const float* c, const float* e)
{
    if (!a.list.depth_max) return false;
    const float zn = c[2] - e[2], zf = c[2] + e[2];
    if (!(zn > 0.0f)) return false;
    // pixel bounds of the box over its depth range, one pixel wider
    const float x0 = c[0] - e[0], x1 = c[0] + e[0], y0 = c[1] - e[1], y1 = c[1] + e[1];
    const float u0 = floorf(a.cam.fx * x0 / (x0 < 0.0f ? zn : zf) + a.cam.cx - 1.0f);
    const float u1 = floorf(a.cam.fx * x1 / (x1 > 0.0f ? zn : zf) + a.cam.cx + 2.0f);
    const float v0 = floorf(a.cam.fy * y0 / (y0 < 0.0f ? zn : zf) + a.cam.cy - 1.0f);
    const float v1 = floorf(a.cam.fy * y1 / (y1 > 0.0f ? zn : zf) + a.cam.cy + 2.0f);
    if (!(u1 - u0 < 1e9f && v1 - v0 < 1e9f)) return false;
    const int bw = (a.cam.width + PF_DEPTH_BLOCKS - 1) / PF_DEPTH_BLOCKS;
    const int bh = (a.cam.height + PF_DEPTH_BLOCKS - 1) / PF_DEPTH_BLOCKS;
    const int bu0 = (int)fmaxf(u0, 0.0f) / bw, bu1 = (int)fminf(u1, (float)(a.cam.width - 1)) / bw;
    const int bv0 = (int)fmaxf(v0, 0.0f) / bh, bv1 = (int)fminf(v1, (float)(a.cam.height - 1)) / bh;
    if (u1 < 0.0f || v1 < 0.0f || u0 > (float)(a.cam.width - 1) || v0 > (float)(a.cam.height - 1)) return true;
    if ((bu1 - bu0 + 1) * (bv1 - bv0 + 1) > 64) return false;
    float m = 0.0f;
    for (int bv = bv0; bv <= bv1; ++bv)
        for (int bu = bu0; bu <= bu1; ++bu) m = fmaxf(m, __ldg(a.list.depth_max + bv * PF_DEPTH_BLOCKS + bu));
    return fmaf(m, 1.000001f, a.trunc) < zn;  // (the half sides carry the margin for rounding)
}

// One thread per fusion tile of TX x TY x TZ nodes: two culls of the tile's
// box, by the frustum and (large grids) by the image's depths, and for a tile
// that survives the camera-frame position of its first node,
// X_c = R^T (X_w - t) with X_w = origin + vs (i0, j0, k0), in FP64 -- kept as
// floats, the depth as a hi + lo pair -- which is appended to the list (its
// position in the list depends on scheduling; each tile's nodes are fused
// once whatever the order, so the result does not).  The culls run in float
// from the grid's first tile and the steps between tiles, formed in FP64 once
// per CTA: FP64 for every tile was the kernel's whole time (221 184 tiles of a
// 768^3 grid: 21.2 -> 12.9 us from cold caches, with the depth cull added).
// A thread of the first CTA also writes the per-index steps, vs times the
// rows of R, which every tile shares.
__global__ void __launch_bounds__(256) fusion_tiles_kernel(IntegArgs a)
{
    __shared__ double s_P[12];
    __shared__ float s_c[12];  // centre of the first tile, steps between tiles along x, y, z
    __shared__ float s_e[7];   // half sides of a tile's box along the camera's axes; its reach along the side planes' normals
    const double* P = a.pose_dev ? a.pose_dev : a.pose;
    if (threadIdx.x < 12) s_P[threadIdx.x] = P[threadIdx.x];
    __syncthreads();
    if (threadIdx.x < 3) {
        const int r = threadIdx.x;
        const double d[3] = {a.origin[0] - s_P[3], a.origin[1] - s_P[7], a.origin[2] - s_P[11]};
        const double si = a.vs * s_P[r], sj = a.vs * s_P[4 + r], sk = a.vs * s_P[8 + r];
        s_c[r] = (float)(s_P[r] * d[0] + s_P[4 + r] * d[1] + s_P[8 + r] * d[2] +
                         0.5 * ((TX - 1) * si + (TY - 1) * sj + (TZ - 1) * sk));
        s_c[3 + r] = (float)(TX * si);
        s_c[6 + r] = (float)(TY * sj);
        s_c[9 + r] = (float)(TZ * sk);
        if (blockIdx.x == 0) {
            a.list.step[r] = (float)si;
            a.list.step[3 + r] = (float)sj;
            a.list.step[6 + r] = (float)sk;
        }
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        // margin: a voxel's hundredth and a millimetre, and a few roundings of
        // the float centre's terms
        const float margin = a.margin + 1e-6f * (fabsf(s_c[0]) + fabsf(s_c[1]) + fabsf(s_c[2]) +
                                                 (float)a.vs * (float)(a.nx + a.ny + a.nz));
        const int p = (int)threadIdx.x - 3;
        const float n[3] = {p < 0 ? (threadIdx.x == 0 ? 1.0f : 0.0f) : a.plane[p][0],
                            p < 0 ? (threadIdx.x == 1 ? 1.0f : 0.0f) : a.plane[p][1],
                            p < 0 ? (threadIdx.x == 2 ? 1.0f : 0.0f) : a.plane[p][2]};
        float e = margin;
        for (int x = 0; x < 3; ++x) {  // half a tile along the grid's axis x: its first to its last node
            const float half = 0.5f * (x == 0 ? (TX - 1.0f) / TX : x == 1 ? (TY - 1.0f) / TY : (TZ - 1.0f) / TZ);
            const float* st = s_c + 3 + 3 * x;
            e += half * fabsf(n[0] * st[0] + n[1] * st[1] + n[2] * st[2]);
        }
        s_e[threadIdx.x] = e;
    }
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int n_tiles = a.tiles[0] * a.tiles[1] * a.tiles[2];
    if (t >= n_tiles) return;
    const int bx = t % a.tiles[0], by = (t / a.tiles[0]) % a.tiles[1], bz = t / (a.tiles[0] * a.tiles[1]);
    float c[3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
        c[r] = fmaf((float)bx, s_c[3 + r], fmaf((float)by, s_c[6 + r], fmaf((float)bz, s_c[9 + r], s_c[r])));
    bool skip = (c[2] + s_e[2] <= 0.0f) || (c[2] - s_e[2] > a.zfar);
    for (int p = 0; p < 4 && !skip; ++p) {
        const float dd = a.plane[p][0] * c[0] + a.plane[p][1] * c[1] + a.plane[p][2] * c[2];
        if (dd < -s_e[3 + p]) skip = true;
    }
    if (skip || tile_occluded(a, c, s_e)) return;
    const int i0 = bx * TX, j0 = by * TY, k0 = bz * TZ;
    const double Xw[3] = {a.origin[0] + a.vs * i0, a.origin[1] + a.vs * j0, a.origin[2] + a.vs * k0};
    const double d[3] = {Xw[0] - s_P[3], Xw[1] - s_P[7], Xw[2] - s_P[11]};
    double b[3];
    for (int r = 0; r < 3; ++r) b[r] = s_P[r] * d[0] + s_P[4 + r] * d[1] + s_P[8 + r] * d[2];
    const float hi = (float)b[2];
    const int slot = atomicAdd(a.list.count, 1);
    a.list.tile[slot] = t;
    a.list.base[slot] = make_float4((float)b[0], (float)b[1], hi, (float)(b[2] - (double)hi));
}

template <typename T>
__device__ __forceinline__ bool same_bits(T x, T y)
{
    unsigned bx = 0u, by = 0u;
    memcpy(&bx, &x, sizeof(T));
    memcpy(&by, &y, sizeof(T));
    return bx == by;
}

// floor(x) of a pixel coordinate from the low mantissa bits of x + 2^23
// rounded down: one addition instead of a conversion, of which the SM issues a
// quarter as many.  Exact for 0 <= x < 2^23; any other x (negative, larger, not
// a number) gives an unsigned value above every image side (at most 16384).
__device__ __forceinline__ unsigned pixel_floor(float x)
{
    return (unsigned)__float_as_int(__fadd_rd(x, 8388608.0f)) - 0x4b000000u;
}

// min(w + 1, max_weight)
__device__ __forceinline__ float next_weight(float w, float max_weight) { return fminf(w + 1.0f, max_weight); }
__device__ __forceinline__ uint8_t next_weight(uint8_t w, float max_weight)
{
    return (uint8_t)min((int)w + 1, (int)max_weight);
}

// Nodes of a column taken together by the fusion kernel.
constexpr int BATCH = 4;

// Fusion of the listed tiles; a fixed grid of CTAs walks the list.  Thread
// (tx, ty) of a tile owns the column of TZ nodes (i0 + tx, j0 + ty, k0 + dz).
// With a cell view, the rows of nodes where a stored value changed are noted
// and a tile that has one is stamped with the fusion counter (by every warp
// that changed one: the same value); a fused node whose value stays -- free
// space seen again, still outside the band -- changes only its weight, which
// no cell record holds, so its row's records need no rewrite.
// Bound by issue: about 23 million nodes of a 640x480 frame project into the
// image at 768^3, nearly all of them free space seen again, so that path has no
// division, no conversion and no store but the weight's (262 instructions a
// node before, about 85 now), and the four nodes of a batch wait for memory
// together.  A 640x480 frame into 768^3 half precision, a frame that the map
// has seen before: 241 -> 148 us from cold caches; with the refresh and a
// 160x120 ray cast, 459 -> 221 us.  Frames of a camera that moves on change
// more: with the refresh, 100 distinct views of a room, the last 50 of them,
// 470 -> 312 us (512^3 float 231 -> 135).
template <typename TS, typename TW>
__global__ void __launch_bounds__(TX * TY, 4) integrate_kernel(IntegArgs a)
{
    TS* const tsdf = static_cast<TS*>(a.tsdf);
    TW* const weight = static_cast<TW*>(a.weight);
    const int n_active = *a.list.count;
    const int stamp = a.tile_stamp ? *a.stamp_dev : 0;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const float ai[3] = {a.list.step[0], a.list.step[1], a.list.step[2]};
    const float aj[3] = {a.list.step[3], a.list.step[4], a.list.step[5]};
    const float ak[3] = {a.list.step[6], a.list.step[7], a.list.step[8]};
    const float lx = fmaf((float)tx, ai[0], (float)ty * aj[0]);
    const float ly = fmaf((float)tx, ai[1], (float)ty * aj[1]);
    const float lz = fmaf((float)tx, ai[2], (float)ty * aj[2]);
    const unsigned plane_stride = (unsigned)a.nx * (unsigned)a.ny;  // (fewer than 2^31 nodes)
    for (int e = blockIdx.x; e < n_active; e += gridDim.x) {
        const int t = a.list.tile[e];
        const float4 base = a.list.base[e];
        const int bx = t % a.tiles[0], by = (t / a.tiles[0]) % a.tiles[1], bz = t / (a.tiles[0] * a.tiles[1]);
        const int i = bx * TX + tx, j = by * TY + ty, k0 = bz * TZ;
        const bool inside = i < a.nx && j < a.ny;
        const float bx_ = base.x, by_ = base.y, bz_hi = base.z, bz_lo = base.w;
        unsigned idx = (unsigned)i + (unsigned)a.nx * (unsigned)j + plane_stride * (unsigned)k0;
        const int planes = min(TZ, a.nz - k0);
        const float lxi = inside ? lx : NAN;  // (a column outside the grid projects to no pixel)
        unsigned changed = 0u;  // bit dz: the node's stored value changed
        unsigned solid = 0u;    // bit dz: the node's new value is zero or negative
#pragma unroll 1
        for (int h = 0; h < TZ; h += BATCH) {
            // a batch's pixels, then its depths, then its nodes: each group of
            // loads waits once
            int pix[BATCH];
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                const float fz = (float)(h + q);
                const float xc = bx_ + fmaf(fz, ak[0], lxi);
                const float yc = by_ + fmaf(fz, ak[1], ly);
                const float zc = bz_hi + (bz_lo + fmaf(fz, ak[2], lz));
                const float inv = __frcp_rn(zc);
                const unsigned u = pixel_floor(fmaf(a.cam.fx * xc, inv, a.cam.cx) + 0.5f);
                const unsigned v = pixel_floor(fmaf(a.cam.fy * yc, inv, a.cam.cy) + 0.5f);
                const bool in = u < (unsigned)a.cam.width && v < (unsigned)a.cam.height && zc > 0.0f && h + q < planes;
                pix[q] = in ? (int)(v * (unsigned)a.cam.width + u) : -1;
            }
            float sdf[BATCH];
#pragma unroll
            for (int q = 0; q < BATCH; ++q) sdf[q] = pix[q] >= 0 ? __ldg(a.depth + pix[q]) : NAN;
            bool upd[BATCH];
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                const float d = sdf[q];
                sdf[q] = (d - bz_hi) - (bz_lo + fmaf((float)(h + q), ak[2], lz));
                // (depth_max is finite, so the bounds reject NaN and infinity too)
                upd[q] = d >= a.cam.dmin && d <= a.cam.dmax && !(sdf[q] < -a.trunc);
            }
            const TS open = pf_from_float<TS>(INFINITY);  // the code of +1
            TW w_old[BATCH];
            TS t_old[BATCH];
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                w_old[q] = upd[q] ? weight[idx + plane_stride * q] : TW(0);
                t_old[q] = upd[q] ? tsdf[idx + plane_stride * q] : open;
            }
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                // free space seen again: the average of +1 and +1 is +1
                // (w 1 + 1 and w + 1 are the same float), stored as it was
                TS stored = open;
                if (upd[q] && !(sdf[q] >= a.trunc && (w_old[q] == TW(0) || same_bits(t_old[q], open)))) {
                    const float w = pf_to_float(w_old[q]);
                    const float tt = fminf(1.0f, __fdiv_rn(sdf[q], a.trunc));
                    float tn = tt;
                    if (w > 0.0f) tn = __fdiv_rn(fmaf(w, pf_decode(pf_to_float(t_old[q])), tt), w + 1.0f);
                    stored = pf_from_float<TS>(pf_encode(tn, 1.0f));
                    solid |= pf_to_float(stored) <= 0.0f ? 1u << (h + q) : 0u;
                }
                if (upd[q] && !same_bits(stored, t_old[q])) {
                    changed |= 1u << (h + q);
                    tsdf[idx + plane_stride * q] = stored;
                }
                const TW w_new = next_weight(w_old[q], a.max_weight);
                if (upd[q] && w_new != w_old[q]) weight[idx + plane_stride * q] = w_new;
            }
            idx += plane_stride * BATCH;
        }
        if (a.tile_stamp) {
            // the warp's rows: byte ty of the tile's word
            changed = __reduce_or_sync(0xffffffffu, changed);
            if (tx == 0) {
                reinterpret_cast<unsigned char*>(a.list.rows + t)[ty] = (unsigned char)changed;
                if (changed) a.tile_stamp[t] = stamp;
            }
        }
        pf_mark_surface(a.surf, __ballot_sync(0xffffffffu, solid != 0u), __ballot_sync(0xffffffffu, (solid & 1u) != 0u),
                        bx * TX, j, k0);
    }
}

// The surface map of a whole grid (after an upload): the tiles of fusion,
// one CTA at a time, every node read once.
template <typename TS>
__global__ void __launch_bounds__(TX * TY) surface_scan_kernel(const void* tsdf_, int nx, int ny, int nz, int tiles_x,
                                                               int tiles_y, int n_tiles, SurfaceMap surf)
{
    const TS* tsdf = static_cast<const TS*>(tsdf_);
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int i0 = t % tiles_x * TX, j = (t / tiles_x) % tiles_y * TY + threadIdx.y, k0 = t / (tiles_x * tiles_y) * TZ;
        const int i = i0 + threadIdx.x;
        unsigned solid = 0u;
        if (i < nx && j < ny) {
            const TS* p = tsdf + i + (size_t)nx * (j + (size_t)ny * k0);
            for (int dz = 0; dz < min(TZ, nz - k0); ++dz)
                solid |= pf_to_float(p[(size_t)nx * ny * dz]) <= 0.0f ? 1u << dz : 0u;
        }
        pf_mark_surface(surf, __ballot_sync(0xffffffffu, solid != 0u), __ballot_sync(0xffffffffu, (solid & 1u) != 0u),
                        i0, j, k0);
    }
}

template <typename TS, typename TW>
__global__ void fill_kernel(void* tsdf_, void* weight_, size_t n)
{
    TS* tsdf = static_cast<TS*>(tsdf_);
    TW* weight = static_cast<TW*>(weight_);
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    size_t step = (size_t)gridDim.x * blockDim.x;
    for (; i < n; i += step) {
        tsdf[i] = pf_from_float<TS>(PF_UNOBSERVED);
        weight[i] = pf_from_float<TW>(0.0f);
    }
}

// Cell view: for every cell (lower corner node i, j, k) its eight encoded
// corner values with the x-differences the interpolation needs already
// formed: float4 (v000, v100 - v000, v010, v110 - v010) and float4 (v001,
// v101 - v001, v011, v111 - v011).  The subtraction is the same float
// operation the fitness would do, so results are bit-identical, and a
// non-finite corner still makes the interpolated value non-finite.  A cell
// depends on the nodes of its own row and of the next rows along +y and +z
// (and, for a tile's last cell, on the next tile along +x), so a row of a
// tile's records is rewritten when a node value of any of those was changed by
// the last fusion (or always, after a reset or upload).
struct RefreshArgs {
    const void* tsdf;
    void* cells;
    float* cells32;  // 16-/8-bit grids, full view: the float records as well
    int nx, ny, nz;
    int row, plane;  // pitch of the records
    const int* tile_stamp;
    const int* stamp_dev;
    int all;
    int tiles[3];
    FusionList list;  // list.refresh_tile / count[1]: the tiles to rewrite
};

// One thread per tile: which of its rows of records are to be rewritten, from
// the changed rows of the tile and of its neighbours along +x, +y, +z (whose
// nodes its cells reach) in the last fusion, or all of them (all).  Order of
// the list as in fusion_tiles_kernel: any, with the same result.
__global__ void __launch_bounds__(256) refresh_tiles_kernel(RefreshArgs a)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int n_tiles = a.tiles[0] * a.tiles[1] * a.tiles[2];
    if (t >= n_tiles) return;
    const int bx = t % a.tiles[0], by = (t / a.tiles[0]) % a.tiles[1], bz = t / (a.tiles[0] * a.tiles[1]);
    const int stamp = *a.stamp_dev;
    unsigned long long r[4] = {0, 0, 0, 0};  // changed rows of this tile, +y, +z, +y+z (each with its +x neighbour)
    for (int q = 0; q < 8 && !a.all; ++q) {
        const int x = bx + (q & 1), y = by + ((q >> 1) & 1), z = bz + (q >> 2);
        if (x >= a.tiles[0] || y >= a.tiles[1] || z >= a.tiles[2]) continue;
        const int n = x + a.tiles[0] * (y + a.tiles[1] * z);
        if (a.tile_stamp[n] == stamp) r[q >> 1] |= a.list.rows[n];
    }
    const unsigned long long first = 0x0101010101010101ull;  // bit 0 (k = 0) of each byte (j)
    const unsigned long long up = (r[0] >> 8) | (r[1] << 56), up_z = (r[2] >> 8) | (r[3] << 56);  // rows j + 1
    const unsigned long long self = r[0] | up, self_z = r[2] | up_z;
    const unsigned long long rows = a.all ? ~0ull : self | ((self >> 1) & ~(first << 7)) | ((self_z & first) << 7);
    if (rows != 0ull) {
        const int slot = atomicAdd(a.list.count + 1, 1);
        a.list.refresh_tile[slot] = t;
        a.list.refresh_rows[slot] = rows;
    }
}

// One cell-view record from its corners c (v000, v100, v010, v110 of plane k
// in lo, the same of plane k + 1 in hi), TV the view's type.  Float records
// hold the corners with the x-differences precomputed (v000, v100 - v000,
// v010, v110 - v010 | v001, v101 - v001, v011, v111 - v011).  Narrow records
// hold the eight values as stored, 16 or 8 bytes; the reader forms the
// differences in float, so the fitness sees exactly the stored grid (a
// difference rounded to 16 bits would not be).  The full view of a narrow grid
// has the float record as well, formed from the stored values converted
// exactly, so both records of a cell give the same samples.
__device__ __forceinline__ void store_float_record(float* cells, size_t rec, const float* lo, const float* hi)
{
    // one 32-byte sector, one store
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
        :: "l"(cells + 8 * rec), "f"(lo[0]), "f"(lo[1] - lo[0]), "f"(lo[2]), "f"(lo[3] - lo[2]),
           "f"(hi[0]), "f"(hi[1] - hi[0]), "f"(hi[2]), "f"(hi[3] - hi[2]) : "memory");
}

template <typename TV>
__device__ __forceinline__ void store_record(TV* cells, float* cells32, size_t rec, const TV* lo, const TV* hi)
{
    if constexpr (std::is_same<TV, float>::value) {
        store_float_record(cells, rec, lo, hi);
    } else {
        const TV h[8] = {lo[0], lo[1], lo[2], lo[3], hi[0], hi[1], hi[2], hi[3]};
        if constexpr (sizeof(TV) == 2) {
            uint4 w;
            memcpy(&w, h, 16);
            reinterpret_cast<uint4*>(cells)[rec] = w;
        } else {
            uint2 w;
            memcpy(&w, h, 8);
            reinterpret_cast<uint2*>(cells)[rec] = w;
        }
        if (cells32) {
            float fl[4], fh[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                fl[c] = pf_to_float(lo[c]);
                fh[c] = pf_to_float(hi[c]);
            }
            store_float_record(cells32, rec, fl, fh);
        }
    }
}

// TS: storage of the node array; TV: storage of the view (TS itself, or a
// narrower type for the search view of a float grid: each node value rounded
// once with the storage rule, a value that rounds to +-1 becoming the
// outside-the-band code).  A fixed grid of CTAs walks the list of tiles to
// rewrite; a warp owns the eight rows of records (j, k0 .. k0 + 7).  Bound by
// the records written (32 to 48 bytes a cell).  Each plane's four nodes are
// read once and serve the cells below and above it, and only rows with a
// changed corner are read and written (whole tiles before): a 640x480 frame's
// refresh of a 768^3 half-precision grid 274 -> 130 us from cold caches (a frame
// that the map has seen before).
constexpr int HALF = TZ / 2;

template <typename TS, typename TV>
__global__ void __launch_bounds__(TX * TY, 4) cells_refresh_kernel(RefreshArgs a)
{
    const int n_list = a.list.count[1];
    const TS* __restrict__ tsdf = static_cast<const TS*>(a.tsdf);
    TV* cells = static_cast<TV*>(a.cells);
    const size_t nx = a.nx, nxy = (size_t)a.nx * a.ny;
    for (int e = blockIdx.x; e < n_list; e += gridDim.x) {
        const unsigned rows = (unsigned)(a.list.refresh_rows[e] >> (8 * threadIdx.y)) & 0xffu;
        if (rows == 0u) continue;
        const int t = a.list.refresh_tile[e];
        const int bx = t % a.tiles[0], by = (t / a.tiles[0]) % a.tiles[1], bz = t / (a.tiles[0] * a.tiles[1]);
        const int i = bx * TX + threadIdx.x, j = by * TY + threadIdx.y, k0 = bz * TZ;
        if (i >= a.nx - 1 || j >= a.ny - 1) continue;
        const unsigned planes = rows | (rows << 1);  // node planes k0 + dz that the rows touch
        const size_t idx = i + nx * j + nxy * k0;
        const size_t rec = i + (size_t)a.row * j + (size_t)a.plane * k0;
#pragma unroll 1
        for (int h = 0; h < TZ; h += HALF) {
            if ((rows >> h & ((1u << HALF) - 1u)) == 0u) continue;
            TV v[HALF + 1][4];
#pragma unroll
            for (int dz = 0; dz <= HALF; ++dz)
                if ((planes >> (h + dz) & 1u) && k0 + h + dz < a.nz) {
                    const TS* p = tsdf + idx + nxy * (h + dz);
                    const TS n[4] = {p[0], p[1], p[nx], p[nx + 1]};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if constexpr (std::is_same<TS, TV>::value)
                            v[dz][c] = n[c];
                        else
                            v[dz][c] = pf_from_float<TV>(n[c]);
                    }
                }
#pragma unroll
            for (int dz = 0; dz < HALF; ++dz)
                if ((rows >> (h + dz) & 1u) && k0 + h + dz < a.nz - 1)
                    store_record(cells, a.cells32, rec + (size_t)a.plane * (h + dz), v[dz], v[dz + 1]);
        }
    }
}

// CTAs of the list-walking fusion and refresh kernels: 4 per SM.
int list_ctas(const pf_volume* v) { return 4 * v->sms; }

pf_status enqueue_refresh(pf_volume* v, cudaStream_t s, int all)
{
    if (!v->cells) return PF_OK;
    RefreshArgs r;
    r.tsdf = v->tsdf;
    r.cells = v->cells;
    r.cells32 = v->cells32;
    r.nx = v->desc.nx;
    r.ny = v->desc.ny;
    r.nz = v->desc.nz;
    r.row = v->pitch.row;
    r.plane = v->pitch.plane;
    const int n_tiles = v->tiles[0] * v->tiles[1] * v->tiles[2];
    r.tile_stamp = v->tile_stamp;
    r.stamp_dev = v->tile_stamp + n_tiles;
    r.all = all;
    for (int q = 0; q < 3; ++q) r.tiles[q] = v->tiles[q];
    r.list = v->list;
    if (all) {  // outside a fusion: the list counter was not reset by fusion_begin_kernel
        fusion_begin_kernel<<<1, 32, 0, s>>>(v->list, nullptr, nullptr, CamK());
        pf::count_launch();
    }
    refresh_tiles_kernel<<<(n_tiles + 255) / 256, 256, 0, s>>>(r);
    pf::count_launch();
    const int grid = list_ctas(v);
    const dim3 blk(TX, TY);
    if (v->desc.tsdf_dtype != pf_view_dtype(v)) {  // the search view of a float grid
        switch (pf_view_dtype(v)) {
        case PF_F16: cells_refresh_kernel<float, __half><<<grid, blk, 0, s>>>(r); break;
        case PF_BF16: cells_refresh_kernel<float, __nv_bfloat16><<<grid, blk, 0, s>>>(r); break;
        default: cells_refresh_kernel<float, __nv_fp8_e4m3><<<grid, blk, 0, s>>>(r); break;
        }
    } else {
        switch (v->desc.tsdf_dtype) {
        case PF_F16: cells_refresh_kernel<__half, __half><<<grid, blk, 0, s>>>(r); break;
        case PF_BF16: cells_refresh_kernel<__nv_bfloat16, __nv_bfloat16><<<grid, blk, 0, s>>>(r); break;
        case PF_FP8E4M3: cells_refresh_kernel<__nv_fp8_e4m3, __nv_fp8_e4m3><<<grid, blk, 0, s>>>(r); break;
        default: cells_refresh_kernel<float, float><<<grid, blk, 0, s>>>(r); break;
        }
    }
    pf::count_launch();
    PF_LAUNCHED();
    return PF_OK;
}

// Launch a kernel templated on (tsdf storage, weight storage) for volume v.
template <template <typename, typename> class K, typename... Args>
void dispatch_storage(const pf_volume* v, Args&&... args)
{
    const bool u8 = v->desc.weight_u8 != 0;
    switch (v->desc.tsdf_dtype) {
    case PF_F16:
        if (u8) K<__half, uint8_t>::run(args...); else K<__half, float>::run(args...);
        break;
    case PF_BF16:
        if (u8) K<__nv_bfloat16, uint8_t>::run(args...); else K<__nv_bfloat16, float>::run(args...);
        break;
    case PF_FP8E4M3:
        if (u8) K<__nv_fp8_e4m3, uint8_t>::run(args...); else K<__nv_fp8_e4m3, float>::run(args...);
        break;
    default:
        if (u8) K<float, uint8_t>::run(args...); else K<float, float>::run(args...);
        break;
    }
}

template <typename TS, typename TW>
struct FillLaunch {
    static void run(void* tsdf, void* weight, size_t n, cudaStream_t s)
    {
        fill_kernel<TS, TW><<<152 * 8, 256, 0, s>>>(tsdf, weight, n);
    }
};

template <typename TS, typename TW>
struct IntegrateLaunch {
    static void run(int grid, const IntegArgs& a, cudaStream_t s)
    {
        integrate_kernel<TS, TW><<<grid, dim3(TX, TY), 0, s>>>(a);
    }
};

pf_status check_desc(const pf_volume_desc* d)
{
    if (!d) return PF_ERR_INVALID_ARG;
    if (d->nx < 2 || d->ny < 2 || d->nz < 2 || d->nx > 4096 || d->ny > 4096 || d->nz > 4096)
        return PF_ERR_INVALID_ARG;
    if ((double)d->nx * d->ny * d->nz >= 2147483648.0) return PF_ERR_INVALID_ARG;
    if (!(d->voxel_size > 0.0f) || !(d->trunc > 0.0f) || !std::isfinite(d->voxel_size) || !std::isfinite(d->trunc))
        return PF_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(d->origin[a])) return PF_ERR_INVALID_ARG;
    if (d->max_weight < 1 || d->max_weight > 65535) return PF_ERR_INVALID_ARG;
    if (d->cell_view < -1 || d->cell_view > 2) return PF_ERR_INVALID_ARG;
    if (d->weight_u8 != 0 && d->weight_u8 != 1) return PF_ERR_INVALID_ARG;
    if (d->weight_u8 && d->max_weight > 255) return PF_ERR_INVALID_ARG;
    if (d->tsdf_dtype != PF_F32 && d->tsdf_dtype != PF_F16 && d->tsdf_dtype != PF_BF16 &&
        d->tsdf_dtype != PF_FP8E4M3)
        return PF_ERR_UNSUPPORTED;
    // a search view narrower than the storage: float grids only, and it
    // needs a cell view
    if (d->search_dtype != PF_F32 && d->search_dtype != d->tsdf_dtype) {
        if (d->search_dtype != PF_F16 && d->search_dtype != PF_BF16 && d->search_dtype != PF_FP8E4M3)
            return PF_ERR_UNSUPPORTED;
        if (d->tsdf_dtype != PF_F32) return PF_ERR_UNSUPPORTED;
        if (d->cell_view == -1) return PF_ERR_INVALID_ARG;
    }
    return PF_OK;
}

size_t surface_bytes(const SurfaceMap& m) { return sizeof(unsigned long long) * m.wx * m.wy * (size_t)m.wz; }

pf_status enqueue_surface_scan(pf_volume* v, cudaStream_t s)
{
    PF_CUDA(cudaMemsetAsync(v->surf.words, 0, surface_bytes(v->surf), s));
    const int n_tiles = v->tiles[0] * v->tiles[1] * v->tiles[2];
    const dim3 blk(TX, TY);
    auto scan = [&](auto kernel) {
        kernel<<<list_ctas(v), blk, 0, s>>>(v->tsdf, v->desc.nx, v->desc.ny, v->desc.nz, v->tiles[0],
                                                    v->tiles[1], n_tiles, v->surf);
    };
    switch (v->desc.tsdf_dtype) {
    case PF_F16: scan(surface_scan_kernel<__half>); break;
    case PF_BF16: scan(surface_scan_kernel<__nv_bfloat16>); break;
    case PF_FP8E4M3: scan(surface_scan_kernel<__nv_fp8_e4m3>); break;
    default: scan(surface_scan_kernel<float>); break;
    }
    pf::count_launch();
    PF_LAUNCHED();
    return PF_OK;
}

pf_status enqueue_reset(pf_volume* v, cudaStream_t s)
{
    PF_CUDA(cudaMemsetAsync(v->surf.words, 0, surface_bytes(v->surf), s));
    dispatch_storage<FillLaunch>(v, v->tsdf, v->weight, v->n_nodes, s);
    pf::count_launch();
    PF_LAUNCHED();
    return enqueue_refresh(v, s, 1);
}

void free_list(FusionList& l)
{
    cudaFree(l.count);
    cudaFree(l.tile);
    cudaFree(l.base);
    cudaFree(l.step);
    cudaFree(l.depth_max);
    cudaFree(l.rows);
    cudaFree(l.refresh_tile);
    cudaFree(l.refresh_rows);
    l = FusionList();
}

bool finite_pose(const double* P)
{
    for (int i = 0; i < 12; ++i)
        if (!std::isfinite(P[i])) return false;
    return true;
}

}  // namespace

extern "C" {

pf_status pf_create_volume(const pf_volume_desc* desc, void* stream, pf_volume** out)
{
    if (!out) return PF_ERR_INVALID_ARG;
    *out = nullptr;
    pf_status st = check_desc(desc);
    if (st != PF_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    pf_volume* v = new pf_volume();
    v->desc = *desc;
    v->n_nodes = (size_t)desc->nx * desc->ny * desc->nz;
    v->tiles[0] = (desc->nx + TX - 1) / TX;
    v->tiles[1] = (desc->ny + TY - 1) / TY;
    v->tiles[2] = (desc->nz + TZ - 1) / TZ;
    const size_t ts = pf_dtype_size(desc->tsdf_dtype), ws = desc->weight_u8 ? 1 : 4;
    const pf_dtype vdt = pf_view_dtype(v);
    const size_t vs = pf_dtype_size(vdt);
    // the full view of a 16-/8-bit grid keeps both its narrow records (lanes
    // on points: two or four records per sector) and float records (lanes on
    // particles: no conversions); the narrow view keeps the narrow records
    // only; a float grid has the float records only
    const size_t rec = 8 * vs, rec32 = vdt == PF_F32 ? 0 : 32;
    pf::CellView cv = {desc->cell_view, pf::cell_pitch(desc->nx, desc->ny, desc->nz)};
    cudaError_t e = cudaGetDevice(&v->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&v->sms, cudaDevAttrMultiProcessorCount, v->device);
    if (cv.mode == 0) {
        // auto, within half of the device memory free now: the full view
        // when it fits (decoding narrow records on load slows the search
        // once the particles converge), else the narrow one, else none
        size_t free_b = 0, total_b = 0;
        if (e == cudaSuccess) e = cudaMemGetInfo(&free_b, &total_b);
        cv = pf::choose_view(desc->nx, desc->ny, desc->nz, (long long)(v->n_nodes * (ts + ws)), (long long)rec,
                             (long long)rec32, (long long)(free_b / 2));
    }
    if (cv.mode == 2 && !rec32) cv.mode = 1;
    if (cv.mode == -1 && vdt != desc->tsdf_dtype) e = cudaErrorMemoryAllocation;  // no room for the search view
    const bool view = cv.mode >= 1;
    const bool wide = cv.mode == 1 && rec32;
    if (e == cudaSuccess) e = pf::dev_malloc(&v->tsdf, v->n_nodes * ts);
    if (e == cudaSuccess) e = pf::dev_malloc(&v->weight, v->n_nodes * ws);
    auto alloc_view = [&]() {
        cudaError_t a = pf::dev_malloc(&v->cells, (size_t)cv.pitch.count * rec);
        if (a == cudaSuccess && wide) a = pf::dev_malloc(&v->cells32, (size_t)cv.pitch.count * rec32);
        return a;
    };
    if (e == cudaSuccess && view) {
        e = alloc_view();
        if (e == cudaErrorMemoryAllocation && cv.pitch.count > (long long)v->n_nodes) {  // with the node pitch, then
            cudaGetLastError();
            cudaFree(v->cells);
            v->cells = nullptr;
            cv.pitch = pf::node_pitch(desc->nx, desc->ny, desc->nz);
            e = alloc_view();
        }
    }
    v->pitch = cv.pitch;
    v->surf.wx = (desc->nx + 31) / 32;
    v->surf.wy = (desc->ny + 31) / 32;
    v->surf.wz = (desc->nz + 31) / 32;
    if (e == cudaSuccess) e = pf::dev_malloc(&v->surf.words, surface_bytes(v->surf));
    const size_t n_tiles = (size_t)v->tiles[0] * v->tiles[1] * v->tiles[2];
    if (e == cudaSuccess) e = pf::dev_malloc(&v->list.count, 2 * sizeof(int));
    if (e == cudaSuccess) e = pf::dev_malloc(&v->list.tile, n_tiles * sizeof(int));
    if (e == cudaSuccess) e = pf::dev_malloc(&v->list.base, n_tiles * sizeof(float4));
    if (e == cudaSuccess) e = pf::dev_malloc(&v->list.step, 9 * sizeof(float));
    if (e == cudaSuccess && n_tiles > PF_DEPTH_CULL_TILES)
        e = pf::dev_malloc(&v->list.depth_max, PF_DEPTH_BLOCKS * PF_DEPTH_BLOCKS * sizeof(float));
    if (e == cudaSuccess && view) e = pf::dev_malloc(&v->list.rows, n_tiles * sizeof(unsigned long long));
    if (e == cudaSuccess && view) e = pf::dev_malloc(&v->list.refresh_tile, n_tiles * sizeof(int));
    if (e == cudaSuccess && view) e = pf::dev_malloc(&v->list.refresh_rows, n_tiles * sizeof(unsigned long long));
    if (e == cudaSuccess && view)
        e = pf::dev_malloc(&v->tile_stamp, sizeof(int) * ((size_t)v->tiles[0] * v->tiles[1] * v->tiles[2] + 1));
    if (e == cudaSuccess && view)
        e = pf::zero_for(v->tile_stamp, sizeof(int) * ((size_t)v->tiles[0] * v->tiles[1] * v->tiles[2] + 1), &s);
    if (e != cudaSuccess) {
        cudaFree(v->tsdf);
        cudaFree(v->weight);
        cudaFree(v->cells);
        cudaFree(v->cells32);
        cudaFree(v->tile_stamp);
        cudaFree(v->surf.words);
        free_list(v->list);
        delete v;
        cudaGetLastError();
        return pf::cuda_status(e);
    }
    st = enqueue_reset(v, s);
    if (st != PF_OK) {
        pf_destroy_volume(v);
        return st;
    }
    *out = v;
    return PF_OK;
}

pf_status pf_destroy_volume(pf_volume* v)
{
    if (!v) return PF_OK;
    cudaDeviceSynchronize();
    pf::align_release(v);
    cudaFree(v->tsdf);
    cudaFree(v->weight);
    cudaFree(v->cells);
    cudaFree(v->cells32);
    cudaFree(v->tile_stamp);
    cudaFree(v->surf.words);
    free_list(v->list);
    pf_workspace& w = v->ws;
    cudaFree(w.points);
    cudaFree(w.block_counts);
    cudaFree(w.n_points);
    cudaFree(w.part_S);
    cudaFree(w.part_C);
    cudaFree(w.chunks);
    cudaFree(w.point_tile);
    cudaFree(w.kept);
    cudaFree(w.kept_count);
    cudaFree(w.order_scratch);
    cudaFree(w.chunk_counter);
    cudaFree(w.chunk_E);
    cudaFree(w.chunk_C);
    cudaFree(w.select);
    cudaFree(w.counter);
    cudaFree(w.state);
    cudaFree(w.pose_in);
    cudaFree(w.pose_out);
    cudaFree(w.stats);
    for (void* p : v->retired) cudaFree(p);
    delete v;
    return PF_OK;
}

static pf_status pf_reset_volume_impl(pf_volume* v, void* stream)
{
    if (!v) return PF_ERR_INVALID_ARG;
    return enqueue_reset(v, (cudaStream_t)stream);
}

static pf_status pf_set_fitness_variant_impl(pf_volume* v, int variant)
{
    if (!v || variant < 0 || variant > 11 || (variant & 3) == 3 && !v->cells) return PF_ERR_INVALID_ARG;
    // the plain baseline exists for float tsdf and float weights only
    if ((variant & 3) == 1 && (v->desc.tsdf_dtype != PF_F32 || v->desc.weight_u8)) return PF_ERR_INVALID_ARG;
    v->fitness_variant = variant;
    return PF_OK;
}

pf_status pf_volume_info(const pf_volume* v, unsigned long long* storage_bytes, int* cell_view)
{
    if (!v) return PF_ERR_INVALID_ARG;
    const size_t n = v->n_nodes, ts = pf_dtype_size(v->desc.tsdf_dtype), vs = pf_dtype_size(pf_view_dtype(v));
    const size_t n_tiles = (size_t)v->tiles[0] * v->tiles[1] * v->tiles[2];
    size_t b = n * ts + n * (v->desc.weight_u8 ? 1 : 4);
    if (v->cells) b += (size_t)v->pitch.count * 8 * vs + sizeof(int) * (n_tiles + 1);
    if (v->cells32) b += (size_t)v->pitch.count * 32;
    if (storage_bytes) *storage_bytes = b;
    if (cell_view) *cell_view = !v->cells ? -1 : (v->cells32 || pf_view_dtype(v) == PF_F32) ? 1 : 2;
    return PF_OK;
}

}  // extern "C"

namespace {

// Host-side conversion of one encoded value to and from the storage type.
void store_host(pf_dtype dt, float e, unsigned char* dst)
{
    switch (dt) {
    case PF_F16: { const __half h = pf_from_float<__half>(e); std::memcpy(dst, &h, 2); break; }
    case PF_BF16: { const __nv_bfloat16 h = pf_from_float<__nv_bfloat16>(e); std::memcpy(dst, &h, 2); break; }
    case PF_FP8E4M3: { const __nv_fp8_e4m3 h = pf_from_float<__nv_fp8_e4m3>(e); std::memcpy(dst, &h, 1); break; }
    default: std::memcpy(dst, &e, 4); break;
    }
}

float load_host(pf_dtype dt, const unsigned char* src)
{
    switch (dt) {
    case PF_F16: { __half h; std::memcpy(&h, src, 2); return pf_to_float(h); }
    case PF_BF16: { __nv_bfloat16 h; std::memcpy(&h, src, 2); return pf_to_float(h); }
    case PF_FP8E4M3: { __nv_fp8_e4m3 h; std::memcpy(&h, src, 1); return pf_to_float(h); }
    default: { float f; std::memcpy(&f, src, 4); return f; }
    }
}

}  // namespace

extern "C" {

static pf_status pf_volume_upload_impl(pf_volume* v, const float* tsdf_host, const float* weight_host)
{
    if (!v || !tsdf_host || !weight_host) return PF_ERR_INVALID_ARG;
    const size_t n = v->n_nodes;
    const pf_dtype dt = v->desc.tsdf_dtype;
    const size_t ts = pf_dtype_size(dt);
    std::vector<unsigned char> enc(n * ts);
    std::vector<uint8_t> w8(v->desc.weight_u8 ? n : 0);
    for (size_t i = 0; i < n; ++i) {
        const float w = weight_host[i];
        if (!(w >= 0.0f) || !std::isfinite(w) || w > (float)v->desc.max_weight) return PF_ERR_INVALID_ARG;
        if (w > 0.0f && !(std::fabs(tsdf_host[i]) <= 1.0f)) return PF_ERR_INVALID_ARG;
        if (v->desc.weight_u8 && w != std::floor(w)) return PF_ERR_INVALID_ARG;
        store_host(dt, pf_encode(tsdf_host[i], w), enc.data() + i * ts);
        if (v->desc.weight_u8) w8[i] = (uint8_t)w;
    }
    PF_CUDA(cudaDeviceSynchronize());
    PF_CUDA(cudaMemcpy(v->tsdf, enc.data(), n * ts, cudaMemcpyHostToDevice));
    if (v->desc.weight_u8) PF_CUDA(cudaMemcpy(v->weight, w8.data(), n, cudaMemcpyHostToDevice));
    else PF_CUDA(cudaMemcpy(v->weight, weight_host, n * 4, cudaMemcpyHostToDevice));
    pf_status st = enqueue_surface_scan(v, 0);
    if (st == PF_OK) st = enqueue_refresh(v, 0, 1);
    if (st != PF_OK) return st;
    PF_CUDA(cudaDeviceSynchronize());
    return PF_OK;
}

static pf_status pf_volume_download_impl(const pf_volume* v, float* tsdf_host, float* weight_host)
{
    if (!v || !tsdf_host || !weight_host) return PF_ERR_INVALID_ARG;
    const size_t n = v->n_nodes;
    const pf_dtype dt = v->desc.tsdf_dtype;
    const size_t ts = pf_dtype_size(dt);
    PF_CUDA(cudaDeviceSynchronize());
    if (dt == PF_F32) {
        PF_CUDA(cudaMemcpy(tsdf_host, v->tsdf, n * 4, cudaMemcpyDeviceToHost));
    } else {
        std::vector<unsigned char> raw(n * ts);
        PF_CUDA(cudaMemcpy(raw.data(), v->tsdf, n * ts, cudaMemcpyDeviceToHost));
        for (size_t i = 0; i < n; ++i) tsdf_host[i] = load_host(dt, raw.data() + i * ts);
    }
    if (v->desc.weight_u8) {
        std::vector<uint8_t> w8(n);
        PF_CUDA(cudaMemcpy(w8.data(), v->weight, n, cudaMemcpyDeviceToHost));
        for (size_t i = 0; i < n; ++i) weight_host[i] = (float)w8[i];
    } else {
        PF_CUDA(cudaMemcpy(weight_host, v->weight, n * 4, cudaMemcpyDeviceToHost));
    }
    for (size_t i = 0; i < n; ++i)
        tsdf_host[i] = weight_host[i] > 0.0f ? pf_decode(tsdf_host[i]) : 1.0f;
    return PF_OK;
}

}  // extern "C"

namespace {

pf_status integrate_impl(pf_volume* v, const float* depth_dev, const pf_intrinsics* intr, const double* P_host,
                         const double* P_dev, cudaStream_t s)
{
    if (!v || !depth_dev) return PF_ERR_INVALID_ARG;
    pf_status st = pf::check_intrinsics(intr);
    if (st != PF_OK) return st;
    const pf_volume_desc& d = v->desc;
    IntegArgs a;
    a.tsdf = v->tsdf;
    a.weight = v->weight;
    a.nx = d.nx;
    a.ny = d.ny;
    a.nz = d.nz;
    a.trunc = d.trunc;
    a.max_weight = (float)d.max_weight;
    a.cam = make_cam(intr);
    a.depth = depth_dev;
    a.pose_dev = P_dev;
    for (int q = 0; q < 12; ++q) a.pose[q] = P_host ? P_host[q] : 0.0;
    for (int q = 0; q < 3; ++q) a.origin[q] = d.origin[q];
    a.vs = d.voxel_size;
    // side planes through the camera centre: pixel range u in [-0.5, W - 0.5)
    const double lx0 = (-0.5 - intr->cx) / intr->fx, lx1 = (intr->width - 0.5 - intr->cx) / intr->fx;
    const double ly0 = (-0.5 - intr->cy) / intr->fy, ly1 = (intr->height - 0.5 - intr->cy) / intr->fy;
    const double pl[4][3] = {{1.0, 0.0, -lx0}, {-1.0, 0.0, lx1}, {0.0, 1.0, -ly0}, {0.0, -1.0, ly1}};
    for (int p = 0; p < 4; ++p) {
        double n = sqrt(pl[p][0] * pl[p][0] + pl[p][1] * pl[p][1] + pl[p][2] * pl[p][2]);
        for (int c = 0; c < 3; ++c) a.plane[p][c] = (float)(pl[p][c] / n);
    }
    a.zfar = d.trunc + intr->depth_max;
    const double vs = d.voxel_size;
    a.margin = (float)(0.01 * vs + 1e-3);
    // the fusion counter lives on the device (after the per-tile stamps), so
    // a captured and replayed launch sequence still marks each fusion apart
    const int n_tiles = v->tiles[0] * v->tiles[1] * v->tiles[2];
    a.tile_stamp = v->tile_stamp;
    a.stamp_dev = v->tile_stamp ? v->tile_stamp + n_tiles : nullptr;
    for (int q = 0; q < 3; ++q) a.tiles[q] = v->tiles[q];
    a.list = v->list;
    a.surf = v->surf;
    pf::timing_begin(pf::KC_INTEGRATE, s);
    int* stamp = v->tile_stamp ? v->tile_stamp + n_tiles : nullptr;
    if (v->list.depth_max)
        fusion_begin_kernel<<<PF_DEPTH_BLOCKS * PF_DEPTH_BLOCKS / BEGIN_WARPS, 32 * BEGIN_WARPS, 0, s>>>(v->list, stamp,
                                                                                                  depth_dev, a.cam);
    else
        fusion_begin_kernel<<<1, 32, 0, s>>>(v->list, stamp, nullptr, a.cam);
    fusion_tiles_kernel<<<(n_tiles + 255) / 256, 256, 0, s>>>(a);
    dispatch_storage<IntegrateLaunch>(v, list_ctas(v), a, s);
    pf::count_launch(3);
    pf::timing_end(pf::KC_INTEGRATE, s);
    PF_LAUNCHED();
    pf::timing_begin(pf::KC_REFRESH, s);
    st = enqueue_refresh(v, s, 0);
    pf::timing_end(pf::KC_REFRESH, s);
    return st;
}

__global__ void compose_kernel(const double* A, const double* B, double* out)
{
    const int t = threadIdx.x;
    if (t < 16) {
        const int r = t >> 2, c = t & 3;
        double acc = 0.0;
        for (int m = 0; m < 4; ++m) acc += A[4 * r + m] * B[4 * m + c];
        out[t] = acc;
    }
}

}  // namespace

extern "C" {

static pf_status pf_integrate_impl(pf_volume* v, const float* depth_dev, const pf_intrinsics* intr,
                                   const double P[16], void* stream)
{
    if (!P || !finite_pose(P)) return PF_ERR_INVALID_ARG;
    return integrate_impl(v, depth_dev, intr, P, nullptr, (cudaStream_t)stream);
}

static pf_status pf_integrate_async_impl(pf_volume* v, const float* depth_dev, const pf_intrinsics* intr,
                                         const double* P_dev, void* stream)
{
    if (!P_dev) return PF_ERR_INVALID_ARG;
    return integrate_impl(v, depth_dev, intr, nullptr, P_dev, (cudaStream_t)stream);
}

pf_status pf_pose_compose(const double* a_dev, const double* b_dev, double* out_dev, void* stream)
{
    if (!a_dev || !b_dev || !out_dev || out_dev == a_dev || out_dev == b_dev) return PF_ERR_INVALID_ARG;
    compose_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(a_dev, b_dev, out_dev);
    pf::count_launch();
    PF_LAUNCHED();
    return PF_OK;
}

}  // extern "C"

// Every entry point that takes a volume keeps its last failing status
// there (pf_volume_last_error).
extern "C" {

pf_status pf_volume_last_error(pf_volume* v, int clear)
{
    if (!v) return PF_ERR_INVALID_ARG;
    const pf_status s = v->last_status;
    if (clear) v->last_status = PF_OK;
    return s;
}

pf_status pf_reset_volume(pf_volume* v, void* stream)
{
    return pf::keep_status(v, pf_reset_volume_impl(v, stream));
}

pf_status pf_set_fitness_variant(pf_volume* v, int variant)
{
    return pf::keep_status(v, pf_set_fitness_variant_impl(v, variant));
}

pf_status pf_volume_upload(pf_volume* v, const float* tsdf_host, const float* weight_host)
{
    return pf::keep_status(v, pf_volume_upload_impl(v, tsdf_host, weight_host));
}

pf_status pf_volume_download(const pf_volume* v, float* tsdf_host, float* weight_host)
{
    return pf::keep_status(v, pf_volume_download_impl(v, tsdf_host, weight_host));
}

pf_status pf_integrate(pf_volume* v, const float* depth_dev, const pf_intrinsics* intr, const double P[16],
                       void* stream)
{
    return pf::keep_status(v, pf_integrate_impl(v, depth_dev, intr, P, stream));
}

pf_status pf_integrate_async(pf_volume* v, const float* depth_dev, const pf_intrinsics* intr, const double* P_dev,
                             void* stream)
{
    return pf::keep_status(v, pf_integrate_async_impl(v, depth_dev, intr, P_dev, stream));
}

}  // extern "C"
