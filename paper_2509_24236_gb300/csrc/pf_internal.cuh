// Internal declarations shared by the translation units of libprofusion.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cmath>
#include <vector>

#include "../../include/profusion.h"
#include "cellpitch.h"
#include "growbuf.h"

// --------------------------------------------------------------------------
// TSDF value encoding in the f32 tsdf array.
//
// A node is usable by the fitness when it is observed and within the
// truncation band (|tsdf| < 1).  Storing the other nodes as non-finite
// values makes that test fall out of the interpolation itself: a linear
// interpolation with a NaN or infinite end point is never finite, so the
// trilinear value of a cell is finite exactly when all eight nodes are
// usable.  Encoding:
//   unobserved (weight 0)        -> quiet NaN
//   observed, tsdf == +1 / -1    -> +inf / -inf
//   observed, |tsdf| < 1         -> the value
// --------------------------------------------------------------------------
#define PF_UNOBSERVED __int_as_float(0x7fc00000)

__host__ __device__ inline float pf_encode(float t, float w)
{
#ifdef __CUDA_ARCH__
    if (!(w > 0.0f)) return __int_as_float(0x7fc00000);
    if (t >= 1.0f) return __int_as_float(0x7f800000);
    if (t <= -1.0f) return __int_as_float(0xff800000);
    return t;
#else
    if (!(w > 0.0f)) return NAN;
    if (t >= 1.0f) return INFINITY;
    if (t <= -1.0f) return -INFINITY;
    return t;
#endif
}

// Value of an observed node (weight > 0): infinities stand for +-1.
__host__ __device__ inline float pf_decode(float e)
{
    return isinf(e) ? copysignf(1.0f, e) : e;
}

// --------------------------------------------------------------------------
// Storage types.  The tsdf (and the cell view) are stored as float, half,
// bfloat16 or scaled e4m3 -- the encoding above survives the conversion
// (NaN and infinities are kept; e4m3 codes them as below) and a value that
// rounds to +-1 is stored as +-infinity, so a finite stored value always
// lies inside the band -- and the weight as float or uint8.  All arithmetic
// is float.
// --------------------------------------------------------------------------
__host__ __device__ inline float pf_to_float(float v) { return v; }
__host__ __device__ inline float pf_to_float(__half v) { return __half2float(v); }
__host__ __device__ inline float pf_to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__host__ __device__ inline float pf_to_float(uint8_t v) { return (float)v; }

// 8-bit storage (PF_FP8E4M3): the value scaled by 2^8 in e4m3 (a value in
// (-1, 1) keeps 3 mantissa bits; the scale lifts the values near the surface
// out of the e4m3 subnormals).  e4m3 has no infinities: the largest finite
// code, +-448, stands for the outside-the-band +-1 and the NaN code for
// unobserved.  Scaled values stay below 256 in magnitude, so 448 never
// collides with a value.
constexpr float PF_FP8_SCALE = 256.0f;
constexpr unsigned char PF_FP8_NAN = 0x7f, PF_FP8_POS = 0x7e, PF_FP8_NEG = 0xfe;
__host__ __device__ inline float pf_to_float(__nv_fp8_e4m3 v)
{
    const __half h(__nv_cvt_fp8_to_halfraw(v.__x, __NV_E4M3));
    const float f = __half2float(h);
    if (f != f) return f;
    return fabsf(f) >= 448.0f ? copysignf(INFINITY, f) : f * (1.0f / PF_FP8_SCALE);
}

template <typename T> __host__ __device__ inline T pf_from_float(float v);
template <> __host__ __device__ inline float pf_from_float<float>(float v) { return v; }
template <> __host__ __device__ inline __half pf_from_float<__half>(float v)
{
    const float r = __half2float(__float2half_rn(v));
    return __float2half_rn(r >= 1.0f ? INFINITY : (r <= -1.0f ? -INFINITY : v));
}
template <> __host__ __device__ inline __nv_bfloat16 pf_from_float<__nv_bfloat16>(float v)
{
    const float r = __bfloat162float(__float2bfloat16_rn(v));
    return __float2bfloat16_rn(r >= 1.0f ? INFINITY : (r <= -1.0f ? -INFINITY : v));
}
template <> __host__ __device__ inline uint8_t pf_from_float<uint8_t>(float v) { return (uint8_t)v; }
template <> __host__ __device__ inline __nv_fp8_e4m3 pf_from_float<__nv_fp8_e4m3>(float v)
{
    __nv_fp8_e4m3 r;
    if (v != v) {
        r.__x = PF_FP8_NAN;
    } else if (v >= 1.0f || v <= -1.0f) {
        r.__x = v > 0.0f ? PF_FP8_POS : PF_FP8_NEG;
    } else {
        r.__x = __nv_cvt_float_to_fp8(v * PF_FP8_SCALE, __NV_SATFINITE, __NV_E4M3);
        const float back = __half2float(__half(__nv_cvt_fp8_to_halfraw(r.__x, __NV_E4M3)));
        if (back >= PF_FP8_SCALE) r.__x = PF_FP8_POS;       // rounds to +-1: outside the band
        else if (back <= -PF_FP8_SCALE) r.__x = PF_FP8_NEG;
    }
    return r;
}

inline size_t pf_dtype_size(pf_dtype t) { return t == PF_F32 ? 4 : t == PF_FP8E4M3 ? 1 : 2; }

// --------------------------------------------------------------------------
// Volume and workspace
// --------------------------------------------------------------------------
struct pf_workspace {
    int pix_cap = 0;        // max pixels per frame
    int k_cap = 0;          // max particles
    int part_cap = 0;       // partial slots (tiles x particles)
    float4* points = nullptr;        // pix_cap
    int* block_counts = nullptr;     // back-projection blocks
    int* n_points = nullptr;         // 1
    float* part_S = nullptr;         // part_cap
    int* part_C = nullptr;           // part_cap
    unsigned int* counter = nullptr; // last-block tickets (zeroed, reset by the last block)
    void* chunks = nullptr;          // the particle chunks of a search iteration, see track.cu
    int chunk_cap = 0;               // chunks it holds
    unsigned int* chunk_counter = nullptr;  // per chunk: tickets of its point tiles (zeroed, reset by the last)
    float* chunk_E = nullptr;        // per particle: fitness of the search iteration (chunk_cap x 32)
    int* chunk_C = nullptr;          // per particle: valid points
    void* select = nullptr;          // partial results of the selection, see track.cu
    // decimated point sets in a locality order (see track.cu): each point's
    // tile, the reordered kept points of up to three strides, counters
    int* point_tile = nullptr;       // pix_cap
    float4* kept = nullptr;          // 2 x pix_cap
    int* kept_count = nullptr;       // 3: kept points of each stride
    int* order_scratch = nullptr;    // order_cap: per (block of tiles, tile row) counts and first indices, offsets
    int order_cap = 0;
    double* state = nullptr;         // search state, see track.cu
    double* pose_in = nullptr;       // 16 (sync entry point)
    double* pose_out = nullptr;      // 16
    pf_track_stats* stats = nullptr; // 1
};

// Fusion works on tiles of 32 x 8 x 8 nodes; the cell view is refreshed
// tile by tile after fusion.
constexpr int PF_TX = 32, PF_TY = 8, PF_TZ = 8;
constexpr int PF_DEPTH_BLOCKS = 64;  // per axis, whatever the image's size
// Grids of more fusion tiles than this drop tiles behind the image's depths;
// reducing the image to its blocks' depths and looking them up cost 3 to 15 us a
// fusion, the tiles that it drops less than that up to 512^3 (65 536 tiles).
// A 640x480 frame into float nodes, with the depth cull -> without, and a
// 1920x1080 one: 128^3 25 -> 19, 29 -> 19 us; 256^3 31 -> 23, 35 -> 22; 512^3
// 62 -> 53, 58 -> 46; 768^3 (221 184 tiles) 114 -> 129, 99 -> 102.
constexpr int PF_DEPTH_CULL_TILES = 100000;

// Per-fusion tile lists (device memory, one slot per tile): the tiles that
// survive the culls with the camera-frame position of their first node, which
// of each tile's rows of nodes changed, and the tiles whose cell-view records
// must be rewritten with the rows of records concerned.  A tile's rows are
// bits of a 64-bit word: bit 8 j + k is the row of 32 nodes at (j, k).
struct FusionList {
    int* count = nullptr;         // [0] fused tiles, [1] tiles to refresh
    int* tile = nullptr;          // fused tile indices
    float4* base = nullptr;       // their first node in the camera frame: x, y, z hi, z lo
    float* step = nullptr;        // 9: camera-frame step per node index along i, j, k
    float* depth_max = nullptr;   // largest usable depth of each of PF_DEPTH_BLOCKS^2 blocks of the image (null: no depth cull)
    unsigned long long* rows = nullptr;  // per tile: changed rows (valid where the tile's stamp is the last fusion's)
    int* refresh_tile = nullptr;  // tiles to refresh
    unsigned long long* refresh_rows = nullptr;  // and their rows
};

// Where the ray cast can meet the surface: one bit per brick of 8^3 cells,
// set when some cell of the brick has a corner whose value was ever fused or
// uploaded as zero or negative (never cleared but by a reset or an upload, so
// a set bit may be stale; a clear one is certain).  A 64-bit word holds 4^3
// bricks (32^3 cells): 32 KB at 512^3, small enough to stay in L1.
struct SurfaceMap {
    unsigned long long* words = nullptr;
    int wx = 0, wy = 0, wz = 0;  // words per axis: ceil(n / 32)
};

struct pf_volume {
    pf_volume_desc desc;
    int device = 0;
    int sms = 0;               // of the device (calls of other volumes run in other threads: no shared cache)
    size_t n_nodes = 0;
    void* tsdf = nullptr;      // encoded, see above; float, half or bfloat16 (desc.tsdf_dtype)
    void* weight = nullptr;    // float, or uint8 when desc.weight_u8
    void* cells = nullptr;     // cell view: a record of 8 values per cell, pitched as `pitch` says
    float* cells32 = nullptr;  // 16-/8-bit grids, full view: the same records as floats (x-differences formed)
    int* tile_stamp = nullptr; // per fusion tile: stamp of the last fusion that reached it
    int tiles[3] = {0, 0, 0};
    pf::CellPitch pitch = {0, 0, 0};  // of the records in cells and cells32
    int fitness_variant = 0;
    pf_status last_status = PF_OK;  // last failing status of a call on this volume
    FusionList list;
    SurfaceMap surf;
    pf_workspace ws;
    std::vector<void*> retired;  // outgrown scratch, kept for the graphs and tables that hold it
};

// Storage type of the cell view's records: the node array's, or the search
// view type of a float grid (pf_volume_desc.search_dtype).
inline pf_dtype pf_view_dtype(const pf_volume* v)
{
    return v->desc.search_dtype != PF_F32 ? v->desc.search_dtype : v->desc.tsdf_dtype;
}

// Type the fitness kernel is instantiated on for a layout: the cell view's
// (layout 3) or the node array's (layouts 1 and 2).
inline pf_dtype pf_fitness_dtype(const pf_volume* v, int layout)
{
    return layout == 3 ? pf_view_dtype(v) : v->desc.tsdf_dtype;
}

// --------------------------------------------------------------------------
// Host helpers
// --------------------------------------------------------------------------
namespace pf {

extern std::atomic<unsigned long long> g_launches;
extern std::atomic<unsigned long long> g_allocs;

inline void count_launch(unsigned n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }

// Every device allocation the library makes goes through these two, so that
// pf_alloc_count can tell a caller whether a call allocated.
template <typename T>
inline cudaError_t dev_malloc(T** p, size_t bytes)
{
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    return cudaMalloc(reinterpret_cast<void**>(p), bytes);
}

template <typename T>
inline cudaError_t dev_malloc_async(T** p, size_t bytes, cudaStream_t s)
{
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    return cudaMallocAsync(reinterpret_cast<void**>(p), bytes, s);
}

// Zeroes device memory before it returns, on a stream of its own.  A fill on
// the legacy default stream is ordered neither before work on a caller's
// non-blocking stream nor before the host's next step; one on the caller's
// stream, which may be capturing, would only be recorded, and a call before the
// graph's first launch, or after the graph is dropped, would find the memory as
// it came.
inline cudaError_t zero_now(void* p, size_t bytes)
{
    cudaStream_t z = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&z, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(p, 0, bytes, z);
    const cudaError_t e2 = cudaStreamSynchronize(z);
    cudaStreamDestroy(z);
    return e != cudaSuccess ? e : e2;
}

// Zeroes device memory for calls on the caller's stream (null: any): in that
// stream's order when it is not capturing (the wait of zero_now, with a stream
// made for it, is 20 to 40 us), else at once.
inline cudaError_t zero_for(void* p, size_t bytes, const cudaStream_t* s)
{
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusActive;
    if (s && cudaStreamIsCapturing(*s, &c) != cudaSuccess) {  // the legacy stream beside a capture
        cudaGetLastError();
        c = cudaStreamCaptureStatusActive;
    }
    return s && c == cudaStreamCaptureStatusNone ? cudaMemsetAsync(p, 0, bytes, *s) : zero_now(p, bytes);
}

// Replaces scratch buffers of a volume by larger ones (see growbuf.h), for a
// call on the given stream (null: for any).
inline cudaError_t grow_scratch(pf_volume* v, std::initializer_list<Grow> set, const cudaStream_t* s)
{
    const cudaError_t e = grow_all(
        v->retired, set,
        [s](void** p, size_t bytes, bool zero) {
            cudaError_t a = dev_malloc(p, bytes);
            if (a == cudaSuccess && zero) a = zero_for(*p, bytes, s);
            if (a != cudaSuccess) {
                cudaFree(*p);
                *p = nullptr;
            }
            return a;
        },
        [](void* p) { cudaFree(p); });
    if (e != cudaSuccess) cudaGetLastError();  // reported here, not by the next launch
    return e;
}

template <typename T>
inline Grow grow(T** p, size_t count, bool zero = false)
{
    return {p, count * sizeof(T), zero};
}

enum KernelClass { KC_FITNESS = 0, KC_FITNESS1, KC_INTEGRATE, KC_REFRESH, KC_BACKPROJECT, KC_RAYCAST, KC_COUNT };

// Event bracketing of launches (no-ops unless timing is enabled).
void timing_begin(KernelClass kc, cudaStream_t s);
void timing_end(KernelClass kc, cudaStream_t s);

pf_status check_intrinsics(const pf_intrinsics* intr);
pf_status workspace_reserve(pf_volume* vol, int max_pixels, int k_max, const cudaStream_t* s);

// Records a failing status (anything but PF_OK and PF_ERR_TRACK_LOST, which
// describes the frame rather than the call) in the volume it concerns.
inline pf_status keep_status(const pf_volume* v, pf_status s)
{
    if (v && s != PF_OK && s != PF_ERR_TRACK_LOST) const_cast<pf_volume*>(v)->last_status = s;
    return s;
}

inline pf_status cuda_status(cudaError_t e)
{
    if (e == cudaSuccess) return PF_OK;
    if (e == cudaErrorMemoryAllocation) return PF_ERR_OOM;
    return PF_ERR_CUDA;
}

}  // namespace pf

#define PF_CUDA(call)                                   \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return pf::cuda_status(e_); \
    } while (0)

#define PF_LAUNCHED()                                   \
    do {                                                \
        cudaError_t e_ = cudaGetLastError();            \
        if (e_ != cudaSuccess) return pf::cuda_status(e_); \
    } while (0)

// Camera parameters in the form the kernels use.
struct CamK {
    int width, height;
    float fx, fy, cx, cy, dmin, dmax;
};

inline CamK make_cam(const pf_intrinsics* in)
{
    CamK c;
    c.width = in->width;
    c.height = in->height;
    c.fx = in->fx;
    c.fy = in->fy;
    c.cx = in->cx;
    c.cy = in->cy;
    c.dmin = in->depth_min;
    c.dmax = in->depth_max;
    return c;
}

__device__ inline bool pf_depth_usable(float z, float dmin, float dmax)
{
    return isfinite(z) && z >= dmin && z <= dmax;
}

// Marks the bricks that hold a cell with one of these nodes as a corner: the
// warp's lane l stands for node (i0 + l, j, k0 ... k0 + 7), i0 a multiple of
// 32 and k0 of 8; bit l of any is set when one of its eight nodes is zero or
// negative, bit l of first when the one at k0 is.  Called by a whole warp.
__device__ inline void pf_mark_surface(const SurfaceMap& s, unsigned any, unsigned first, int i0, int j, int k0)
{
    if (any == 0u) return;
    // lanes 0..19: bricks i0/8 + q (q = -1..3) x (j/8 or the one below) x (k0/8 or the one below)
    const int lane = threadIdx.x & 31;
    const int q = lane % 5 - 1, below_y = (lane / 5) & 1, below_z = lane / 10;
    if (lane >= 20 || (below_y && (j & 7) != 0)) return;
    const unsigned m = below_z ? first : any;
    // a brick's cells reach the first node of the next brick
    const unsigned nodes = q < 0 ? m & 1u : (m >> (8 * q)) & 0x1ffu;
    const int bx = (i0 >> 3) + q, by = (j >> 3) - below_y, bz = (k0 >> 3) - below_z;
    if (nodes == 0u || bx < 0 || by < 0 || bz < 0) return;
    unsigned long long* w = s.words + (bx >> 2) + (size_t)s.wx * ((by >> 2) + (size_t)s.wy * (bz >> 2));
    const unsigned long long bit = 1ull << ((bx & 3) | ((by & 3) << 2) | ((bz & 3) << 4));
    if ((__ldcg(w) & bit) == 0ull) atomicOr(w, bit);
}
