// Alignment loss, its derivatives and the Gauss-Newton polish.
//
// The residual of a point x under pose T is the TSDF of Sec. III-B at the
// transformed point, r = tsdf(T x) (normalised by tau, trilinear, defined
// when the point falls in a valid cell -- all eight nodes observed and
// inside the band).  The loss of a frame is L = sum r^2.  A pose is
// perturbed on the left, q = Exp(omega) (R x + t) + v with xi = (omega, v),
// so dq/dv = I and dq/domega = -[q - v]x J_l(omega) (J_l the left Jacobian
// of SO(3)); with grad r the gradient of the trilinear interpolant in
// metres,
//     dL/dv = sum 2 r grad r,      dL/domega = J_l^T sum 2 r ((q - v) x grad r),
// and the derivative with respect to the stored value of node n is
// dL/dV_n = sum 2 r w_n(q) over the samples whose cell has node n.
//
// GPU design
//   * align_kernel: grid = (point tiles) x frames.  Per-sample arithmetic is
//     float: each frame's pose is prepared once in FP64 (perturbation,
//     rotation in grid units split into a float pair, translation split into
//     an integer cell and a fraction), and each point's grid coordinate is
//     formed with error-free products and sums, so the cell and fractions
//     carry no rounding at the scale of the grid coordinate.  Node values are
//     read in their storage type.  Per-thread float sums, then FP64 from the
//     block sums on: per-block sums in a fixed order into per-tile partials;
//     align_finish reduces the tiles of each frame in a fixed order and
//     applies J_l^T.  dL/dV goes to an int64 fixed-point
//     accumulator (2^-40 units) by integer atomics: integer addition is
//     associative, so the result does not depend on the order of arrival
//     and the output is bit-reproducible.
//   * Polish: a damped Gauss-Newton (Levenberg-Marquardt) with its state in
//     device memory.  gn_kernel accumulates H = sum J^T J (upper triangle),
//     b = sum J^T r, sum r^2 and the count for the state's candidate pose
//     (float per thread, FP64 across threads and tiles); the last block of
//     the launch accepts the candidate if it lowers the mean squared residual
//     (lambda /= 10) or drops it (lambda *= 10), solves
//     (H + lambda diag H) d = -b and forms the next candidate
//     [Exp(d_omega) | d_v] T.  No host round trip: a polish is a fixed launch
//     sequence.
#include <algorithm>
#include <climits>
#include <mutex>
#include <unordered_map>

#include "pf_internal.cuh"

namespace {

constexpr int AL_THREADS = 256;
constexpr int AL_TILES = 296;          // most point tiles per frame (2 per SM)
constexpr int AL_BLOCKS = 2432;        // target blocks per launch (2 waves of 8 per SM)
constexpr int RED_THREADS = 256;       // tile reductions
// dL/dV accumulates in int64 units of 2^-40 (fix40 / fixed40_to_float)
constexpr float kRound = 12582912.0f;  // 1.5 * 2^23: adding it rounds |v| < 2^22 to an integer
constexpr int kRoundBits = 0x4B400000;  // its bit pattern
constexpr int GN_VALS = 29;            // 21 (upper H) + 6 (b) + loss + count
constexpr int GN_CLASSES = RED_THREADS / GN_VALS;  // 8 classes of tiles, summed apart

struct AlignScratch {
    double* part = nullptr;       // align partials: frames x tiles x 8 (tiles <= AL_TILES)
    size_t part_cap = 0;          // doubles
    long long* acc = nullptr;     // n_nodes fixed-point dL/dV
    bool acc_zero = false;        // and it is zero whenever no call is in flight
    double* gn_part = nullptr;    // (AL_TILES + GN_CLASSES) x GN_VALS
    double* gn_state = nullptr;   // see GnState
    void* frame_pose = nullptr;   // frames x FramePose (the poses prepared once per frame)
    int frame_cap = 0;            // frames
    void* gn_pose = nullptr;      // one PoseF: the polish's candidate, prepared once per step
};

std::mutex g_mu;
std::unordered_map<const pf_volume*, AlignScratch> g_scratch;

struct GnState {
    double T[12];      // current (accepted) pose
    double Tc[12];     // candidate pose
    double H[36], b[6];
    double obj;        // mean squared residual at T
    double lambda;
    int have_cand;     // a candidate is pending evaluation
    int accepted;
    int step;
    // of the running launch: finished blocks of each class, finished classes
    unsigned class_ticket[GN_CLASSES], ticket;
};

// ---------------------------------------------------------------------------
// FP64 helpers
// ---------------------------------------------------------------------------
// left Jacobian of SO(3): I + (1 - cos th)/th^2 [w]x + (th - sin th)/th^3 [w]x^2
__device__ inline void so3_left_jacobian(const double w[3], double J[9])
{
    const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    const double th = sqrt(th2);
    double a, b;
    if (th < 1e-6) {
        a = 0.5 - th2 / 24.0;
        b = 1.0 / 6.0 - th2 / 120.0;
    } else {
        a = (1.0 - cos(th)) / th2;
        b = (th - sin(th)) / (th2 * th);
    }
    const double K[9] = {0.0, -w[2], w[1], w[2], 0.0, -w[0], -w[1], w[0], 0.0};
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            double kk = 0.0;
            for (int m = 0; m < 3; ++m) kk += K[3 * r + m] * K[3 * m + c];
            J[3 * r + c] = (r == c ? 1.0 : 0.0) + a * K[3 * r + c] + b * kk;
        }
}

struct GridInfo {
    int nx, ny, nz;
    double inv_vs, org[3];
};

// A pose prepared for float sampling: the rotation in grid units as a float
// pair (hi + lo), the translation in grid units as an integer cell o and a
// float fraction b, and the pose in metres as floats (for q itself).
struct PoseF {
    float Ahi[9], Alo[9];
    int o[3];
    float b[3];
    float R[9], t[3];
    int ok;  // the camera lies within 2^21 voxels of the grid
};

// The pose preparations by the first two warps of a block.  Each is a chain of
// dependent FP64 operations, a hundred cycles and more apiece, which is
// microseconds in one thread; every element of a matrix is formed by a thread
// of its own with the expression one thread would use for it, and the sine and
// the cosine by the two warps at a time, so the results are the same bits.
__device__ __forceinline__ void pair_sync() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

// T (shared) to a PoseF.
__device__ inline void pair_make_posef(const double* T, const GridInfo& g, PoseF* out, int* sh_ok)
{
    const int tid = threadIdx.x;
    if (tid == 0) *sh_ok = 1;
    pair_sync();
    if (tid < 9) {
        const int r = tid / 3, c = tid % 3;
        const double A = T[4 * r + c] * g.inv_vs;
        const float hi = (float)A;
        out->Ahi[tid] = hi;
        out->Alo[tid] = (float)(A - (double)hi);
        out->R[tid] = (float)T[4 * r + c];
    } else if (tid >= 32 && tid < 35) {
        const int r = tid - 32;
        const double tg = (T[4 * r + 3] - g.org[r]) * g.inv_vs;
        const bool ok = fabs(tg) < 2097152.0;
        if (!ok) *sh_ok = 0;
        const double o = ok ? floor(tg) : 0.0;
        out->o[r] = (int)o;
        out->b[r] = (float)(tg - o);
        out->t[r] = (float)T[4 * r + 3];
    }
    pair_sync();
    if (tid == 0) out->ok = *sh_ok;
}

// [Exp(omega) R | Exp(omega) t + v] (shared out, 12) from a 3x4 pose P, Exp
// Rodrigues' formula.  xi: 6 doubles; sh: 16 doubles of shared memory.
__device__ inline void pair_perturb(const double* P, const double* xi, double* out, double* sh)
{
    const int tid = threadIdx.x;
    const double th2 = xi[0] * xi[0] + xi[1] * xi[1] + xi[2] * xi[2];
    if (tid == 0 || tid == 32) {
        const double th = sqrt(th2);
        if (th < 1e-8)
            sh[tid >> 5] = tid == 0 ? 1.0 - th2 / 6.0 : 0.5 - th2 / 24.0;
        else if (tid == 0)
            sh[0] = sin(th) / th;
        else
            sh[1] = (1.0 - cos(th)) / th2;
    }
    pair_sync();
    if (tid < 9) {
        const int r = tid / 3, c = tid % 3;
        const double K[9] = {0.0, -xi[2], xi[1], xi[2], 0.0, -xi[0], -xi[1], xi[0], 0.0};
        double kr[3], kc[3], krc = 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) {  // (constant indices: the array stays in registers)
            if (q / 3 == r) kr[q % 3] = K[q];
            if (q % 3 == c) kc[q / 3] = K[q];
            if (q == tid) krc = K[q];
        }
        double kk = 0.0;
        for (int m = 0; m < 3; ++m) kk += kr[m] * kc[m];
        sh[4 + tid] = (r == c ? 1.0 : 0.0) + sh[0] * krc + sh[1] * kk;
    }
    pair_sync();
    if (tid < 12) {
        const int r = tid / 4, c = tid % 4;
        double acc = 0.0;
        for (int m = 0; m < 3; ++m) acc += sh[4 + 3 * r + m] * P[4 * m + c];
        out[tid] = c == 3 ? acc + xi[3 + r] : acc;
    }
    pair_sync();
}

// One frame of pf_align_loss, prepared once per frame (FP64 work that every
// block of the frame would otherwise repeat): the perturbed pose for
// sampling, the translation part v of the perturbation (q - v enters the
// rotation gradient) and the weight 2 W of the node gradient.
struct FramePose {
    PoseF P;
    float V[3];
    float w2;
};

// Copy a record of 4-byte words from global to shared memory with the
// whole block (call from every thread; a barrier follows).
template <typename T>
__device__ inline void block_copy_words(const T* src, T* dst)
{
    static_assert(sizeof(T) % 4 == 0, "4-byte words");
    const int* s = reinterpret_cast<const int*>(src);
    int* d = reinterpret_cast<int*>(dst);
    for (int i = threadIdx.x; i < (int)(sizeof(T) / 4); i += blockDim.x) d[i] = s[i];
    __syncthreads();
}

// y = (hi + lo) . x as an integer part and a float fraction, to ~1e-12 of
// |y|: the products are split exactly (p = hi*x rounded, fma(hi, x, -p) its
// error), the three-term sum carries its rounding errors (two-sum), and the
// lo part is added to the error term.  Explicit round-to-nearest intrinsics
// keep the compiler from fusing any step.  False when |y| >= 2^22.
__device__ inline bool row_split(const float* hi, const float* lo, float x, float y, float z, int& yi, float& yf)
{
    const float p0 = __fmul_rn(hi[0], x), p1 = __fmul_rn(hi[1], y), p2 = __fmul_rn(hi[2], z);
    float err = __fadd_rn(__fadd_rn(fmaf(hi[0], x, -p0), fmaf(hi[1], y, -p1)), fmaf(hi[2], z, -p2));
    const float s1 = __fadd_rn(p0, p1);
    float bb = __fsub_rn(s1, p0);
    err = __fadd_rn(err, __fadd_rn(__fsub_rn(p0, __fsub_rn(s1, bb)), __fsub_rn(p1, bb)));
    const float s2 = __fadd_rn(s1, p2);
    bb = __fsub_rn(s2, s1);
    err = __fadd_rn(err, __fadd_rn(__fsub_rn(s1, __fsub_rn(s2, bb)), __fsub_rn(p2, bb)));
    err = fmaf(lo[0], x, fmaf(lo[1], y, fmaf(lo[2], z, err)));
    if (!(fabsf(s2) < 4194304.0f)) return false;
    // nearest integer (ties to even) by adding 1.5 * 2^23, whose unit in the
    // last place is 1; its bits give the integer without a conversion
    const float m = __fadd_rn(s2, kRound);
    const float r = __fsub_rn(m, kRound);
    yi = __float_as_int(m) - kRoundBits;
    yf = __fadd_rn(__fsub_rn(s2, r), err);
    return true;
}

// What a sample reads: the node array, or (records not null) the cell view's
// 32-byte float records, whose first differences are the ones formed here, so
// both give the same bits.
template <typename TS>
struct Field {
    const TS* tsdf;
    const float* records;
    int row, plane;  // of the records
};

// Trilinear value t, its gradient in grid units, the cell (linear index of
// its lower corner) and the fractions of point x under pose P; false when
// the sample lies in no valid cell (outside the grid, or a node that is
// unobserved or outside the band -- non-finite in the encoded storage).
// One 256-bit load of a record in place of eight of nodes, or the eight
// before any test of them, so that they wait together: a test after each was
// eight waits in a row (4.9 M points' loss 98 -> 63 us, with all derivatives
// 209 -> 173 us, the scatter's integer reductions being the rest).
template <typename TS, bool RECORDS>
__device__ __forceinline__ bool sample_f(const Field<TS>& F, const GridInfo& g, const PoseF& P, float x, float y,
                                         float z, float& t, float dg[3], int& base, float f[3])
{
    if (!P.ok || !isfinite(x) || !isfinite(y) || !isfinite(z)) return false;
    const int n[3] = {g.nx, g.ny, g.nz};
    int ci[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        int yi;
        float yf;
        if (!row_split(P.Ahi + 3 * r, P.Alo + 3 * r, x, y, z, yi, yf)) return false;
        const float u = __fadd_rn(yf, P.b[r]);
        // floor(u) the same way with round-down (|u| is a few units)
        const float m = __fadd_rd(u, kRound);
        const float fl = __fsub_rn(m, kRound);
        // (|o| < 2^21, |yi| <= 2^22: no overflow)
        ci[r] = P.o[r] + yi + (__float_as_int(m) - kRoundBits);
        f[r] = __fsub_rn(u, fl);
        if ((unsigned)ci[r] > (unsigned)(n[r] - 2)) return false;
    }
    const int nx = g.nx, nxy = g.nx * g.ny;
    base = ci[0] + nx * ci[1] + nxy * ci[2];
    float v0, v2, v4, v6, dx00, dx10, dx01, dx11;
    if (RECORDS) {
        const float* p = F.records + 8 * (size_t)(unsigned)(ci[0] + F.row * ci[1] + F.plane * ci[2]);
        // (volatile: not to be moved above the range test)
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(v0), "=f"(dx00), "=f"(v2), "=f"(dx10), "=f"(v4), "=f"(dx01), "=f"(v6), "=f"(dx11) : "l"(p));
    } else {
        const TS* p = F.tsdf + base;
        const TS e[8] = {p[0], p[1], p[nx], p[nx + 1], p[nxy], p[nxy + 1], p[nxy + nx], p[nxy + nx + 1]};
        v0 = pf_to_float(e[0]);
        v2 = pf_to_float(e[2]);
        v4 = pf_to_float(e[4]);
        v6 = pf_to_float(e[6]);
        dx00 = pf_to_float(e[1]) - v0;
        dx10 = pf_to_float(e[3]) - v2;
        dx01 = pf_to_float(e[5]) - v4;
        dx11 = pf_to_float(e[7]) - v6;
    }
    // a difference is finite exactly when both its nodes are
    if (!(isfinite(dx00) && isfinite(dx10) && isfinite(dx01) && isfinite(dx11))) return false;
    const float x00 = fmaf(f[0], dx00, v0);
    const float x10 = fmaf(f[0], dx10, v2);
    const float x01 = fmaf(f[0], dx01, v4);
    const float x11 = fmaf(f[0], dx11, v6);
    const float y0 = fmaf(f[1], x10 - x00, x00);
    const float y1 = fmaf(f[1], x11 - x01, x01);
    t = fmaf(f[2], y1 - y0, y0);
    const float dy0 = fmaf(f[1], dx10 - dx00, dx00), dy1 = fmaf(f[1], dx11 - dx01, dx01);
    dg[0] = fmaf(f[2], dy1 - dy0, dy0);
    dg[1] = fmaf(f[2], (x11 - x01) - (x10 - x00), x10 - x00);
    dg[2] = y1 - y0;
    return true;
}

__device__ inline void transform_f(const PoseF& P, float x, float y, float z, float q[3])
{
#pragma unroll
    for (int r = 0; r < 3; ++r) q[r] = fmaf(P.R[3 * r], x, fmaf(P.R[3 * r + 1], y, fmaf(P.R[3 * r + 2], z, P.t[r])));
}

// round(x * 2^40) to nearest (ties to even) as an int64, from the bits of
// the float: exactly the value an FP64 multiply by 2^40 and conversion would
// give (both are exact up to that one rounding), without the FP64 pipe.
// Magnitudes of 2^23 and more saturate.
__device__ __forceinline__ long long fix40(float x)
{
    const unsigned b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xffu);
    if (e == 0) return 0;  // zero or subnormal: below 2^-126, rounds to 0
    const int sh = e - 110;  // x * 2^40 = m * 2^(e - 127 - 23 + 40)
    long long r;
    if (sh > 39) {  // |x| >= 2^23: beyond int64
        r = LLONG_MAX;
    } else if (sh >= 0) {
        r = (long long)(((unsigned long long)((b & 0x7fffffu) | 0x800000u)) << sh);
    } else if (sh > -26) {
        const unsigned long long m = (b & 0x7fffffu) | 0x800000u;
        const int s = -sh;
        unsigned long long q = m >> s;
        const unsigned long long rem = m & ((1ull << s) - 1ull), half = 1ull << (s - 1);
        q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
        r = (long long)q;
    } else {
        r = 0;  // below 2^-41
    }
    return (b >> 31) ? -r : r;
}

// Points [beg, end) of this block: n split into gridDim.x contiguous ranges
// of n / G or n / G + 1 points, with 32-bit arithmetic (a 64-bit division
// would run through the FP64 pipe).
__device__ __forceinline__ void block_range(int n, long long& beg, long long& end)
{
    const unsigned G = gridDim.x, b = blockIdx.x, un = (unsigned)n;
    const unsigned q = un / G, r = un % G;
    beg = (long long)b * q + (b < r ? b : r);
    end = beg + q + (b < r ? 1 : 0);
}

// Fixed-order block sum of NV floats per thread, each lane's value carried
// as an unevaluated float pair (s, c) through the warp's shuffle tree with
// error-free additions (TwoSum), so the warp sum keeps about twice float
// precision without the FP64 pipe; thread i then adds value i over the warps
// in order, in FP64.  The warps' sums go through shared memory as floats and
// become FP64 in that thread: converting in each warp, on a FP64 pipe that all
// of them share, made this sum 9 700 cycles of a polish step (29 values), now
// 3 900.  Block totals in out[0 .. NV) (shared), visible to every thread.
template <int NV>
__device__ inline void block_sum_ff(const float* v, float* sh, double* out)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float sv[NV], cv[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        sv[i] = v[i];
        cv[i] = 0.0f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float s2 = __shfl_xor_sync(0xffffffffu, sv[i], o), c2 = __shfl_xor_sync(0xffffffffu, cv[i], o);
            // the same operand order on both lanes of a pair (lower lane's
            // value first), so both hold bit-identical results
            const bool low = (lane & o) == 0;
            const float a = low ? sv[i] : s2, b = low ? s2 : sv[i];
            const float ca = low ? cv[i] : c2, cb = low ? c2 : cv[i];
            const float h = __fadd_rn(a, b);
            const float bb = __fsub_rn(h, a);
            const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(h, bb)), __fsub_rn(b, bb));
            sv[i] = h;
            cv[i] = __fadd_rn(__fadd_rn(ca, cb), err);
        }
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            sh[2 * (warp * NV + i)] = sv[i];
            sh[2 * (warp * NV + i) + 1] = cv[i];
        }
    __syncthreads();
    if (tid < NV) {
        double s = 0.0;
        for (int w = 0; w < AL_THREADS / 32; ++w)
            s += (double)sh[2 * (w * NV + tid)] + (double)sh[2 * (w * NV + tid) + 1];
        out[tid] = s;
    }
    __syncthreads();
}

// Fixed-order block sum of NV floats per thread: the 32 lanes of a warp in
// float (about one sample per lane in the polish, so float keeps ~1e-6 of
// the sum), the warps in FP64 by thread i as above (out[0 .. NV)).
template <int NV>
__device__ inline void block_sum_f(float* v, float* sh, double* out)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i)
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sh[warp * NV + i] = v[i];
    __syncthreads();
    if (tid < NV) {
        double s = 0.0;
        for (int w = 0; w < AL_THREADS / 32; ++w) s += (double)sh[w * NV + tid];
        out[tid] = s;
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Loss and derivatives of F frames
// ---------------------------------------------------------------------------
struct AlignArgs {
    const void* tsdf;
    GridInfo g;
    const float4* pts;
    const int* counts;
    int n_max;
    const double* poses;  // F x 16
    const double* xi;     // F x 6 or null
    const double* dloss;  // F or null
    const float* records; // float records of the cell view, or null
    int row, plane;
    double* part;         // F x tiles x 8
    long long* acc;       // n_nodes or null
    const FramePose* fposes;  // F, from align_prep
};

// Block f prepares frame f: its perturbed pose, v and 2 W (64 frames: 14.5 us
// with a thread each in one block, 7.4 us so).
__global__ void __launch_bounds__(64) align_prep(const double* poses, const double* xi, const double* dloss, GridInfo g,
                                                 FramePose* out)
{
    __shared__ double s_xi[6], s_P[12], s_T[12], sh[16];
    __shared__ int sh_ok;
    const int f = blockIdx.x, tid = threadIdx.x;
    if (tid < 6) s_xi[tid] = xi ? xi[6 * (size_t)f + tid] : 0.0;
    if (tid >= 32 && tid < 44) s_P[tid - 32] = poses[16 * (size_t)f + tid - 32];
    __syncthreads();
    pair_perturb(s_P, s_xi, s_T, sh);
    pair_make_posef(s_T, g, &out[f].P, &sh_ok);
    if (tid < 3) out[f].V[tid] = (float)s_xi[3 + tid];
    if (tid == 32) out[f].w2 = (float)(2.0 * (dloss ? dloss[f] : 1.0));
}

template <typename TS, bool RECORDS>
__global__ void __launch_bounds__(AL_THREADS) align_kernel(AlignArgs a)
{
    __shared__ FramePose sF;
    __shared__ float sh[(AL_THREADS / 32) * 8 * 2];
    const int f = blockIdx.y, tid = threadIdx.x;
    block_copy_words(a.fposes + f, &sF);
    const PoseF& sP = sF.P;
    const float* sV = sF.V;
    const int n = a.counts ? min(a.counts[f], a.n_max) : a.n_max;
    long long beg, end;
    block_range(n, beg, end);
    const Field<TS> field = {static_cast<const TS*>(a.tsdf), a.records, a.row, a.plane};
    const float inv_vs = (float)a.g.inv_vs;
    // dL/dV increments in units of 2^-40: round(2 W t w 2^40), formed in
    // float (exact for W = 1, one float rounding otherwise)
    const float w2 = sF.w2;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // L, C, gw[3], gv[3]
    const float4* pts = a.pts + (size_t)f * a.n_max;
    float4 next = beg + tid < end ? __ldg(pts + beg + tid) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (long long e = beg + tid; e < end; e += AL_THREADS) {
        // (the next point is on its way while this one's record is)
        const float4 p = next;
        if (e + AL_THREADS < end) next = __ldg(pts + e + AL_THREADS);
        float t, dg[3], fr[3];
        int base;
        if (!sample_f<TS, RECORDS>(field, a.g, sP, p.x, p.y, p.z, t, dg, base, fr)) continue;
        float q[3];
        transform_f(sP, p.x, p.y, p.z, q);
        const float gt[3] = {dg[0] * inv_vs, dg[1] * inv_vs, dg[2] * inv_vs};
        const float rr[3] = {q[0] - sV[0], q[1] - sV[1], q[2] - sV[2]};
        const float t2 = 2.0f * t;
        acc[0] = fmaf(t, t, acc[0]);
        acc[1] += 1.0f;
        acc[2] = fmaf(t2, rr[1] * gt[2] - rr[2] * gt[1], acc[2]);
        acc[3] = fmaf(t2, rr[2] * gt[0] - rr[0] * gt[2], acc[3]);
        acc[4] = fmaf(t2, rr[0] * gt[1] - rr[1] * gt[0], acc[4]);
        acc[5] = fmaf(t2, gt[0], acc[5]);
        acc[6] = fmaf(t2, gt[1], acc[6]);
        acc[7] = fmaf(t2, gt[2], acc[7]);
        if (a.acc) {
            const int nx = a.g.nx, nxy = a.g.nx * a.g.ny;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float w = ((c & 1) ? fr[0] : 1.0f - fr[0]) * (((c >> 1) & 1) ? fr[1] : 1.0f - fr[1]) *
                                (((c >> 2) & 1) ? fr[2] : 1.0f - fr[2]);
                const int idx = base + ((c & 1) ? 1 : 0) + (((c >> 1) & 1) ? nx : 0) + (((c >> 2) & 1) ? nxy : 0);
                const long long inc = fix40(w2 * (t * w));
                if (inc != 0) atomicAdd(reinterpret_cast<unsigned long long*>(a.acc + idx), (unsigned long long)inc);
            }
        }
    }
    __shared__ double tot[8];
    block_sum_ff<8>(acc, sh, tot);
    if (tid < 8) a.part[((size_t)f * gridDim.x + blockIdx.x) * 8 + tid] = tot[tid];
}

// Sums of NV values over `tiles` partial records (record y at part + y *
// NV) by one block: thread (i, j) adds value i over tiles j, j + J, ... in
// order, then thread i adds its J partial sums in order (a fixed order
// whatever the scheduling).  Results in out[0 .. NV) of shared memory.
template <int NV>
__device__ inline void tile_sum(const double* part, int tiles, double* sh, double* out)
{
    constexpr int J = RED_THREADS / NV;
    const int tid = threadIdx.x, i = tid % NV, j = tid / NV;
    if (j < J) {
        double acc = 0.0;
#pragma unroll 4
        for (int y = j; y < tiles; y += J) acc += __ldcg(part + (size_t)y * NV + i);
        sh[j * NV + i] = acc;
    }
    __syncthreads();
    if (tid < NV) {
        double acc = 0.0;
        for (int q = 0; q < J; ++q) acc += sh[q * NV + tid];
        out[tid] = acc;
    }
    __syncthreads();
}

// one block per frame
__global__ void __launch_bounds__(RED_THREADS) align_finish(const double* part, int tiles, const double* xi,
                                                            const double* dloss, double* loss, int* count,
                                                            double* grad)
{
    __shared__ double sh[RED_THREADS];
    __shared__ double s[8];
    const int f = blockIdx.x;
    tile_sum<8>(part + (size_t)f * tiles * 8, tiles, sh, s);
    if (threadIdx.x != 0) return;
    loss[f] = s[0];
    if (count) count[f] = (int)s[1];
    if (grad) {
        double w[3] = {0, 0, 0};
        if (xi)
            for (int i = 0; i < 3; ++i) w[i] = xi[6 * (size_t)f + i];
        double J[9];
        so3_left_jacobian(w, J);
        const double sc = dloss ? dloss[f] : 1.0;
        for (int i = 0; i < 3; ++i) {
            grad[6 * (size_t)f + i] = sc * (J[i] * s[2] + J[3 + i] * s[3] + J[6 + i] * s[4]);
            grad[6 * (size_t)f + 3 + i] = sc * s[5 + i];
        }
    }
}

// v * 2^-40 rounded to the nearest float (ties to even), by integer
// operations: the same float as the FP64 conversion and multiply for |v| <
// 2^53, without the FP64 pipe (v * 2^-40 stays inside the normal floats).
__device__ __forceinline__ float fixed40_to_float(long long v)
{
    if (v == 0) return 0.0f;
    const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int msb = 63 - __clzll((long long)m);
    int e = msb - 40;
    unsigned long long q;
    if (msb <= 23) {
        q = m << (23 - msb);
    } else {
        const int s = msb - 23;
        q = m >> s;
        const unsigned long long rem = m & ((1ull << s) - 1ull), half = 1ull << (s - 1);
        q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
        if (q == (1ull << 24)) {
            q >>= 1;
            ++e;
        }
    }
    return __uint_as_float((v < 0 ? 0x80000000u : 0u) | ((unsigned)(e + 127) << 23) | ((unsigned)q & 0x7fffffu));
}

// The accumulator to floats, and back to zero where it was not, so that the
// next call finds it zero (a separate fill wrote 8 bytes a node more).  Bound
// by HBM: 8 bytes read and 4 written a node.  Four nodes a thread at a time
// when the output is 16-byte aligned, else one.
template <bool QUADS>
__global__ void __launch_bounds__(256) fixed_to_float(long long* acc, float* out, size_t n)
{
    const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    size_t done = 0;
    if constexpr (QUADS) {
        longlong2* acc2 = reinterpret_cast<longlong2*>(acc);
        for (size_t i = first; i < n / 4; i += step) {
            const longlong2 a = __ldcs(acc2 + 2 * i), b = __ldcs(acc2 + 2 * i + 1);
            reinterpret_cast<float4*>(out)[i] = make_float4(fixed40_to_float(a.x), fixed40_to_float(a.y),
                                                            fixed40_to_float(b.x), fixed40_to_float(b.y));
            if ((a.x | a.y | b.x | b.y) != 0) {
                acc2[2 * i] = make_longlong2(0, 0);
                acc2[2 * i + 1] = make_longlong2(0, 0);
            }
        }
        done = n / 4 * 4;
    }
    for (size_t i = done + first; i < n; i += step) {
        const long long v = acc[i];
        out[i] = fixed40_to_float(v);
        if (v != 0) acc[i] = 0;
    }
}

// ---------------------------------------------------------------------------
// Gauss-Newton polish
// ---------------------------------------------------------------------------
struct GnArgs {
    const void* tsdf;
    GridInfo g;
    const float* records;  // float records of the cell view, or null
    int row, plane;
    const float4* pts;
    const int* n_dev;
    int n_max;
    GnState* st;
    double* part;      // (tiles + GN_CLASSES) x GN_VALS
    PoseF* pc;         // the candidate prepared by gn_begin or the step before
    // the step at the end of the launch
    int mode;          // 0: take the evaluated input pose; 1: accept or drop the candidate
    double* pose_out;  // or null: not the last step
    double* trace;     // or null
    int* accepted_out; // or null
};

// The 6x6 system A d = y by Gaussian elimination with partial pivoting, by the
// first warp: A | y in shared memory as 6 rows of 7, each element eliminated
// by a lane of its own with the operations of the serial loop, in its order
// (so a column costs one division and two more FP64 instructions; magnitudes
// are compared as integers).  False (in each lane) when a pivot column is zero
// or not a number.
__device__ inline bool warp_solve6(double (*A)[7], double* d)
{
    const int lane = threadIdx.x;
    auto magnitude = [](double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; };
    const long long inf = 0x7ff0000000000000ll;
#pragma unroll
    for (int col = 0; col < 6; ++col) {
        int piv = col;
        long long big = magnitude(A[col][col]);
        for (int q = col + 1; q < 6; ++q) {
            const long long v = magnitude(A[q][col]);
            if (v <= inf && big <= inf && v > big) {
                piv = q;
                big = v;
            }
        }
        if (big == 0 || big > inf) return false;
        // exchange rows col and piv
        double x = 0.0, y = 0.0;
        if (lane < 7) {
            x = A[piv][lane];
            y = A[col][lane];
        }
        __syncwarp();
        if (lane < 7) {
            A[piv][lane] = y;
            A[col][lane] = x;
        }
        __syncwarp();
        const int w = 6 - col, r = col + 1 + lane / w, c = col + 1 + lane % w;  // 30 elements at most
        if (r < 6) {
            const double m = A[r][col] / A[col][col];
            A[r][c] = A[r][c] - m * A[col][c];  // (column col is not written)
        }
        __syncwarp();
    }
    // back substitution: the products with a new unknown by a lane per row,
    // each row's subtractions in their order
    double prod[6] = {0, 0, 0, 0, 0, 0};  // lane r: A[r][c] d[c]
    const int row = lane < 6 ? lane : 5;
#pragma unroll
    for (int q = 5; q >= 0; --q) {
        double acc = A[row][6];
#pragma unroll
        for (int k = q + 1; k < 6; ++k) acc -= prod[k];
        const double x = __shfl_sync(0xffffffffu, acc / A[row][row], q);
        prod[q] = A[row][q] * x;
        if (lane == q) d[q] = x;
    }
    __syncwarp();
    return true;
}

// Shared memory of the step.
struct GnShared {
    double s[GN_VALS];
    double A[6][7];
    double d[6], T[12], Tc[12], rot[16];
    double obj, lambda;
    int take, ok, solved;
};

// One step by the block's first two warps, after the candidate's sums (sh.s):
// mode 0 takes the evaluated input pose as the current one, mode 1 accepts or
// drops the evaluated candidate; then the next candidate is formed.
__device__ inline void gn_step(const GnArgs& a, bool evaluated, GnShared& sh)
{
    const int tid = threadIdx.x;
    GnState* st = a.st;
    if (tid == 0) {
        double obj = st->obj, lambda = st->lambda;
        int take = 0, accepted = st->accepted;
        if (evaluated) {
            const double objc = sh.s[28] > 0.0 ? sh.s[27] / sh.s[28] : INFINITY;
            take = a.mode == 0 || objc < obj;
            if (take) obj = objc;
            if (a.mode == 1) {
                lambda = take ? lambda / 10.0 : lambda * 10.0;
                accepted += take;
            }
        }
        const int step = st->step + (a.mode == 1 ? 1 : 0);
        st->obj = sh.obj = obj;
        st->lambda = sh.lambda = lambda;
        st->accepted = accepted;
        st->step = step;
        st->have_cand = 0;
        sh.take = take;
        if (a.trace) a.trace[step] = obj;
        if (a.accepted_out) *a.accepted_out = accepted;
    }
    pair_sync();
    // the accepted pose and its system, kept in the state
    const bool take = sh.take != 0;
    if (tid < 12) {
        sh.T[tid] = take ? st->Tc[tid] : st->T[tid];
        st->T[tid] = sh.T[tid];
    }
    if (tid < 42) {
        const int r = tid / 7, c = tid % 7, lo = min(r, c), hi = max(r, c);
        double v;
        if (c == 6) {
            v = take ? sh.s[21 + r] : st->b[r];
            st->b[r] = v;
            v = -v;
        } else {
            v = take ? sh.s[lo * 6 - lo * (lo - 1) / 2 + hi - lo] : st->H[6 * r + c];
            st->H[6 * r + c] = v;
            if (r == c) v += sh.lambda * v;
        }
        sh.A[r][c] = v;
    }
    pair_sync();
    if (a.pose_out && tid < 16) a.pose_out[tid] = tid < 12 ? sh.T[tid] : tid == 15 ? 1.0 : 0.0;
    // next candidate
    if (!(sh.obj < INFINITY)) return;
    if (tid < 32) {
        const bool solved = warp_solve6(sh.A, sh.d);
        if (tid == 0) sh.solved = solved;
    }
    pair_sync();
    if (!sh.solved) return;
    pair_perturb(sh.T, sh.d, sh.Tc, sh.rot);
    if (tid < 12) st->Tc[tid] = sh.Tc[tid];
    pair_make_posef(sh.Tc, a.g, a.pc, &sh.ok);
    if (tid == 0) st->have_cand = 1;
}

// Sums of H, b, the squared residuals and the count over the block's points
// for the candidate.  The blocks' sums are added by classes (tile y is of class
// y mod 8), each by the last block of the class to finish, and the last class
// to finish adds the classes and makes the step (ticket counters, no
// spinning): a step is one launch.  Bound by the latency of its parts: a point
// a thread, a gather and the sums about 13 000 cycles, then the step's chain of
// FP64 operations about 20 000, twelve of them the 6x6 solve.  320x240 points,
// ten steps: 497 -> 271 us (a step was two launches, the second one thread's
// work of 35 us).
template <typename TS, bool RECORDS>
__global__ void __launch_bounds__(AL_THREADS) gn_kernel(GnArgs a)
{
    __shared__ PoseF sP;
    __shared__ float sh[(AL_THREADS / 32) * GN_VALS];
    __shared__ GnShared step;
    __shared__ int s_last;
    const int tid = threadIdx.x;
    if (a.st->have_cand) {  // (else the step ignores the partials)
        block_copy_words(static_cast<const PoseF*>(a.pc), &sP);
        const int n = a.n_dev ? min(*a.n_dev, a.n_max) : a.n_max;
        long long beg, end;
        block_range(n, beg, end);
        const Field<TS> field = {static_cast<const TS*>(a.tsdf), a.records, a.row, a.plane};
        const float inv_vs = (float)a.g.inv_vs;
        float acc[GN_VALS];
#pragma unroll
        for (int i = 0; i < GN_VALS; ++i) acc[i] = 0.0f;
        for (long long e = beg + tid; e < end; e += AL_THREADS) {
            const float4 p = __ldg(a.pts + e);
            float t, dg[3], fr[3];
            int base;
            if (!sample_f<TS, RECORDS>(field, a.g, sP, p.x, p.y, p.z, t, dg, base, fr)) continue;
            float q[3];
            transform_f(sP, p.x, p.y, p.z, q);
            const float gt[3] = {dg[0] * inv_vs, dg[1] * inv_vs, dg[2] * inv_vs};
            const float J[6] = {q[1] * gt[2] - q[2] * gt[1], q[2] * gt[0] - q[0] * gt[2], q[0] * gt[1] - q[1] * gt[0],
                                gt[0], gt[1], gt[2]};
            int m = 0;
#pragma unroll
            for (int r = 0; r < 6; ++r)
#pragma unroll
                for (int c = r; c < 6; ++c) {
                    acc[m] = fmaf(J[r], J[c], acc[m]);
                    ++m;
                }
#pragma unroll
            for (int r = 0; r < 6; ++r) acc[21 + r] = fmaf(J[r], t, acc[21 + r]);
            acc[27] = fmaf(t, t, acc[27]);
            acc[28] += 1.0f;
        }
        __shared__ double tot[GN_VALS];
        block_sum_f<GN_VALS>(acc, sh, tot);
        if (tid < GN_VALS) a.part[(size_t)blockIdx.x * GN_VALS + tid] = tot[tid];
    }
    __threadfence();
    __syncthreads();
    const int tiles = gridDim.x, cls = blockIdx.x % GN_CLASSES;
    if (tid == 0) {
        const unsigned members = (unsigned)((tiles - cls + GN_CLASSES - 1) / GN_CLASSES);
        s_last = atomicAdd(&a.st->class_ticket[cls], 1u) == members - 1;
    }
    __syncthreads();
    if (!s_last || tid >= 64) return;
    __threadfence();
    double* sums = a.part + (size_t)tiles * GN_VALS;
    const bool evaluated = a.st->have_cand != 0;
    if (evaluated && tid < GN_VALS) {
        // loads 13 at a time (37 tiles in a class): one by one each addition
        // waits for L2
        double s = 0.0;
        for (int y0 = cls; y0 < tiles; y0 += 13 * GN_CLASSES) {
            double v[13];
#pragma unroll
            for (int q = 0; q < 13; ++q) {
                const int y = y0 + q * GN_CLASSES;
                v[q] = __ldcg(a.part + (size_t)min(y, tiles - 1) * GN_VALS + tid);
            }
#pragma unroll
            for (int q = 0; q < 13; ++q)
                if (y0 + q * GN_CLASSES < tiles) s += v[q];
        }
        sums[cls * GN_VALS + tid] = s;
        __threadfence();
    }
    pair_sync();
    if (tid == 0) {
        a.st->class_ticket[cls] = 0u;
        s_last = atomicAdd(&a.st->ticket, 1u) == (unsigned)min(tiles, GN_CLASSES) - 1;
    }
    pair_sync();
    if (!s_last) return;
    __threadfence();
    if (evaluated && tid < GN_VALS) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < GN_CLASSES; ++q) s += __ldcg(sums + q * GN_VALS + tid);
        step.s[tid] = s;
    }
    pair_sync();
    if (tid == 0) a.st->ticket = 0u;
    gn_step(a, evaluated, step);
}

// The input pose becomes the first candidate to evaluate.
__global__ void __launch_bounds__(64) gn_begin(GnState* st, const double* pose_in, GridInfo g, PoseF* pc)
{
    __shared__ double T[12];
    __shared__ int sh_ok;
    const int tid = threadIdx.x;
    if (tid < 12) st->Tc[tid] = T[tid] = pose_in[tid];
    __syncthreads();
    pair_make_posef(T, g, pc, &sh_ok);
    if (tid != 0) return;
    st->lambda = 1e-3;
    st->accepted = 0;
    st->step = 0;
    st->obj = INFINITY;
    st->have_cand = 1;
    for (int q = 0; q < GN_CLASSES; ++q) st->class_ticket[q] = 0u;
    st->ticket = 0u;
}

GridInfo grid_info(const pf_volume* v)
{
    GridInfo g;
    g.nx = v->desc.nx;
    g.ny = v->desc.ny;
    g.nz = v->desc.nz;
    g.inv_vs = 1.0 / (double)v->desc.voxel_size;
    for (int q = 0; q < 3; ++q) g.org[q] = v->desc.origin[q];
    return g;
}

// Float records of the volume's own stored values, which samples can read in
// place of its nodes: a float grid's view, or a narrow grid's full view (not a
// float grid's narrower search view, which holds rounded values).
const float* float_records(const pf_volume* v)
{
    if (pf_view_dtype(v) != v->desc.tsdf_dtype) return nullptr;
    return v->desc.tsdf_dtype == PF_F32 ? static_cast<const float*>(v->cells) : v->cells32;
}

template <template <typename, bool> class K, typename Args>
void launch_storage(const pf_volume* v, dim3 grid, cudaStream_t s, Args& a)
{
    a.records = float_records(v);
    a.row = v->pitch.row;
    a.plane = v->pitch.plane;
    if (a.records) {  // (the storage type of the nodes does not matter)
        K<float, true>::run(grid, s, a);
        return;
    }
    switch (v->desc.tsdf_dtype) {
    case PF_F16: K<__half, false>::run(grid, s, a); break;
    case PF_BF16: K<__nv_bfloat16, false>::run(grid, s, a); break;
    case PF_FP8E4M3: K<__nv_fp8_e4m3, false>::run(grid, s, a); break;
    default: K<float, false>::run(grid, s, a); break;
    }
}

template <typename TS, bool RECORDS>
struct AlignLaunch {
    static void run(dim3 grid, cudaStream_t s, const AlignArgs& a)
    {
        align_kernel<TS, RECORDS><<<grid, AL_THREADS, 0, s>>>(a);
    }
};

template <typename TS, bool RECORDS>
struct GnLaunch {
    static void run(dim3 grid, cudaStream_t s, const GnArgs& a) { gn_kernel<TS, RECORDS><<<grid, AL_THREADS, 0, s>>>(a); }
};

AlignScratch& scratch_of(const pf_volume* v)
{
    std::lock_guard<std::mutex> lk(g_mu);
    return g_scratch[v];
}

}  // namespace

namespace pf {
// Frees the scratch of a volume (called by pf_destroy_volume).
void align_release(const pf_volume* v)
{
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_scratch.find(v);
    if (it == g_scratch.end()) return;
    cudaFree(it->second.part);
    cudaFree(it->second.acc);
    cudaFree(it->second.gn_part);
    cudaFree(it->second.gn_state);
    cudaFree(it->second.frame_pose);
    cudaFree(it->second.gn_pose);
    g_scratch.erase(it);
}
}  // namespace pf

extern "C" {

static pf_status pf_align_loss_impl(const pf_volume* v, const float* points_dev, const int* counts_dev, int n_max,
                                    int n_frames, const double* poses_dev, const double* xi_dev,
                                    const double* dloss_dev, double* loss_dev, int* count_dev, double* grad_xi_dev,
                                    float* grad_tsdf_dev, void* stream)
{
    if (!v || !poses_dev || !loss_dev || n_frames < 1 || n_max < 0 || n_frames > 65535) return PF_ERR_INVALID_ARG;
    if (n_max > 0 && !points_dev) return PF_ERR_INVALID_ARG;
    if (((uintptr_t)points_dev & 15) != 0) return PF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    AlignScratch& sc = scratch_of(v);
    const int tiles = std::max(1, std::min(AL_TILES, (AL_BLOCKS + n_frames - 1) / n_frames));
    const size_t need = (size_t)n_frames * tiles * 8;
    pf_volume* owner = const_cast<pf_volume*>(v);
    if (sc.part_cap < need) {
        const size_t cap = (size_t)pf::grown_capacity((long long)sc.part_cap, (long long)need);
        PF_CUDA(pf::grow_scratch(owner, {pf::grow(&sc.part, cap)}, &s));
        sc.part_cap = cap;
    }
    if (sc.frame_cap < n_frames) {
        const int cap = (int)pf::grown_capacity(sc.frame_cap, n_frames);
        PF_CUDA(pf::grow_scratch(owner, {pf::grow(reinterpret_cast<FramePose**>(&sc.frame_pose), (size_t)cap)}, &s));
        sc.frame_cap = cap;
    }
    // the accumulator is zero between calls: fixed_to_float leaves it so
    if (grad_tsdf_dev && !sc.acc_zero) {
        if (!sc.acc) PF_CUDA(pf::dev_malloc(&sc.acc, v->n_nodes * sizeof(long long)));
        else PF_CUDA(cudaDeviceSynchronize());  // a call that failed half-way may still write to it
        PF_CUDA(pf::zero_for(sc.acc, v->n_nodes * sizeof(long long), &s));
        sc.acc_zero = true;
    }
    AlignArgs a;
    a.tsdf = v->tsdf;
    a.g = grid_info(v);
    a.pts = reinterpret_cast<const float4*>(points_dev);
    a.counts = counts_dev;
    a.n_max = n_max;
    a.poses = poses_dev;
    a.xi = xi_dev;
    a.dloss = dloss_dev;
    a.part = sc.part;
    a.acc = grad_tsdf_dev ? sc.acc : nullptr;
    a.fposes = static_cast<const FramePose*>(sc.frame_pose);
    align_prep<<<n_frames, 64, 0, s>>>(poses_dev, xi_dev, dloss_dev, a.g, static_cast<FramePose*>(sc.frame_pose));
    launch_storage<AlignLaunch>(v, dim3(tiles, n_frames), s, a);
    align_finish<<<n_frames, RED_THREADS, 0, s>>>(sc.part, tiles, xi_dev, dloss_dev, loss_dev, count_dev,
                                                  grad_xi_dev);
    pf::count_launch(3);
    if (grad_tsdf_dev) {
        if (((uintptr_t)grad_tsdf_dev & 15) == 0)
            fixed_to_float<true><<<8 * 152, 256, 0, s>>>(sc.acc, grad_tsdf_dev, v->n_nodes);
        else
            fixed_to_float<false><<<8 * 152, 256, 0, s>>>(sc.acc, grad_tsdf_dev, v->n_nodes);
        pf::count_launch();
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess && grad_tsdf_dev) sc.acc_zero = false;  // (its address may be in a captured graph: kept)
    return pf::cuda_status(e);
}

static pf_status pf_polish_impl(const pf_volume* v, const float* points_dev, const int* n_dev, int n_max,
                                double* pose_dev, int steps, double* trace_dev, int* accepted_dev, void* stream)
{
    if (!v || !pose_dev || n_max < 0 || steps < 0 || steps > 1000) return PF_ERR_INVALID_ARG;
    if (n_max > 0 && !points_dev) return PF_ERR_INVALID_ARG;
    if (((uintptr_t)points_dev & 15) != 0) return PF_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    AlignScratch& sc = scratch_of(v);
    if (!sc.gn_part) PF_CUDA(pf::dev_malloc(&sc.gn_part, (size_t)(AL_TILES + GN_CLASSES) * GN_VALS * sizeof(double)));
    if (!sc.gn_state) PF_CUDA(pf::dev_malloc(&sc.gn_state, sizeof(GnState)));
    if (!sc.gn_pose) PF_CUDA(pf::dev_malloc(&sc.gn_pose, sizeof(PoseF)));
    PoseF* pc = static_cast<PoseF*>(sc.gn_pose);
    GnState* st = reinterpret_cast<GnState*>(sc.gn_state);

    GnArgs a;
    a.tsdf = v->tsdf;
    a.g = grid_info(v);
    a.pts = reinterpret_cast<const float4*>(points_dev);
    a.n_dev = n_dev;
    a.n_max = n_max;
    a.st = st;
    a.part = sc.gn_part;
    a.pc = pc;
    // evaluate the input pose, then `steps` candidates
    a.trace = trace_dev;
    a.accepted_out = accepted_dev;
    gn_begin<<<1, 64, 0, s>>>(st, pose_dev, a.g, pc);
    pf::count_launch();
    for (int k = 0; k <= steps; ++k) {
        a.mode = k == 0 ? 0 : 1;
        a.pose_out = k == steps ? pose_dev : nullptr;
        launch_storage<GnLaunch>(v, dim3(AL_TILES), s, a);
        pf::count_launch();
        PF_LAUNCHED();
    }
    return PF_OK;
}

}  // extern "C"

// Every entry point that takes a volume keeps its last failing status
// there (pf_volume_last_error).
extern "C" {

pf_status pf_align_loss(const pf_volume* v, const float* points_dev, const int* counts_dev, int n_max, int n_frames,
                        const double* poses_dev, const double* xi_dev, const double* dloss_dev, double* loss_dev,
                        int* count_dev, double* grad_xi_dev, float* grad_tsdf_dev, void* stream)
{
    return pf::keep_status(v, pf_align_loss_impl(v, points_dev, counts_dev, n_max, n_frames, poses_dev, xi_dev,
                                                 dloss_dev, loss_dev, count_dev, grad_xi_dev, grad_tsdf_dev, stream));
}

pf_status pf_polish(const pf_volume* v, const float* points_dev, const int* n_dev, int n_max, double* pose_dev,
                    int steps, double* trace_dev, int* accepted_dev, void* stream)
{
    return pf::keep_status(v, pf_polish_impl(v, points_dev, n_dev, n_max, pose_dev, steps, trace_dev, accepted_dev,
                                             stream));
}

}  // extern "C"
